// kin_step_f64.cu -- fixed-shape step kernels in FP64.
#include "kin_aux.h"
#include "kin_device.cuh"
#include "kin_fixed.cuh"

namespace kin {

// (dim, degree, system, B0, B1, B2, threads, min blocks per SM).  These are
// bound by the FP64 units (2 FMA per clock and SM), so what counts is the
// number of instructions that feed them.  Before (generic kernel) -> now:
// Maxwell 48^3, p = 1, 8 steps 14.2 -> 7.0 ms; Euler 48^3, p = 1, 5 steps
// 8.1 -> 3.7; 24^3, p = 2, 5 steps 2.6 -> 1.8; 2D 256^2, p = 1, 6 steps
// 0.87 -> 0.72.  Default blocks as before in their thinnest extent, so the
// summaries are no larger.
#define KIN_FIXED_F64(X)                    \
    X(2, 1, kEuler, 8, 8, 1, 128, 4)        \
    X(2, 3, kEuler, 8, 4, 1, 128, 3)        \
    X(3, 1, kEuler, 4, 4, 2, 128, 3)        \
    X(3, 2, kEuler, 2, 2, 2, 128, 3)        \
    X(3, 3, kEuler, 2, 2, 1, 128, 3)        \
    X(3, 1, kMaxwell, 4, 4, 2, 128, 3)      \
    X(3, 2, kMaxwell, 2, 2, 2, 128, 3)      \
    X(3, 3, kMaxwell, 2, 2, 1, 128, 3)

FixedKernel fixed_kernel_f64(int dim, int degree, int system, const int B[3])
{
    FixedKernel k{nullptr, nullptr, 0, 0};
#define KIN_TRY(DD, PP, SY, X0, X1, X2, NT, MB)                                                         \
    if (dim == DD && degree == PP && system == SY && B[0] == X0 && B[1] == X1 && B[2] == X2) {          \
        k.fn = (StepKernel)step_kernel_fixed<DD, PP, SY, double, X0, X1, X2, NT, MB, 1>;                   \
        k.threads = NT;                                                                                 \
        k.smem = Shape<DD, PP, SY, double, X0, X1, X2>::SMEM + Shape<DD, PP, SY, double, X0, X1, X2>::TIN_BYTES;\
        return k;                                                                                       \
    }
    KIN_FIXED_F64(KIN_TRY)
#undef KIN_TRY
    return k;
}

}  // namespace kin
