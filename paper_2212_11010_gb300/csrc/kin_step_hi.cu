// kin_step_hi.cu -- fixed-shape step kernels for 3D problems of degrees 2 and 3, FP32.
#include "kin_aux.h"
#include "kin_device.cuh"
#include "kin_fixed.cuh"

namespace kin {

// (dim, degree, system, B0, B1, B2, threads, min blocks per SM).  Rows must be
// whole 16-byte words (4 cells at p = 2); tiles of 52 to 74 KB leave three or
// four per SM.  On the generic kernel these ran with 26 KB tiles of unaligned
// rows.  Set-up, steps and read-back, before -> now: Euler 48^3, p = 2, 15 steps
// 15.8 -> 5.2 ms; 32^3, p = 3, 8 steps 4.5 -> 1.4; Maxwell 48^3, p = 2, 8 steps
// 16.4 -> 3.6; 32^3, p = 3 5.8 -> 1.8.
#define KIN_FIXED_HI(X)                     \
    X(3, 2, kEuler, 4, 2, 2, 256, 3)        \
    X(3, 3, kEuler, 2, 2, 2, 256, 3)        \
    X(3, 2, kMaxwell, 4, 2, 2, 256, 3)      \
    X(3, 3, kMaxwell, 2, 2, 2, 256, 2)

FixedKernel fixed_kernel_hi(int dim, int degree, int system, const int B[3])
{
    FixedKernel k{nullptr, nullptr, 0, 0};
#define KIN_TRY(DD, PP, SY, X0, X1, X2, NT, MB)                                                         \
    if (dim == DD && degree == PP && system == SY && B[0] == X0 && B[1] == X1 && B[2] == X2) {          \
        k.fn = (StepKernel)step_kernel_fixed<DD, PP, SY, float, X0, X1, X2, NT, MB, 1>;                    \
        k.threads = NT;                                                                                 \
        k.smem = Shape<DD, PP, SY, float, X0, X1, X2>::SMEM + Shape<DD, PP, SY, float, X0, X1, X2>::TIN_BYTES;  \
        return k;                                                                                       \
    }
    KIN_FIXED_HI(KIN_TRY)
#undef KIN_TRY
    return k;
}

}  // namespace kin
