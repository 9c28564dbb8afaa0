// kin_init.cuh -- f = M(W) of an FP64 macroscopic state (Sec. 2.2), shared by
// the three initialisation kernels (axis sets, d + 1 sets, tetrahedra).
//
// What bounds it: the traffic is m doubles read and nvel m values written per
// node, but one FP64 operation costs 64 FP32 ones on sm_103a (2 per clock and
// SM), and the Maxwellians of a node take 100 to 400 of them with their
// divisions.  Before, 128^3 cells of 3D Euler (p = 1, 2.7 GB) took 11.2 ms, 4%
// of the copy rate; now 0.6 ms (67%).  An FP64 state keeps its FP64
// operations, with one reciprocal per node instead of a division per use
// (48^3 cells of Maxwell: 0.64 -> 0.08 ms).  For an FP32 state the Maxwellians
// are therefore evaluated on unevaluated FP32 pairs (Dekker, "A floating-point
// technique for extending the available precision", 1971; 47 bits).  The double
// is split into its pair with integer instructions, so a node issues no FP64
// instruction at all.
//   What a pair loses against FP64 counts where values cancel: the pressure is a
// small difference at high Mach numbers, and W/(2d) -+ Q/(2 lambda) changes
// sign.  Each node checks that (init_flux, init_put), and one where a difference
// is smaller than 2^-5 (pressure) or 2^-6 (2^-12 for the linear systems) of its terms, or
// whose values leave the range in which no partial result can leave the FP32 exponent
// range (init_fast), is evaluated again in FP64.  So every value is
// off by less than 2^-32 of itself before its rounding to FP32: an input is cut
// to 2^-47, a product or sum adds at most 2^-45, at most eight of them follow
// one another, and the two differences lose 5 and 6 bits.
#pragma once

#include <math.h>

#include <type_traits>

#include "kin_device.cuh"

namespace kin {

struct F2 {
    float h, l;              // value h + l, |l| <= ulp(h) / 2
};

// (products are kept apart from the sums that follow: a contraction would
// change the error terms)
__device__ __forceinline__ F2 f2_fast(float h, float l)
{
    F2 r;
    r.h = __fadd_rn(h, l);
    r.l = __fadd_rn(l, -__fadd_rn(r.h, -h));
    return r;
}
__device__ __forceinline__ F2 operator+(F2 a, F2 b)
{
    const float s = __fadd_rn(a.h, b.h), bb = __fadd_rn(s, -a.h);
    const float e = __fadd_rn(__fadd_rn(a.h, -__fadd_rn(s, -bb)), __fadd_rn(b.h, -bb));
    return f2_fast(s, __fadd_rn(e, __fadd_rn(a.l, b.l)));
}
__device__ __forceinline__ F2 operator-(F2 a) { return F2{-a.h, -a.l}; }
__device__ __forceinline__ F2 operator-(F2 a, F2 b) { return a + (-b); }
__device__ __forceinline__ F2 operator*(F2 a, F2 b)
{
    const float p = __fmul_rn(a.h, b.h);
    return f2_fast(p, __fmaf_rn(a.l, b.h, __fmaf_rn(a.h, b.l, __fmaf_rn(a.h, b.h, -p))));
}
// Newton step on the rounded reciprocal: the residual 1 - b r0 is exact up to 2^-48
__device__ __forceinline__ F2 rcp_of(F2 b)
{
    const float r = __frcp_rn(b.h);
    return f2_fast(r, __fmul_rn(r, __fmaf_rn(-b.l, r, __fmaf_rn(-b.h, r, 1.0f))));
}
__device__ __forceinline__ double rcp_of(double b) { return 1.0 / b; }

__host__ __device__ __forceinline__ F2 f2_make(double x)
{
    F2 r;
    r.h = (float)x;
    r.l = (float)(x - (double)r.h);
    return r;
}
template <typename V> __device__ __forceinline__ V init_const(double x);
template <> __device__ __forceinline__ double init_const<double>(double x) { return x; }
template <> __device__ __forceinline__ F2 init_const<F2>(double x) { return f2_make(x); }

// A double with 2^-75 <= |x| < 2^100, or zero, as a pair: the upper 24
// significand bits, then the next 23.
__device__ __forceinline__ F2 f2_of_bits(unsigned hi, unsigned lo)
{
    const unsigned a = hi & 0x7fffffffu, sg = hi & 0x80000000u;
    if ((a | lo) == 0) return F2{0.0f, 0.0f};
    const float h = __uint_as_float(__funnelshift_l(lo, a - 0x38000000u, 3) | sg);
    // scale 2^(e - 46) of the 23 bits below; e + 127 - 46 >= 6 by the range
    const float sc = __uint_as_float(((((a >> 20) - 1023u + 127u - 46u) & 0xffu) << 23) | sg);
    const float r = __uint_as_float(0x4b000000u | ((lo & 0x1fffffffu) >> 6)) - 8388608.0f;
    return f2_fast(h, r * sc);
}

// Constants of the Maxwellians, in either arithmetic.
template <typename V>
struct InitK {
    V gm1, adv[3], inv_nv, inv2l;      // gamma - 1, a, 1 / (2d), 1 / (2 lambda)
};

struct InitArgs {
    long long nodes;
    int fast;                          // the model's constants allow the pair arithmetic
    InitK<double> kd;
    InitK<F2> kf;
};
InitArgs init_args(long long nodes, int dim, double lambda, double gamma, const double* adv);   // kin_aux.cu

template <typename V> __device__ __forceinline__ const InitK<V>& init_k(const InitArgs& A);
template <> __device__ __forceinline__ const InitK<double>& init_k<double>(const InitArgs& A) { return A.kd; }
template <> __device__ __forceinline__ const InitK<F2>& init_k<F2>(const InitArgs& A) { return A.kf; }

// Magnitude of a value, for the checks of the pair arithmetic.
__device__ __forceinline__ float init_mag(F2 x) { return fabsf(x.h); }
__device__ __forceinline__ float init_mag(double) { return 0.0f; }

// Q^a(W) for every axis: Euler, advection, or Maxwell (3D; Sec. 6.1.1).  Negative
// when the pressure is less than 2^-5 of (gamma - 1) E (pairs), else zero.
template <int D, int SYS, typename V>
__device__ __forceinline__ float init_flux(const InitK<V>& K, const V* W, V (*Q)[nvars(D, SYS)])
{
    float worst = 0.0f;
    if constexpr (SYS == kAdvection) {
#pragma unroll
        for (int a = 0; a < D; ++a) Q[a][0] = K.adv[a] * W[0];
    } else if constexpr (SYS == kMaxwell) {
        const V zero = init_const<V>(0.0);
#pragma unroll
        for (int a = 0; a < 3; ++a) maxwell_flux(W, a, Q[a], zero);
    } else {
        const V inv = rcp_of(W[0]);
        V ke = W[1] * W[1];
#pragma unroll
        for (int b = 1; b < D; ++b) ke = ke + W[1 + b] * W[1 + b];
        const V in = W[1 + D] - init_const<V>(0.5) * (ke * inv), pr = K.gm1 * in;
        if constexpr (std::is_same<V, F2>::value) worst = fminf(0.0f, fmaf(-0.03125f, W[1 + D].h, in.h));
#pragma unroll
        for (int a = 0; a < D; ++a) {
            const V ua = W[1 + a] * inv;
            Q[a][0] = W[1 + a];
#pragma unroll
            for (int b = 0; b < D; ++b) {
                const V q = W[1 + b] * ua;
                Q[a][1 + b] = b == a ? q + pr : q;
            }
            Q[a][1 + D] = (W[1 + D] + pr) * ua;
        }
    }
    return worst;
}

// Whether the pair arithmetic may be used on W: every value zero or in
// [2^-75, 2^100) when nothing but constants multiplies it, in
// [2^-48, 2^24) with rho >= 2^-12 for Euler, so that the largest product
// ((E + p) u, below 2^108 with gamma - 1 < 2^8) stays finite and the smallest
// (m^2 / rho, 2^-120) is not zero.  NaN and infinities fail the test.  (lambda and the other constants are checked on
// the host, init_fast_model.)
template <int M, int SYS>
__device__ __forceinline__ bool init_fast(const unsigned (&hi)[M], const unsigned (&lo)[M])
{
    bool ok = true;
#pragma unroll
    for (int v = 0; v < M; ++v) {
        const unsigned a = hi[v] & 0x7fffffffu;
        const unsigned top = SYS == kEuler ? 1023u + 24u : 1023u + 100u, low = SYS == kEuler ? 1023u - 48u : 1023u - 75u;
        ok = ok && ((a | lo[v]) == 0 || (a >= (low << 20) && a < (top << 20)));
    }
    if (SYS == kEuler) ok = ok && hi[0] >= ((1023u - 12u) << 20) && hi[0] < 0x7ff00000u;
    return ok;
}

inline int init_fast_model(double lambda, double gamma, const double* adv)
{
    auto in = [](double x, double lo, double hi) { return x >= lo && x <= hi; };
    return in(lambda, 1e-3, 1e6) && in(gamma - 1.0, 1e-6, 256.0) && in(fabs(adv[0]), 0.0, 1e6) &&
           in(fabs(adv[1]), 0.0, 1e6) && in(fabs(adv[2]), 0.0, 1e6);
}

// emit(W) with the node's m values, as pairs where the state is FP32 and the
// values allow it; as doubles else, and where emit on pairs returns false (a
// value that it stored has lost too much and is stored again).
template <int D, int SYS, typename T, typename E>
__device__ __forceinline__ void init_node(const double* __restrict__ Wd, long long nodes, long long i, int fast,
                                          const E& emit)
{
    constexpr int M = nvars(D, SYS);
    double w[M];
    if constexpr (sizeof(T) == 4) {
        unsigned hi[M], lo[M];
#pragma unroll
        for (int v = 0; v < M; ++v) {
            const double x = __ldg(Wd + (long long)v * nodes + i);
            hi[v] = (unsigned)__double2hiint(x);
            lo[v] = (unsigned)__double2loint(x);
        }
        if (fast && init_fast<M, SYS>(hi, lo)) {
            F2 W[M];
#pragma unroll
            for (int v = 0; v < M; ++v) W[v] = f2_of_bits(hi[v], lo[v]);
            if (emit(W)) return;
        }
    }
    // (read again: held over the pairs they cost registers on every node)
#pragma unroll
    for (int v = 0; v < M; ++v) w[v] = *(const volatile double*)(Wd + (long long)v * nodes + i);
    emit(w);
}

// Stores x, the sum of terms of magnitude mag; worst becomes negative when x has
// lost more than 6 bits (12 for the linear systems) to cancellation.
template <int SYS>
__device__ __forceinline__ void init_put(float& f, F2 x, float mag, float& worst)
{
    constexpr float part = SYS == kEuler ? 0.015625f : 0.000244140625f;
    f = x.h;
    worst = fminf(worst, fmaf(-part, mag, fabsf(x.h)));
}
template <int SYS, typename T>
__device__ __forceinline__ void init_put(T& f, double x, float, float&) { f = (T)x; }

}  // namespace kin
