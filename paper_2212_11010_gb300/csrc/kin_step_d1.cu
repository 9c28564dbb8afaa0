// kin_step_d1.cu -- instantiations of the fused sweep + relaxation kernel for
// 1 space dimension(s), degrees 1..3, scalar advection and Euler, FP32/FP64.
#include "kin_aux.h"
#include "kin_device.cuh"

#include <cooperative_groups.h>

namespace kin {

template <int P, int SYS>
static StepKernel pick(int prec)
{
    return prec == 1 ? (StepKernel)step_kernel<1, P, SYS, float>
                     : (StepKernel)step_kernel<1, P, SYS, double>;
}

StepKernel step_kernel_d1(int degree, int system, int prec)
{
    switch (degree * 4 + system) {        // (Maxwell is 3D only)
    case 4: return pick<1, kAdvection>(prec);
    case 5: return pick<1, kEuler>(prec);
    case 8: return pick<2, kAdvection>(prec);
    case 9: return pick<2, kEuler>(prec);
    case 12: return pick<3, kAdvection>(prec);
    case 13: return pick<3, kEuler>(prec);
    default: return nullptr;
    }
}

// ---------------------------------------------------------------------------
// small problems: all steps of a call in one launch
// ---------------------------------------------------------------------------

// A 1D problem of a few thousand values is bound by its launches: one step of
// 256 cells (p = 1, FP64) took 10.4 us, of which the arithmetic is a fraction.
// Here one cluster of thread blocks keeps f in shared memory, its cell blocks
// split over them, and exchanges the block summaries (the same ones, in the
// same arithmetic, as the one-step kernel) through distributed shared memory:
// two block barriers and one cluster barrier per step.  A step is a chain of
// dependent operations, so everything that does not change from step to step --
// the thread's line, its look-back walk, every address -- is worked out before
// the first (with the divisions inside the loop a step of 64 cells took 3.3 us).
//   Measured, 100 steps with set-up and read-back, before -> now: FP64 64 cells
// p = 1 843 -> 501 us, 256 cells 1047 -> 604, 2048 cells p = 3 1255 -> 1125;
// FP32 256 cells p = 1 634 -> 177, 8192 cells p = 3 635 -> 468.  What bounds it:
// the chain of a step's operations, in FP64 at about 100 cycles each (some 60 at
// p = 1), and about 1 us per step of cluster barrier and remote loads, so one
// block takes what it can in that time and eight take the rest; beyond the
// limits below the whole GPU is faster in spite of its launches.
template <int P, int SYS, typename T>
__global__ void __launch_bounds__(kMultiThreads) multi_kernel(const __grid_constant__ Inst I, int nsteps)
{
    namespace cg = cooperative_groups;
    constexpr int NP = P + 1, M = nvars(1, SYS), NPOP = 2 * M;
    extern __shared__ __align__(128) unsigned char smem_raw[];
    cg::cluster_group cluster = cg::this_cluster();
    const int B = I.B[0], nbk = I.nblk[0], nb = I.nb[0], NS = I.NS[0], K = I.iters;
    const int nc = gridDim.x, rank = blockIdx.x;          // one cluster
    const int per = (nbk + nc - 1) / nc;
    const int b0 = min(rank * per, nbk), nloc = min(per, nbk - b0);
    const int cells = nloc * B, pstride = cells * NP;
    auto sync = [&]() {
        if (nc == 1) __syncthreads();
        else cluster.sync();
    };
    // summaries [parity][population][own block]: zero-inflow outflow, outflow-node value
    const int half = NPOP * per;
    T* const sig = reinterpret_cast<T*>(smem_raw);
    T* const raw = sig + 2 * half;
    T* const s = raw + 2 * half;
    T* const f = static_cast<T*>(I.f) + (long long)b0 * B * NP;
    for (int pop = 0; pop < NPOP; ++pop)
        for (int e = threadIdx.x; e < pstride; e += blockDim.x) s[pop * pstride + e] = f[(long long)pop * I.nodes + e];

    // this thread's line: one (population, cell block)
    const bool mine = (int)threadIdx.x < NPOP * nloc;
    const int pop = mine ? threadIdx.x / nloc : 0, lb = mine ? threadIdx.x - pop * nloc : 0;
    const int sgn = pop < M ? 0 : 1;
    const int q = sgn == 0 ? b0 + lb : nbk - 1 - (b0 + lb), S = q / nb, r = q - S * nb;
    const int own_at = pop * per + lb;                    // place of its summaries
    T Pm[NP][NP], prow[NP];
#pragma unroll
    for (int i = 0; i < NP; ++i) {
        prow[i] = coef_of(I, sgn, kOffProw + i, T(0));
#pragma unroll
        for (int j = 0; j < NP; ++j) Pm[i][j] = coef_of(I, sgn, i * NP + j, T(0));
    }
    const T RB = coef_of(I, sgn, kOffRhoB, T(0)), rho = coef_of(I, sgn, kOffRho, T(0));
    if (mine) {
        sig[own_at] = static_cast<const T*>(I.sig_in)[(long long)pop * I.sig_stride + q];
        raw[own_at] = r == nb - 1 ? static_cast<const T*>(I.raw_in)[(long long)pop * I.raw_stride + S] : T(0);
    }
    // its look-back (chain_inflow): cnt blocks from block bq0, starting from
    // zero, a boundary value or the raw value at (raw_own, raw_at)
    int s0 = S - K, cnt, qj, kind = 0;
    const bool from_bnd = I.inflow[0] && s0 < 0;
    if (from_bnd) {
        cnt = S * nb + r;
        qj = 0;
        kind = 1;
    } else {
        while (s0 < 0) s0 += NS;
        cnt = (K - 1) * nb + r;
        qj = s0 + 1 == NS ? 0 : (s0 + 1) * nb;
        kind = 2;
    }
    if (cnt > I.lbdepth[sgn]) {
        qj = (qj + cnt - I.lbdepth[sgn]) % nbk;
        cnt = I.lbdepth[sgn];
        kind = 0;
    }
    auto block_of = [&](int qq) { return sgn == 0 ? qq : nbk - 1 - qq; };
    const int rb = block_of(s0 < 0 ? 0 : s0 * nb + nb - 1), raw_own = rb / per, raw_at = pop * per + rb % per;
    const int bq0 = block_of(qj), own0 = bq0 / per, lo0 = bq0 % per;
    const int own_last = (nbk - 1) / per, lo_last = (nbk - 1) % per;
    const T bnd = kind == 1 ? bnd_of<T>(I, pop) : T(0);
    T* const line = s + pop * pstride + (sgn == 0 ? lb * B : lb * B + B - 1) * NP;
    const int cstep = sgn == 0 ? NP : -NP;
    const int sp0 = pop * per;
    sync();

    for (int step = 0; step < nsteps; ++step) {
        const int par = step & 1;
        if (mine) {
            auto remote = [&](const T* p, int own) { return own == rank ? *p : *cluster.map_shared_rank(p, own); };
            T t = kind == 2 ? remote(raw + par * half + raw_at, raw_own) : bnd;
            const T* const sp = sig + par * half + sp0;
            int own = own0, lo = lo0;
#pragma unroll 4
            for (int j = 0; j < cnt; ++j) {
                t = fma(RB, t, remote(sp + lo, own));
                if (sgn == 0) {
                    const bool end = own == own_last && lo == lo_last, wrap = lo + 1 == per;
                    own = end ? 0 : own + wrap;
                    lo = end || wrap ? 0 : lo + 1;
                } else {
                    const bool end = own == 0 && lo == 0, wrap = lo == 0;
                    own = end ? own_last : own - wrap;
                    lo = end ? lo_last : (wrap ? per - 1 : lo - 1);
                }
            }
            // sweep (lines_axis, difference form)
            T* p = line;
#pragma unroll 4
            for (int cc = 0; cc < B; ++cc, p += cstep) {
                T u[NP], du[NP], dlt[NP];
#pragma unroll
                for (int j = 0; j < NP; ++j) {
                    u[j] = p[j];
                    du[j] = u[j] - t;
                }
#pragma unroll
                for (int i = 0; i < NP; ++i) {
                    T acc = Pm[i][0] * du[0];
#pragma unroll
                    for (int j = 1; j < NP; ++j) acc = fma(Pm[i][j], du[j], acc);
                    dlt[i] = acc;
                }
                t = sgn == 0 ? u[NP - 1] + dlt[NP - 1] : u[0] + dlt[0];
#pragma unroll
                for (int i = 0; i < NP; ++i) p[i] = fma(T(2), dlt[i], u[i]);
            }
        }
        __syncthreads();
        relax_block<1, P, SYS, T>(I, s, cells);
        __syncthreads();
        if (mine) {
            const T* p = line;
            T t = 0, last = 0;
#pragma unroll 4
            for (int cc = 0; cc < B; ++cc, p += cstep) {
                T acc = prow[0] * p[0];
#pragma unroll
                for (int j = 1; j < NP; ++j) acc = fma(prow[j], p[j], acc);
                t = fma(rho, t, acc);
                last = sgn == 0 ? p[NP - 1] : p[0];
            }
            sig[(par ^ 1) * half + own_at] = t;
            raw[(par ^ 1) * half + own_at] = last;
            if (step == nsteps - 1) {
                static_cast<T*>(I.sig_out)[(long long)pop * I.sig_stride + q] = t;
                if (r == nb - 1) static_cast<T*>(I.raw_out)[(long long)pop * I.raw_stride + S] = last;
            }
        }
        // this step's summaries are visible to the cluster; the ones it read may be overwritten
        sync();
    }
    for (int pp = 0; pp < NPOP; ++pp)
        for (int e = threadIdx.x; e < pstride; e += blockDim.x) f[(long long)pp * I.nodes + e] = s[pp * pstride + e];
}

template <int P, int SYS>
static const void* multi_pick(int prec)
{
    return prec == 1 ? (const void*)multi_kernel<P, SYS, float> : (const void*)multi_kernel<P, SYS, double>;
}

MultiKernel multi_kernel_d1(int degree, int system, int prec, int n, int B)
{
    MultiKernel k{nullptr, 0, 1, 2};
    const int npop = 2 * nvars(1, system), np = degree + 1, nblk = n / B;
    const long long values = (long long)n * np * npop;
    if (values > (prec == 1 ? 65536 : 16384)) return k;
    // (FP64 lines of up to 20 nodes: at 16 to 20 a step of 16384 values takes
    // 10.3 to 12.2 us against 10.7 to 12.8 of one launch per step, and the gain
    // falls with the chain of a line)
    if (prec != 1 && B * np > 20) return k;
    // (FP32, p = 1, 65536 values: 7.3 us per step either way)
    if (prec == 1 && degree == 1 && values > 32768) return k;
    k.blocks = values <= (prec == 1 ? 3072 : 1536) ? 1 : 8;
    // Calls of few steps take one launch of the grid-wide kernel per step (the results
    // are bitwise the same): one block or cluster spends about 5 us on moving f in and
    // out, the more the fewer values it shares the GPU for.  us of a call of n steps,
    // here against there: FP32, 4096 to 24576 values 8 + 3 (n - 1) and 6.2 n; 32768 10 + 4
    // (n - 1) and 6.2 n; 49152 12.3 + 6.0 (n - 1) and 6.2 n; FP64, 4096 to 8192 values 12
    // to 16 + 8 to 10 (n - 1) and 10 to 12 n; 16384 16 to 18 + 9.9 to 11.8 (n - 1) and 10.3
    // to 12.3 n.
    if (k.blocks > 1) k.from = prec == 1 ? (values <= 24576 ? 2 : (values <= 32768 ? 4 : 33)) : (values <= 8192 ? 5 : 15);
    const int per = (nblk + k.blocks - 1) / k.blocks;
    k.smem = (size_t)(prec == 1 ? 4 : 8) * npop * ((size_t)4 * per + (size_t)per * B * np);
    if (k.smem > 200 * 1024 || npop * per > kMultiThreads) return k;
    switch (degree * 2 + system) {
    case 2: k.fn = multi_pick<1, kAdvection>(prec); break;
    case 3: k.fn = multi_pick<1, kEuler>(prec); break;
    case 4: k.fn = multi_pick<2, kAdvection>(prec); break;
    case 5: k.fn = multi_pick<2, kEuler>(prec); break;
    case 6: k.fn = multi_pick<3, kAdvection>(prec); break;
    case 7: k.fn = multi_pick<3, kEuler>(prec); break;
    default: break;
    }
    return k;
}

}  // namespace kin
