// kin_tet.cu -- the kinetic DG step on tetrahedral meshes (the paper's
// setting: Sec. 3.1 with tetrahedral cells, Sec. 3.2 downwind order, Sec. 5.1
// subdomain iteration).
//
// Basis: P1 Lagrange functions of each cell's four vertices, every integral
// exact: mass |L|/20 (1 + delta_ij); volume term (V . grad psi_i) |L|/4; face
// mass |F|/12 (1 + delta_ij) on the face's three vertices.  The implicit half
// step of Crank-Nicolson (tau = dt/2) of one cell reads
//   A f* = M f^n + tau sum_{inflow faces} |V.N| F f_R,
//   A = M + tau (-K + sum_{outflow faces} (V.N) F),
// and f^{n+1} = 2 f* - f^n.  Since A 1 = M 1 + tau sum_in |V.N| F 1 (the weak
// form of a constant), the kernels solve it in difference form about the
// cell's first node value r: f* - r 1 = A^{-1} [M (f^n - r 1) + tau sum_in
// |V.N| F (f_R - r 1)], exact for constant states whatever the rounding of
// A^{-1} (as on the Cartesian path).
//
// Downwind order (Sec. 3.2): for each velocity the host orients the faces,
// and inside every subdomain sorts the cells breadth-first into levels
// (cells of one level have no upwind neighbour in the same level).  A step
// is K launches of a sweep kernel -- blocks walk the levels of a (subdomain,
// velocity) with a barrier between them, every thread one (cell, variable)
// pair of the level -- and one pointwise launch for the relaxation.  Iteration p reads the
// neighbour's iterate p-1 across a subdomain interface (a face to another
// subdomain, or across the periodic boundary) and the current iterate
// inside (eq. ibvp); iterate 0 is f^n.
#include "kin_aux.h"
#include "kin_device.cuh"
#include "kin_init.cuh"
#include "kin_tma.cuh"

#include <algorithm>
#include <type_traits>

namespace kin {

// ---------------------------------------------------------------------------
// FP64 setup: per (velocity, cell) the record
//   [0, 16)  B = |L|/20 A^{-1} (row-major)
//   [16, 20) tau |V.N_a| |F_a| / 12 / (|L|/20) on inflow faces a, else 0
// (the cell's mass factor |L|/20 is moved into both, which makes a record
// five 16-byte words in FP32)
// ---------------------------------------------------------------------------

__global__ void tet_setup_kernel(TetSetupArgs A)
{
    const long long id = blockIdx.x * (long long)blockDim.x + threadIdx.x;
    if (id >= (long long)A.ncells * A.nvel) return;
    const int k = (int)(id / A.ncells);
    const int c = (int)(id - (long long)k * A.ncells);
    const double* x = A.xyz + (size_t)c * 12;
    const double V[3] = {A.vel[k][0], A.vel[k][1], A.vel[k][2]};
    double e[3][3];
    for (int b = 0; b < 3; ++b)
        for (int i = 0; i < 3; ++i) e[b][i] = x[3 * (b + 1) + i] - x[i];
    auto cross = [](const double* a, const double* b, double* r) {
        r[0] = a[1] * b[2] - a[2] * b[1];
        r[1] = a[2] * b[0] - a[0] * b[2];
        r[2] = a[0] * b[1] - a[1] * b[0];
    };
    double c12[3], c20[3], c01[3];
    cross(e[1], e[2], c12);
    cross(e[2], e[0], c20);
    cross(e[0], e[1], c01);
    const double det = e[0][0] * c12[0] + e[0][1] * c12[1] + e[0][2] * c12[2];
    const double vol = fabs(det) / 6.0;
    double grad[4][3];
    for (int i = 0; i < 3; ++i) {
        grad[1][i] = c12[i] / det;
        grad[2][i] = c20[i] / det;
        grad[3][i] = c01[i] / det;
        grad[0][i] = -(grad[1][i] + grad[2][i] + grad[3][i]);
    }
    double area[4];
    for (int a = 0; a < 4; ++a) {
        // |F_a| = 3 |L| |grad psi_a|: the face opposite vertex a
        const double g2 = grad[a][0] * grad[a][0] + grad[a][1] * grad[a][1] + grad[a][2] * grad[a][2];
        area[a] = 3.0 * vol * sqrt(g2);
    }
    const double tau = 0.5 * A.dt;
    double M[4][8];
    for (int i = 0; i < 4; ++i) {
        const double vg = V[0] * grad[i][0] + V[1] * grad[i][1] + V[2] * grad[i][2];
        for (int j = 0; j < 4; ++j) {
            M[i][j] = vol / 20.0 * (i == j ? 2.0 : 1.0) - tau * vg * vol / 4.0;
            M[i][4 + j] = i == j ? 1.0 : 0.0;
        }
    }
    const unsigned char ft = A.ftype[(size_t)k * A.ncells + c];
    double cin[4] = {0, 0, 0, 0};
    for (int a = 0; a < 4; ++a) {
        const int t = (ft >> (2 * a)) & 3;          // 1 inflow, 2 outflow, 0 parallel
        if (t == 0) continue;
        // V.N_a with N_a = -grad psi_a / |grad psi_a|
        const double gl = sqrt(grad[a][0] * grad[a][0] + grad[a][1] * grad[a][1] + grad[a][2] * grad[a][2]);
        const double vn = -(V[0] * grad[a][0] + V[1] * grad[a][1] + V[2] * grad[a][2]) / gl;
        if (t == 2) {
            for (int i = 0; i < 4; ++i)
                for (int j = 0; j < 4; ++j)
                    if (i != a && j != a) M[i][j] += tau * vn * area[a] / 12.0 * (i == j ? 2.0 : 1.0);
        } else {
            cin[a] = tau * fabs(vn) * area[a] / 12.0;
        }
    }
    // Gauss-Jordan inverse with partial pivoting
    for (int col = 0; col < 4; ++col) {
        int p = col;
        for (int r = col + 1; r < 4; ++r)
            if (fabs(M[r][col]) > fabs(M[p][col])) p = r;
        if (p != col)
            for (int j = 0; j < 8; ++j) {
                const double t = M[col][j];
                M[col][j] = M[p][j];
                M[p][j] = t;
            }
        const double d = 1.0 / M[col][col];
        for (int j = 0; j < 8; ++j) M[col][j] *= d;
        for (int r = 0; r < 4; ++r) {
            if (r == col) continue;
            const double l = M[r][col];
            for (int j = 0; j < 8; ++j) M[r][j] -= l * M[col][j];
        }
    }
    // records in the velocity's level order: a level reads consecutive records
    const size_t pos = (size_t)A.rank[(size_t)k * A.ncells + c];
    double* rec = A.c64 + ((size_t)k * A.ncells + pos) * kTetRec;
    for (int i = 0; i < 4; ++i)
        for (int j = 0; j < 4; ++j) rec[i * 4 + j] = M[i][4 + j] * (vol / 20.0);
    for (int a = 0; a < 4; ++a) rec[16 + a] = cin[a] / (vol / 20.0);
    if (A.c32) {
        // Rounded entry by entry, B acts on sums whose terms nearly cancel, and on a
        // mesh of congruent cells every cell and step has the same error: it adds
        // up (Maxwell, D3Q6, 8 steps: 2.5e-6 of the norm, 6e-7 with an exact B).
        // What counts is its effect on fields that are constant over the nodes,
        // B q with q_j = 5 + 4 (sum of the factors of the faces at node j) (the
        // rows of B q = 1): in each row the four entries are rounded up or down so
        // that the sum of their errors times q is smallest (6.5e-7).
        float* r32 = A.c32 + ((size_t)k * A.ncells + pos) * kTetRec;
        double q[4] = {5.0, 5.0, 5.0, 5.0};
        for (int a = 0; a < 4; ++a) {
            r32[16 + a] = (float)rec[16 + a];
            for (int j = 0; j < 4; ++j)
                if (j != a) q[j] += 4.0 * r32[16 + a];
        }
        for (int i = 0; i < 4; ++i) {
            float lo[4], hi[4];
            double off = 0.0, up[4], least = 0.0;
            for (int j = 0; j < 4; ++j) {
                lo[j] = __double2float_rd(rec[i * 4 + j]);
                hi[j] = __double2float_ru(rec[i * 4 + j]);
                off += ((double)lo[j] - rec[i * 4 + j]) * q[j];
                up[j] = ((double)hi[j] - (double)lo[j]) * q[j];
            }
            int best = 0;
            for (int mask = 0; mask < 16; ++mask) {
                double d = off;
                for (int j = 0; j < 4; ++j)
                    if ((mask >> j) & 1) d += up[j];
                if (mask == 0 || fabs(d) < least) {
                    least = fabs(d);
                    best = mask;
                }
            }
            for (int j = 0; j < 4; ++j) r32[i * 4 + j] = (best >> j) & 1 ? hi[j] : lo[j];
        }
    }
}

// ---------------------------------------------------------------------------
// sweep with the iterate in global memory: one block per (subdomain,
// velocity), levels in order.  For subdomains too wide for the ring sweep.
// ---------------------------------------------------------------------------

// The four node values of a cell as one vector access (FP32: 16 bytes; the
// cell's nodes are contiguous and every population slab starts 16-byte
// aligned).
template <typename T>
__device__ __forceinline__ void load4(const T* p, T (&u)[4])
{
    if constexpr (sizeof(T) == 4) {
        const float4 q = *reinterpret_cast<const float4*>(p);
        u[0] = q.x;
        u[1] = q.y;
        u[2] = q.z;
        u[3] = q.w;
    } else {
        const double2 a = reinterpret_cast<const double2*>(p)[0], b = reinterpret_cast<const double2*>(p)[1];
        u[0] = a.x;
        u[1] = a.y;
        u[2] = b.x;
        u[3] = b.y;
    }
}

template <typename T>
__device__ __forceinline__ void store4(T* p, const T (&u)[4])
{
    if constexpr (sizeof(T) == 4) {
        *reinterpret_cast<float4*>(p) = make_float4(u[0], u[1], u[2], u[3]);
    } else {
        reinterpret_cast<double2*>(p)[0] = make_double2(u[0], u[1]);
        reinterpret_cast<double2*>(p)[1] = make_double2(u[2], u[3]);
    }
}

// Every thread takes one (cell, variable) pair of the level: the m threads
// of a cell read the same coefficient record (one broadcast), and a level of
// c cells offers c m independent solves.  The inflow faces are resolved
// ahead of time, per position of the velocity's level order, one word per
// face: the neighbour cell R << 7, the neighbour's local index of each of
// the face's three vertices (2 bits at bits 5, 3, 1), and bit 0 set when the
// face is a subdomain interface (the value comes from the previous iterate,
// else from the current one); -1 on the faces that are not inflow faces.
// A thread's first pair of a level has its cell and face references loaded
// during the level before,
// so a level waits for one round of loads (the cell's f^n and record and the
// neighbour values, issued together: the face types come from the
// references) rather than for a chain of dependent ones.
template <typename T>
__global__ void __launch_bounds__(kTetSweepThreads, 2) tet_sweep_kernel(TetArgs A, const T* __restrict__ prev, T* cur)
{
    const int s = blockIdx.x, k = blockIdx.y;
    const int* __restrict__ order = A.order + (size_t)k * A.ncells;
    const int* __restrict__ fref = A.fref + (size_t)k * A.ncells * 4;
    const int lb = A.lstart[k * (A.nsub + 1) + s], le = A.lstart[k * (A.nsub + 1) + s + 1];
    const T* __restrict__ coef = static_cast<const T*>(A.coef) + (size_t)k * A.ncells * kTetRec;
    const T* __restrict__ fn = static_cast<const T*>(A.f);
    const long long nodes = A.nodes;
    const int m = A.m;
    const int tid = threadIdx.x, nt = blockDim.x;

    auto solve = [&](int pos, int v, int c, const int4 nr) {
        const T* rec = coef + (size_t)pos * kTetRec;
        const long long pop = (long long)(k * m + v) * nodes;
        T u[4];
        load4(fn + pop + (size_t)c * 4, u);
        const T r = u[0];
        T du[4], sum = T(0);
#pragma unroll
        for (int i = 0; i < 4; ++i) {
            du[i] = u[i] - r;
            sum += du[i];
        }
        T rhs[4];
#pragma unroll
        for (int i = 0; i < 4; ++i) rhs[i] = sum + du[i];
        const int fw[4] = {nr.x, nr.y, nr.z, nr.w};
#pragma unroll
        for (int a = 0; a < 4; ++a) {
            // (the face type comes from the references, already in registers,
            // so the neighbour loads need not wait for the record)
            const int wd = fw[a];
            if (wd < 0) continue;
            const T ca = rec[16 + a];
            const T* src = ((wd & 1) ? prev : cur) + pop + (size_t)(wd >> 7) * 4;
            // the neighbour's values at this cell's face vertices (j != a, ascending)
            T g[4] = {T(0), T(0), T(0), T(0)};
            T gs = T(0);
            int jj = 0;
#pragma unroll
            for (int j = 0; j < 4; ++j) {
                if (j == a) continue;
                g[j] = src[(wd >> (5 - 2 * jj)) & 3] - r;
                gs += g[j];
                ++jj;
            }
#pragma unroll
            for (int i = 0; i < 4; ++i)
                if (i != a) rhs[i] = fma(ca, gs + g[i], rhs[i]);
        }
        T x[4];
#pragma unroll
        for (int i = 0; i < 4; ++i) {
            T acc = rec[i * 4] * rhs[0];
#pragma unroll
            for (int j = 1; j < 4; ++j) acc = fma(rec[i * 4 + j], rhs[j], acc);
            x[i] = acc + r;
        }
        store4(cur + pop + (size_t)c * 4, x);
    };
    auto refs = [&](int pos) { return reinterpret_cast<const int4*>(fref)[pos]; };

    // this thread's first pair of the coming level: cell and face references
    int cn = 0;
    int4 nrn = make_int4(-1, -1, -1, -1);
    if (lb < le && tid < (A.bounds[lb + 1] - A.bounds[lb]) * m) {
        const int pos = A.bounds[lb] + tid / m;
        cn = order[pos];
        nrn = refs(pos);
    }
    for (int l = lb; l < le; ++l) {
        const int p0 = A.bounds[l], p1 = A.bounds[l + 1];
        const int items = (p1 - p0) * m;
        const int cc = cn;
        const int4 nrc = nrn;
        if (l + 1 < le && tid < (A.bounds[l + 2] - p1) * m) {
            const int pos = p1 + tid / m;
            cn = order[pos];
            nrn = refs(pos);
        }
        if (tid < items) solve(p0 + tid / m, tid % m, cc, nrc);
        for (int it = tid + nt; it < items; it += nt) {
            const int pos = p0 + it / m;
            solve(pos, it % m, order[pos], refs(pos));
        }
        __syncthreads();     // the next level reads this level's cells
    }
}

// ---------------------------------------------------------------------------
// ring sweep
// ---------------------------------------------------------------------------

// The current iterate is only ever read by the next few levels, so a block
// keeps its last 'ring' cells (in level order) in shared memory, and nothing
// of it goes to global memory but what other subdomains read across
// interfaces and, in the last iterate, f^{n+1} = 2 f* - f^n itself.  What a
// chunk of cells needs from global memory -- f^n, coefficient records, face
// references and the interface neighbours' values -- does not depend on the
// sweep: loader warps copy it (cp.async) kTetAhead chunks ahead, and the cell
// ids that address it as many chunks before that, so a level costs a barrier,
// shared-memory loads and the solves instead of a round of global loads.
//   A solving thread takes one cell with VPT of the block's MV variables, which
// share the record, the face references and the selection of the face's
// vertices.  The cells of a warp are consecutive (records and iterates of odd
// MV lie an odd number of 16-byte words apart: no bank conflicts), and the host
// orders a level by inflow faces, so that a warp's cells mostly take the same.
//   Measured, 32^3 cubes x 6, D3Q4, FP32, 64 subdomains: 171 us per sweep with
// the iterate in global memory, 81 us here (170 MB read).  What bounds it: with
// the solves taken out a sweep takes 46 us, with the copies taken out 68 us, with
// both out 16 us (loop and barriers): the levels' own latency, at two blocks
// of a few warps per SM.
template <typename T>
__host__ __device__ constexpr size_t tet_stage_bytes(int chunk, int mv)
{
    // records, f^n, interface values, face references, cell ids (of this chunk,
    // and of the cells and interface cells to copy later)
    return (size_t)chunk * (kTetRec * sizeof(T) + 2 * (size_t)mv * 4 * sizeof(T) + 16 + 3 * 4);
}

// 4 values, shared-memory destination
template <typename T>
__device__ __forceinline__ void tet_cp4(T* d, const T* s)
{
    cp16_g2s(d, s);
    if constexpr (sizeof(T) == 8) cp16_g2s(d + 2, s + 2);
}

template <int MV, int VPT, typename T>
__global__ void __launch_bounds__(kTetRingThreads)
    tet_ring_kernel(const __grid_constant__ TetArgs A, const T* __restrict__ prev, T* __restrict__ cur, int final,
                    int whole)
{
    extern __shared__ __align__(128) unsigned char smem_raw[];
    constexpr int NST = kTetAhead + 1;
    const int s = blockIdx.x, k = blockIdx.y, C = A.plan.chunk, R = A.plan.ring;
    const int v0 = blockIdx.z * MV, mvb = min(MV, A.m - v0);
    const int lb = A.lstart[k * (A.nsub + 1) + s], le = A.lstart[k * (A.nsub + 1) + s + 1];
    if (lb >= le) return;
    const long long nodes = A.nodes;
    const int* __restrict__ order = A.order + (size_t)k * A.ncells;
    const long long pop = (long long)(k * A.m + v0) * nodes;
    T* const fp = static_cast<T*>(A.f) + pop;
    T* const ring = reinterpret_cast<T*>(smem_raw);                     // [slot][MV][4]
    int2* const cb = reinterpret_cast<int2*>(smem_raw + (size_t)MV * R * 4 * sizeof(T));   // chunk starts
    unsigned char* const stage0 = reinterpret_cast<unsigned char*>(cb) + 16 * (size_t)A.plan.desc;
    const size_t stride = tet_stage_bytes<T>(C, MV);
    auto st_rec = [&](int q) { return reinterpret_cast<T*>(stage0 + (size_t)q * stride); };
    auto st_fn = [&](int q) { return st_rec(q) + (size_t)C * kTetRec; };        // [cell][MV][4]
    auto st_halo = [&](int q) { return st_fn(q) + (size_t)MV * C * 4; };         // [place][MV][4]
    auto st_ref = [&](int q) { return reinterpret_cast<int4*>(st_halo(q) + (size_t)MV * C * 4); };
    auto st_id = [&](int q) { return reinterpret_cast<int*>(st_ref(q) + C); };
    auto st_want = [&](int q) { return st_id(q) + C; };                          // [cell, interface cell][C]
    const int nch = le - lb;
    for (int e = threadIdx.x; e <= nch; e += blockDim.x) cb[e] = make_int2(A.bounds[lb + e], A.hstart[lb + e]);
    __syncthreads();

    constexpr int VG = (MV + VPT - 1) / VPT;          // solving threads per cell
    if ((int)threadIdx.x >= VG * C) {
        // ---- loaders ----
        const int i = threadIdx.x - VG * C, nl = blockDim.x - VG * C;
        const int* __restrict__ fref = A.fref + (size_t)k * A.ncells * 4;
        const T* __restrict__ coef = static_cast<const T*>(A.coef) + (size_t)k * A.ncells * kTetRec;
        const T* const pp = prev + pop;
        // The ids of a chunk's cells come from global memory too: they are
        // copied kTetAhead chunks before the chunk's data, by the thread that
        // will use them (its own wait makes them visible to it).
        auto fetch_ids = [&](int ch, int q) {
            if (ch < nch) {
                const int2 c0 = cb[ch], c1 = cb[ch + 1];
                if (i < c1.x - c0.x) cp_small_g2s<4>(st_want(q) + i, order + c0.x + i);
                if (i < c1.y - c0.y) cp_small_g2s<4>(st_want(q) + C + i, A.hcell + c0.y + i);
            }
        };
        auto fetch = [&](int ch, int q) {
            if (ch < nch) {
                constexpr int RW = kTetRec * (int)sizeof(T) / 16;         // 16-byte words per record
                const int2 c0 = cb[ch], c1 = cb[ch + 1];
                const int p0 = c0.x, nc = c1.x - p0;
                const T* src = coef + (size_t)p0 * kTetRec;
                T* dst = st_rec(q);
                for (int e = i; e < nc * RW; e += nl)
                    cp16_g2s(dst + e * (16 / (int)sizeof(T)), src + e * (16 / (int)sizeof(T)));
                if (i < nc) {
                    const int id = st_want(q)[i];
                    cp16_g2s(st_ref(q) + i, fref + (size_t)(p0 + i) * 4);
                    st_id(q)[i] = id;
                    T* d = st_fn(q) + i * MV * 4;
                    const T* g = fp + (size_t)(id & (kTetOutFace - 1)) * 4;
#pragma unroll
                    for (int v = 0; v < MV; ++v)
                        if (v < mvb) tet_cp4(d + v * 4, g + v * nodes);
                }
                if (i < c1.y - c0.y) {
                    T* d = st_halo(q) + i * MV * 4;
                    const T* g = pp + (size_t)st_want(q)[C + i] * 4;
#pragma unroll
                    for (int v = 0; v < MV; ++v)
                        if (v < mvb) tet_cp4(d + v * 4, g + v * nodes);
                }
            }
        };
        // groups: the ids of chunks 0 .. kTetAhead - 1; then one per chunk j,
        // with its data and the ids of chunk j + kTetAhead (into the slot that
        // chunk j's ids leave free one step later: NST slots suffice for ids
        // in flight as they do for data)
        for (int j = 0; j < kTetAhead; ++j) fetch_ids(j, j);
        cp_commit();
        cp_wait_group<0>();
        int q = 0, qi = kTetAhead;
        for (int j = 0; j < kTetAhead; ++j) {
            fetch(j, q);
            fetch_ids(j + kTetAhead, qi);
            cp_commit();
            q = q == NST - 1 ? 0 : q + 1;
            qi = qi == NST - 1 ? 0 : qi + 1;
        }
        cp_wait_group<kTetAhead - 1>();
        __syncthreads();
        for (int ch = 0; ch < nch; ++ch) {
            fetch(ch + kTetAhead, q);
            fetch_ids(ch + 2 * kTetAhead, qi);
            cp_commit();
            cp_wait_group<kTetAhead - 1>();
            __syncthreads();          // chunk ch + 1 has landed; chunk ch is solved
            q = q == NST - 1 ? 0 : q + 1;
            qi = qi == NST - 1 ? 0 : qi + 1;
        }
        return;
    }
    // ---- solvers ----
    const int vg = threadIdx.x / C, i = threadIdx.x - vg * C;
    int slot0 = 0, q = 0;
    __syncthreads();
    for (int ch = 0; ch < nch; ++ch) {
        const int nc = cb[ch + 1].x - cb[ch].x;
        if (i < nc) {
            const int word = st_id(q)[i];
            const int4 nr = st_ref(q)[i];
            const int fw[4] = {nr.x, nr.y, nr.z, nr.w};
            const T* const halo = st_halo(q);
            // every load before the first use (the block has few warps, and each
            // waits out its own latencies)
            T nb[4][VPT][4];
#pragma unroll
            for (int a = 0; a < 4; ++a)
#pragma unroll
                for (int v = 0; v < VPT; ++v)
                    if (fw[a] >= 0 && (MV % VPT == 0 || vg * VPT + v < MV))
                        load4(((fw[a] & 1) ? halo : ring) + ((fw[a] >> 7) * MV + vg * VPT + v) * 4, nb[a][v]);
            const T* const fn = st_fn(q) + (i * MV + vg * VPT) * 4;
            T u[VPT][4], rhs[VPT][4], rec[kTetRec];
#pragma unroll
            for (int v = 0; v < VPT; ++v)
                if (MV % VPT == 0 || vg * VPT + v < MV) load4(fn + v * 4, u[v]);
#pragma unroll
            for (int e = 0; e < kTetRec; e += 4) {
                T r4[4];
                load4(st_rec(q) + i * kTetRec + e, r4);
#pragma unroll
                for (int b = 0; b < 4; ++b) rec[e + b] = r4[b];
            }
#pragma unroll
            for (int v = 0; v < VPT; ++v) {
                T du[4];
#pragma unroll
                for (int b = 0; b < 4; ++b) du[b] = u[v][b] - u[v][0];
                const T sum = (du[1] + du[2]) + du[3];
                rhs[v][0] = sum;
#pragma unroll
                for (int b = 1; b < 4; ++b) rhs[v][b] = sum + du[b];
            }
#pragma unroll
            for (int a = 0; a < 4; ++a) {
                const int wd = fw[a];
                if (wd < 0) continue;
                // the neighbour's values at this cell's face vertices (j != a, ascending)
#pragma unroll
                for (int v = 0; v < VPT; ++v) {
                    T g[3];
#pragma unroll
                    for (int jj = 0; jj < 3; ++jj) {
                        const T* const nv = nb[a][v];
                        const T lo = (wd & (1 << (5 - 2 * jj))) ? nv[1] : nv[0];
                        const T hi = (wd & (1 << (5 - 2 * jj))) ? nv[3] : nv[2];
                        g[jj] = ((wd & (2 << (5 - 2 * jj))) ? hi : lo) - u[v][0];
                    }
                    const T gs = (g[0] + g[1]) + g[2];
#pragma unroll
                    for (int b = 0; b < 4; ++b)
                        if (b != a) rhs[v][b] = fma(rec[16 + a], gs + g[b < a ? b : b - 1], rhs[v][b]);
                }
            }
            int slot = slot0 + i;
            if (slot >= R) slot -= R;
            const size_t c4 = (size_t)(word & (kTetOutFace - 1)) * 4;
            const bool send = whole || (word & kTetOutFace);
#pragma unroll
            for (int v = 0; v < VPT; ++v) {
                if (MV % VPT != 0 && vg * VPT + v >= MV) break;
                T x[4], d[4];
#pragma unroll
                for (int b = 0; b < 4; ++b) {
                    d[b] = rec[b * 4] * rhs[v][0];
#pragma unroll
                    for (int j = 1; j < 4; ++j) d[b] = fma(rec[b * 4 + j], rhs[v][j], d[b]);
                    x[b] = d[b] + u[v][0];
                }
                store4(ring + (slot * MV + vg * VPT + v) * 4, x);
                if (vg * VPT + v >= mvb) continue;
                if (final) {
                    // 2 x - f^n, in FP32 without rounding x = d + f^n_0 in between (in FP64 one
                    // more operation per value costs 4% of a step)
#pragma unroll
                    for (int b = 0; b < 4; ++b)
                        x[b] = sizeof(T) == 4 ? fma(T(2), d[b], fma(T(2), u[v][0], -u[v][b])) : fma(T(2), x[b], -u[v][b]);
                    store4(fp + (vg * VPT + v) * nodes + c4, x);
                } else if (send) {
                    store4(cur + pop + (vg * VPT + v) * nodes + c4, x);
                }
            }
        }
        __syncthreads();              // chunk ch is solved; chunk ch + 1 has landed
        slot0 += nc;
        if (slot0 >= R) slot0 -= R;
        q = q == NST - 1 ? 0 : q + 1;
    }
}

template <typename T>
static const void* tet_ring_fn(int mv, int vpt)
{
    if (mv == 1 && vpt == 1) return (const void*)tet_ring_kernel<1, 1, T>;
    if constexpr (sizeof(T) == 4) {
        if (mv == 2 && vpt == 2) return (const void*)tet_ring_kernel<2, 2, T>;
        if (mv == 3 && vpt == 2) return (const void*)tet_ring_kernel<3, 2, T>;
        if (mv == 5 && vpt == 2) return (const void*)tet_ring_kernel<5, 2, T>;
        if (mv == 6 && vpt == 2) return (const void*)tet_ring_kernel<6, 2, T>;
    }
    return nullptr;
}

// The shape of a ring sweep.  One block per (subdomain, velocity) when those
// fill the SMs, so that the m variables share the records; else the variables
// are split over blocks.  Chunks as wide as the thread limit, the widest level
// and shared memory allow, where two blocks per SM (113 KB each) go before
// wider chunks when there are blocks for both: a block waits for its own
// latencies most of the time (32^3 cubes x 6, D3Q4, FP32: 64 cells and two
// blocks 4.14 ms per 15 steps, 96 cells and one block 5.17 ms).  Two variables
// per solving thread measured best of 1, 2 and 3 (5.23, 4.26, 20 ms: three
// spill).  FP64 always splits the variables: its solves are bound by the FP64
// units, not by the records' traffic (21^3 cubes, D3Q6 Euler, 8 steps: 8.3 ms
// together, 5.2 split; global iterate 8.2).  Warps are solvers or loaders as a whole: chunks are multiples of 32.
bool tet_make_plan(int ring, int width, int levels, int cells, int blocks, int m, int prec, TetPlan* plan)
{
    const size_t es = prec == 1 ? 4 : 8;
    for (int groups = 1; groups <= m; ++groups) {
        const int mv = (m + groups - 1) / groups;
        if ((m + mv - 1) / mv != groups) continue;             // the same split as fewer groups
        if (groups < m && ((long long)blocks * groups < 152 || prec == 0)) continue;
        const int vpt = std::min(mv, 2), vg = (mv + vpt - 1) / vpt;
        const int cmax = std::min(kTetRingThreads / (vg + 1) / 32 * 32, (width + 31) / 32 * 32);
        const bool two = (long long)blocks * groups > 152;
        for (int pass = two ? 0 : 1; pass < 2; ++pass)
            for (int c = cmax; c >= 32; c -= 32) {
                if (pass == 0 && c < std::min(64, cmax)) break;
                const size_t stage = prec == 1 ? tet_stage_bytes<float>(c, mv) : tet_stage_bytes<double>(c, mv);
                // chunks of a subdomain at most: one per level, one per c cells, one per
                // c interface cells (3 per cell at most); two chunk starts per 16 bytes
                const int desc = (levels + 4 * (cells / c + 1) + 2) / 2;
                const size_t sm = (size_t)mv * ring * 4 * es + 16 * (size_t)desc + (kTetAhead + 1) * stage;
                if (sm > (pass == 0 ? 113 : 227) * 1024) continue;
                plan->chunk = c;
                plan->mv = mv;
                plan->vpt = vpt;
                plan->groups = groups;
                plan->ring = ring;
                plan->desc = desc;
                plan->threads = c * (vg + 1);
                plan->smem = sm;
                return true;
            }
    }
    return false;
}

cudaError_t tet_configure(const TetPlan& plan, int prec)
{
    const void* fn = prec == 1 ? tet_ring_fn<float>(plan.mv, plan.vpt) : tet_ring_fn<double>(plan.mv, plan.vpt);
    return cudaFuncSetAttribute(fn, cudaFuncAttributeMaxDynamicSharedMemorySize, 227 * 1024);
}

// ---------------------------------------------------------------------------
// equilibria and relaxation at the nodes
// ---------------------------------------------------------------------------

// Q^a(W) of the system (Euler, scalar advection or Maxwell).
template <int SYS, typename V>
__device__ __forceinline__ void tet_flux(const TetArgs& A, const V* W, int a, V* Q)
{
    if constexpr (SYS == kAdvection) {
        Q[0] = relax_k<V>(A.rx).adv[a] * W[0];
    } else if constexpr (SYS == kMaxwell) {
        maxwell_flux(W, a, Q, V(0));
    } else {
        V ke = V(0);
#pragma unroll
        for (int b = 0; b < 3; ++b) ke = fma(W[1 + b], W[1 + b], ke);
        const V inv = V(1) / W[0];
        const V pr = relax_k<V>(A.rx).gm1 * (W[4] - V(0.5) * ke * inv);
        const V ua = W[1 + a] * inv;
        Q[0] = W[1 + a];
#pragma unroll
        for (int b = 0; b < 3; ++b) Q[1 + b] = W[1 + b] * ua + (b == a ? pr : V(0));
        Q[4] = (W[4] + pr) * ua;
    }
}

// Equilibria of all populations: D3Q6 M_{a+-} = W/6 +- Q^a/(2 lambda);
// D3Q4 (cube diagonals V_k = lambda s_k, Sec. 6.1.3)
// M_k = W/4 + sum_a s_k^a Q^a / (4 lambda), which solves eq. maxwell_def.
template <int SYS, int VS, typename V>
__device__ __forceinline__ void tet_equilibria(const TetArgs& A, const V* W, V* M)
{
    constexpr int m = nvars(3, SYS);
    V Q[3][m];
#pragma unroll
    for (int a = 0; a < 3; ++a) tet_flux<SYS>(A, W, a, Q[a]);
    if constexpr (VS == 1) {
        constexpr int sg[4][3] = {{1, 1, 1}, {1, -1, -1}, {-1, 1, -1}, {-1, -1, 1}};
        const V il = relax_k<V>(A.rx).inv4l;
#pragma unroll
        for (int k = 0; k < 4; ++k)
#pragma unroll
            for (int v = 0; v < m; ++v) {
                V q = V(sg[k][0]) * Q[0][v];
                q = fma(V(sg[k][1]), Q[1][v], q);
                q = fma(V(sg[k][2]), Q[2][v], q);
                M[k * m + v] = fma(q, il, W[v] * V(0.25));
            }
    } else {
        const V il = relax_k<V>(A.rx).inv2l;
#pragma unroll
        for (int a = 0; a < 3; ++a)
#pragma unroll
            for (int v = 0; v < m; ++v) {
                const V base = div2d<3>(W[v]);
                M[(2 * a) * m + v] = base + Q[a][v] * il;
                M[(2 * a + 1) * m + v] = base - Q[a][v] * il;
            }
    }
}

// f^{n+1} = 2 f* - f^n (EXTRAP; else f holds f^{n+1}: the ring sweep writes
// it), then W = sum_k f_k (Kahan in FP32) and the relaxation f <- omega M(W) + (1 - omega) f (eq. over_relaxation); Maxwell
// with conductivity relaxes about the equilibrium after the source step,
// f <- M(W+) + (1 - omega)(f - M(W-)).  Compiled per system and velocity
// set, so that every population stays in registers.
template <int SYS, int VS, bool EXTRAP, typename T>
__global__ void __launch_bounds__(256) tet_relax_kernel(const __grid_constant__ TetArgs A, const T* __restrict__ star)
{
    constexpr int m = nvars(3, SYS), NV = VS == 1 ? 4 : 6, NPOP = NV * m;
    T* f = static_cast<T*>(A.f);
    const long long nodes = A.nodes;
    for (long long i = blockIdx.x * (long long)blockDim.x + threadIdx.x; i < nodes;
         i += (long long)gridDim.x * blockDim.x) {
        T fk[NPOP];
#pragma unroll
        for (int p = 0; p < NPOP; ++p) {
            fk[p] = f[p * nodes + i];
            if (EXTRAP) fk[p] = fma(T(2), star[p * nodes + i], -fk[p]);
        }
        T W[m];
#pragma unroll
        for (int v = 0; v < m; ++v) {
            Acc<T> acc;
#pragma unroll
            for (int k = 0; k < NV; ++k) acc.add(fk[k * m + v]);
            W[v] = acc.s;
        }
        T Mm[NPOP];
        tet_equilibria<SYS, VS>(A, W, Mm);
        const T om = relax_k<T>(A.rx).omega, om1 = relax_k<T>(A.rx).om1;
        if constexpr (SYS == kMaxwell) {
            T Wp[m], Mp[NPOP];
#pragma unroll
            for (int v = 0; v < m; ++v) Wp[v] = v < 3 ? relax_k<T>(A.rx).mu * W[v] : W[v];
            tet_equilibria<SYS, VS>(A, Wp, Mp);
#pragma unroll
            for (int p = 0; p < NPOP; ++p) f[p * nodes + i] = fma(om1, fk[p] - Mm[p], Mp[p]);
        } else {
            if (A.rx.two) {
#pragma unroll
                for (int p = 0; p < NPOP; ++p) f[p * nodes + i] = fma(T(2), Mm[p], -fk[p]);
            } else {
#pragma unroll
                for (int p = 0; p < NPOP; ++p) f[p * nodes + i] = om * Mm[p] + om1 * fk[p];
            }
        }
    }
}

// f = M(W) from the FP64 macroscopic state (Sec. 2.2 initialisation), the
// equilibria of tet_equilibria in the arithmetic of kin_init.cuh.
template <int SYS, int VS, typename T>
__global__ void __launch_bounds__(256) tet_init_kernel(const __grid_constant__ InitArgs A,
                                                       const double* __restrict__ W0, T* __restrict__ f)
{
    constexpr int m = nvars(3, SYS);
    const long long nodes = A.nodes;
    for (long long i = blockIdx.x * (long long)blockDim.x + threadIdx.x; i < nodes;
         i += (long long)gridDim.x * blockDim.x) {
        init_node<3, SYS, T>(W0, nodes, i, A.fast, [&](const auto& W) {
            using V = std::remove_cv_t<std::remove_reference_t<decltype(W[0])>>;
            const InitK<V>& K = init_k<V>(A);
            V Q[3][m];
            float worst = init_flux<3, SYS, V>(K, W, Q);
#pragma unroll
            for (int v = 0; v < m; ++v) {
                if constexpr (VS == 1) {
                    // 1 / (4 lambda) and 1/4: halves of the constants of the axis set with d = 2
                    const V half = init_const<V>(0.5), base = W[v] * init_const<V>(0.25);
                    const V il = K.inv2l * half;
                    const V qx = Q[0][v] * il, qy = Q[1][v] * il, qz = Q[2][v] * il;
                    const V a = base + qx, b = base - qx, s = qy + qz, d = qy - qz;
                    // signs (+,+,+), (+,-,-), (-,+,-), (-,-,+)
                    const float mag = init_mag(base) + init_mag(qx) + init_mag(qy) + init_mag(qz);
                    init_put<SYS>(f[(long long)(0 * m + v) * nodes + i], a + s, mag, worst);
                    init_put<SYS>(f[(long long)(1 * m + v) * nodes + i], a - s, mag, worst);
                    init_put<SYS>(f[(long long)(2 * m + v) * nodes + i], b + d, mag, worst);
                    init_put<SYS>(f[(long long)(3 * m + v) * nodes + i], b - d, mag, worst);
                } else {
                    V base;
                    if constexpr (std::is_same<V, double>::value) base = div2d<3>(W[v]);
                    else base = W[v] * K.inv_nv;
#pragma unroll
                    for (int a = 0; a < 3; ++a) {
                        const V q = Q[a][v] * K.inv2l;
                        init_put<SYS>(f[(long long)((2 * a) * m + v) * nodes + i], base + q, init_mag(base), worst);
                        init_put<SYS>(f[(long long)((2 * a + 1) * m + v) * nodes + i], base - q, init_mag(base), worst);
                    }
                }
            }
            return worst >= 0.0f;
        });
    }
}

// Launch a (system, velocity set, precision) instance of a pointwise kernel.
template <template <int, int, typename> class K, typename... Args>
static cudaError_t tet_dispatch(const TetArgs& a, int prec, unsigned grid, cudaStream_t st, Args... args)
{
    auto go = [&](auto sys, auto vs) {
        constexpr int S = decltype(sys)::value, V = decltype(vs)::value;
        if (prec == 1) K<S, V, float>::launch(a, grid, st, args...);
        else K<S, V, double>::launch(a, grid, st, args...);
    };
    using I0 = std::integral_constant<int, 0>;
    using I1 = std::integral_constant<int, 1>;
    using I2 = std::integral_constant<int, 2>;
    const bool d3q4 = a.velset == 1;
    switch (a.system) {
    case kAdvection: d3q4 ? go(I0{}, I1{}) : go(I0{}, I0{}); break;
    case kEuler: d3q4 ? go(I1{}, I1{}) : go(I1{}, I0{}); break;
    default: d3q4 ? go(I2{}, I1{}) : go(I2{}, I0{}); break;
    }
    return cudaGetLastError();
}

template <int S, int V, typename T>
struct RelaxLaunch {
    static void launch(const TetArgs& a, unsigned grid, cudaStream_t st, const void* star)
    {
        if (star) tet_relax_kernel<S, V, true, T><<<grid, 256, 0, st>>>(a, static_cast<const T*>(star));
        else tet_relax_kernel<S, V, false, T><<<grid, 256, 0, st>>>(a, nullptr);
    }
};

template <int S, int V, typename T>
struct InitLaunch {
    static void launch(const TetArgs& a, unsigned grid, cudaStream_t st, const double* W)
    {
        const InitArgs A = init_args(a.nodes, 3, a.lambda, a.gamma, a.adv);
        tet_init_kernel<S, V, T><<<grid, 256, 0, st>>>(A, W, static_cast<T*>(a.f));
    }
};

cudaError_t tet_launch_setup(const TetSetupArgs& a, cudaStream_t st)
{
    const long long n = (long long)a.ncells * a.nvel;
    tet_setup_kernel<<<(unsigned)((n + 127) / 128), 128, 0, st>>>(a);
    return cudaGetLastError();
}

cudaError_t tet_launch_sweep(const TetArgs& a, const void* prev, void* cur, int final, int whole, int prec,
                             cudaStream_t st)
{
    if (a.plan.chunk > 0) {
        void* args[] = {(void*)&a, (void*)&prev, (void*)&cur, (void*)&final, (void*)&whole};
        return cudaLaunchKernel(prec == 1 ? tet_ring_fn<float>(a.plan.mv, a.plan.vpt) : tet_ring_fn<double>(a.plan.mv, a.plan.vpt),
                                dim3(a.nsub, a.nvel, a.plan.groups), dim3(a.plan.threads), args, a.plan.smem, st);
    }
    const dim3 grid(a.nsub, a.nvel);
    if (prec == 1)
        tet_sweep_kernel<float><<<grid, kTetSweepThreads, 0, st>>>(a, static_cast<const float*>(prev),
                                                                  static_cast<float*>(cur));
    else
        tet_sweep_kernel<double><<<grid, kTetSweepThreads, 0, st>>>(a, static_cast<const double*>(prev),
                                                                   static_cast<double*>(cur));
    return cudaGetLastError();
}

cudaError_t tet_launch_relax(const TetArgs& a, const void* star, int prec, cudaStream_t st)
{
    const unsigned grid = (unsigned)std::min<long long>((a.nodes + 255) / 256, 152LL * 8);
    return tet_dispatch<RelaxLaunch>(a, prec, grid, st, star);
}

cudaError_t tet_launch_init(const TetArgs& a, const double* W, int prec, cudaStream_t st)
{
    const unsigned grid = (unsigned)std::min<long long>((a.nodes + 255) / 256, 152LL * 8);
    return tet_dispatch<InitLaunch>(a, prec, grid, st, W);
}

}  // namespace kin
