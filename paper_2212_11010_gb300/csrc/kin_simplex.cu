// kin_simplex.cu -- the paper's d + 1 velocity sets (D2Q3, Sec. 2.4; D3Q4,
// Sec. 6.1.3).  Their velocities are not aligned with the mesh: a cell has an
// inflow face on every axis with V_a != 0, the downwind order is a true
// anti-diagonal wavefront (Sec. 3.2), and subdomains meet at corners
// (Sec. 5.1, the three-iteration case).  The transport is done by the
// subdomain iteration of eq. ibvp as written, K sweeps per step:
//   sweep        one launch per iterate (per velocity when a velocity alone
//                fills the GPU): a thread block streams (variable, subdomain)
//                problems through the subdomain's columns, one cell per lane
//                and wave, lanes skewed so that every upwind neighbour is done
//                the wave before (sx_sweep_velocity); each cell solves its
//                full local block (eq. dg_imp, CN half step) with inflow from
//                its own previous cell, the neighbouring lane, or across the
//                interface (f^n on iterate 1, else the previous iterate's
//                traces); downwind boundary cells write this iterate's traces;
//                the last iterate writes f^{n+1} = 2 f* - f^n; with K = 1 a
//                trace pass first copies iterate 0;
//   relaxation   W = sum_k f_k and f_k <- omega M_k(W) + (1 - omega) f_k with
//                M from the moment system eq. maxwell_def (its inverse is
//                precomputed in FP64).
// Two forms take the sweep's place in FP32: bricks of 2 x 2 x 2 cells per lane
// (3D, degree 1, large meshes; sx_brick_velocity), and in 2D a chain over the
// outflow nodes alone between two passes over all cells at once (SxSplit).
#include "kin_aux.h"
#include "kin_device.cuh"
#include "kin_init.cuh"
#include "kin_tma.cuh"

#include <math.h>
#include <string.h>

#include <algorithm>
#include <type_traits>

namespace kin {

// ---------------------------------------------------------------------------
// FP64 preprocessing: velocity, block inverse and face operators per velocity
// ---------------------------------------------------------------------------

__device__ static void sx_velocity(int dim, int k, double lam, double V[3])
{
    V[0] = V[1] = V[2] = 0.0;
    if (dim == 2) {
        V[0] = lam * cos(2.0 * M_PI * k / 3.0);
        V[1] = lam * sin(2.0 * M_PI * k / 3.0);
    } else {
        const double s[4][3] = {{1, 1, 1}, {1, -1, -1}, {-1, 1, -1}, {-1, -1, 1}};
        for (int a = 0; a < 3; ++a) V[a] = lam * s[k][a];
    }
}

__device__ static void sx_gll(int p, double* xi, double* w)
{
    for (int j = 0; j <= p; ++j) {
        double x = -cos(M_PI * j / p);
        double Pv = 1.0;
        if (j > 0 && j < p) {
            for (int it = 0; it < 60; ++it) {
                double a = 1.0, b = x;
                for (int k = 1; k < p; ++k) {
                    double c = ((2 * k + 1) * x * b - k * a) / (k + 1);
                    a = b;
                    b = c;
                }
                double dP = p * (a - x * b) / (1.0 - x * x);
                double d2P = (2.0 * x * dP - p * (p + 1.0) * b) / (1.0 - x * x);
                double step = dP / d2P;
                x -= step;
                if (fabs(step) < 1e-17) break;
            }
            double a = 1.0, b = x;
            for (int k = 1; k < p; ++k) {
                double c = ((2 * k + 1) * x * b - k * a) / (k + 1);
                a = b;
                b = c;
            }
            Pv = b;
        } else {
            Pv = (j == 0 && (p % 2)) ? -1.0 : 1.0;
        }
        xi[j] = (j == 0) ? 0.0 : (j == p ? 1.0 : 0.5 * (x + 1.0));
        w[j] = 1.0 / (p * (p + 1.0) * Pv * Pv);
    }
}

// One thread per velocity.  Record layout (NN^2 + NN + d TN elements):
//   [0, NN*NN)                 A^{-1}   (row-major)
//   [NN*NN, NN*NN + NN)        W_cell   (tensor Gauss-Lobatto weights)
//   [NN*NN + NN + a*TN, ...)   nu_a W_perp on the inflow face of axis a (0 if V_a = 0)
// with A = W_cell + sum_a nu_a (S_a at axis a, W at the others),
// S_a = Q + e_0 e_0^T (V_a > 0) or -Q + e_p e_p^T (V_a < 0), nu_a = |V_a| dt / (2 h_a),
// so that the CN half step of eq. dg_imp is f* = A^{-1} (W_cell f^n + sum_a nu_a E_a W_perp tr_a),
// E_a the injection onto the inflow face nodes of axis a.
// Thread 0 also writes the inverse of the moment matrix [1...1; V_0 ... V_d].
__global__ void sx_setup_kernel(SxSetupArgs A)
{
    const int k = threadIdx.x;
    const int d = A.dim, p = A.degree, np = p + 1;
    int nn = 1, tn = 1;
    for (int a = 0; a < d; ++a) nn *= np;
    for (int a = 1; a < d; ++a) tn *= np;
    double xi[kMaxNP], w[kMaxNP];
    sx_gll(p, xi, w);
    if (k == 0) {
        // moment matrix and its inverse (Gauss-Jordan), nvel = d + 1
        const int nv = d + 1;
        double M[4][8];
        for (int j = 0; j < nv; ++j) {
            double V[3];
            sx_velocity(d, j, A.lambda, V);
            M[0][j] = 1.0;
            for (int a = 0; a < d; ++a) M[1 + a][j] = V[a];
        }
        for (int i = 0; i < nv; ++i)
            for (int j = 0; j < nv; ++j) M[i][nv + j] = (i == j) ? 1.0 : 0.0;
        for (int c = 0; c < nv; ++c) {
            int piv = c;
            for (int r = c + 1; r < nv; ++r)
                if (fabs(M[r][c]) > fabs(M[piv][c])) piv = r;
            for (int j = 0; j < 2 * nv; ++j) {
                double t = M[c][j];
                M[c][j] = M[piv][j];
                M[piv][j] = t;
            }
            const double inv = 1.0 / M[c][c];
            for (int j = 0; j < 2 * nv; ++j) M[c][j] *= inv;
            for (int r = 0; r < nv; ++r)
                if (r != c) {
                    const double l = M[r][c];
                    for (int j = 0; j < 2 * nv; ++j) M[r][j] -= l * M[c][j];
                }
        }
        for (int i = 0; i < nv; ++i)
            for (int j = 0; j < nv; ++j) A.minv[i * nv + j] = M[i][nv + j];
    }
    if (k > d) return;
    double V[3];
    sx_velocity(d, k, A.lambda, V);
    // 1D pieces
    double bw[kMaxNP], Dm[kMaxNP][kMaxNP];
    for (int i = 0; i < np; ++i) {
        double prod = 1.0;
        for (int j = 0; j < np; ++j)
            if (j != i) prod *= xi[i] - xi[j];
        bw[i] = 1.0 / prod;
    }
    for (int i = 0; i < np; ++i) {
        double diag = 0.0;
        for (int j = 0; j < np; ++j) {
            if (j == i) continue;
            Dm[i][j] = (bw[j] / bw[i]) / (xi[i] - xi[j]);
            diag -= Dm[i][j];
        }
        Dm[i][i] = diag;
    }
    double S[3][kMaxNP][kMaxNP], nu[3];
    for (int a = 0; a < d; ++a) {
        nu[a] = fabs(V[a]) * 0.5 * A.dt / A.h[a];
        for (int i = 0; i < np; ++i)
            for (int j = 0; j < np; ++j) {
                const double q = w[i] * Dm[i][j];
                double v = 0.0;
                if (V[a] > 0) v = q + ((i == 0 && j == 0) ? 1.0 : 0.0);
                else if (V[a] < 0) v = -q + ((i == p && j == p) ? 1.0 : 0.0);
                S[a][i][j] = v;
            }
    }
    // assemble A (nn x nn) and invert; node index = ix + np iy + np^2 iz
    double* Mx = A.work + (size_t)k * 2 * kSxMaxNN * kSxMaxNN;   // [nn][2nn]
    const int w2 = 2 * nn;
    for (int i = 0; i < nn; ++i) {
        int ii[3] = {i % np, (i / np) % np, i / (np * np)};
        for (int j = 0; j < nn; ++j) {
            int jj[3] = {j % np, (j / np) % np, j / (np * np)};
            bool diag = true;
            double wprod = 1.0;
            for (int b = 0; b < d; ++b) {
                if (ii[b] != jj[b]) diag = false;
                wprod *= w[ii[b]];
            }
            double v = diag ? wprod : 0.0;
            for (int a = 0; a < d; ++a) {
                bool same = true;
                double wt = 1.0;
                for (int b = 0; b < d; ++b) {
                    if (b == a) continue;
                    if (ii[b] != jj[b]) same = false;
                    wt *= w[ii[b]];
                }
                if (same) v += nu[a] * S[a][ii[a]][jj[a]] * wt;
            }
            Mx[i * w2 + j] = v;
            Mx[i * w2 + nn + j] = (i == j) ? 1.0 : 0.0;
        }
    }
    for (int c = 0; c < nn; ++c) {
        int piv = c;
        for (int r = c + 1; r < nn; ++r)
            if (fabs(Mx[r * w2 + c]) > fabs(Mx[piv * w2 + c])) piv = r;
        if (piv != c)
            for (int j = 0; j < w2; ++j) {
                const double t = Mx[c * w2 + j];
                Mx[c * w2 + j] = Mx[piv * w2 + j];
                Mx[piv * w2 + j] = t;
            }
        const double inv = 1.0 / Mx[c * w2 + c];
        for (int j = 0; j < w2; ++j) Mx[c * w2 + j] *= inv;
        for (int r = 0; r < nn; ++r) {
            if (r == c) continue;
            const double l = Mx[r * w2 + c];
            if (l != 0.0)
                for (int j = 0; j < w2; ++j) Mx[r * w2 + j] -= l * Mx[c * w2 + j];
        }
    }
    double* rec = A.c64 + (size_t)k * A.stride;
    for (int i = 0; i < nn; ++i)
        for (int j = 0; j < nn; ++j) rec[i * nn + j] = Mx[i * w2 + nn + j];
    for (int j = 0; j < nn; ++j) {
        int jj[3] = {j % np, (j / np) % np, j / (np * np)};
        double wj = 1.0;
        for (int b = 0; b < d; ++b) wj *= w[jj[b]];
        rec[nn * nn + j] = wj;
    }
    for (int a = 0; a < d; ++a)
        for (int t = 0; t < tn; ++t) {
            // transverse node t enumerates the other axes, lowest first
            double wt = 1.0;
            int r = t;
            for (int b = 0; b < d; ++b) {
                if (b == a) continue;
                wt *= w[r % np];
                r /= np;
            }
            rec[nn * nn + nn + a * tn + t] = V[a] == 0.0 ? 0.0 : nu[a] * wt;
        }
}

// ---------------------------------------------------------------------------
// trace pass and sweeps
// ---------------------------------------------------------------------------

// Global line id of the face node (transverse cell, transverse node) of axis a.
__device__ __forceinline__ long long sx_gline(const SxArgs& S, int a, const int c[3], const int j[3], int np)
{
    int t1 = -1, t2 = -1;
    for (int b = 0; b < S.dim; ++b) {
        if (b == a) continue;
        if (t1 < 0) t1 = b;
        else t2 = b;
    }
    long long gt = 0, tnode = 0;
    if (t2 >= 0) {
        gt = (long long)c[t2] * S.n[t1] + c[t1];
        tnode = j[t1] + np * j[t2];
    } else if (t1 >= 0) {
        gt = c[t1];
        tnode = j[t1];
    }
    long long tn = 1;
    for (int b = 1; b < S.dim; ++b) tn *= np;
    return gt * tn + tnode;
}

// Iterate 0 of eq. ibvp: the f^n values on the outflow face of every
// subdomain's downwind boundary, per (population, axis with V_a != 0).
template <typename T>
__global__ void sx_trace0_kernel(SxArgs S)
{
    const int np = S.degree + 1;
    const T* f = static_cast<const T*>(S.f);
    for (long long e = blockIdx.x * (long long)blockDim.x + threadIdx.x; e < S.trace_total;
         e += (long long)gridDim.x * blockDim.x) {
        long long r = e;
        int pop = 0, a = 0;
        // entries: pop-major, then axis, then [NS_a][glines_a]
        for (;;) {
            const int k = pop / S.m;
            bool done = false;
            for (a = 0; a < S.dim; ++a) {
                if (S.vsgn[k][a] == 0) continue;
                const long long cnt = (long long)S.NS[a] * S.glines[a];
                if (r < cnt) {
                    done = true;
                    break;
                }
                r -= cnt;
            }
            if (done) break;
            ++pop;
        }
        const int k = pop / S.m, sg = S.vsgn[k][a];
        const int sa = (int)(r / S.glines[a]);
        const long long gl = r % S.glines[a];
        // decode gline -> transverse cell and node
        long long tn = 1;
        for (int b = 1; b < S.dim; ++b) tn *= np;
        const long long gt = gl / tn;
        const int tnode = (int)(gl % tn);
        int c[3] = {0, 0, 0}, j[3] = {0, 0, 0};
        int t1 = -1, t2 = -1;
        for (int b = 0; b < S.dim; ++b) {
            if (b == a) continue;
            if (t1 < 0) t1 = b;
            else t2 = b;
        }
        if (t2 >= 0) {
            c[t1] = (int)(gt % S.n[t1]);
            c[t2] = (int)(gt / S.n[t1]);
            j[t1] = tnode % np;
            j[t2] = tnode / np;
        } else if (t1 >= 0) {
            c[t1] = (int)gt;
            j[t1] = tnode;
        }
        c[a] = sa * S.L[a] + (sg > 0 ? S.L[a] - 1 : 0);
        j[a] = sg > 0 ? np - 1 : 0;
        const long long cell = ((long long)c[2] * S.n[1] + c[1]) * S.n[0] + c[0];
        const int node = j[0] + np * j[1] + np * np * j[2];
        T* out = static_cast<T*>(S.tr_out[a]);
        out[(long long)pop * S.NS[a] * S.glines[a] + r] = f[(long long)pop * S.nodes + cell * S.nn + node];
    }
}

// Sign of V_k along axis a for the d + 1 sets (D2Q3: 0, 120 and 240 degrees;
// D3Q4: the cube diagonals (1,1,1), (1,-1,-1), (-1,1,-1), (-1,-1,1)).
__host__ __device__ constexpr int sx_sign(int D, int k, int a)
{
    if (D == 2) {
        if (a == 0) return k == 0 ? 1 : -1;
        if (a == 1) return k == 0 ? 0 : (k == 1 ? 1 : -1);
        return 0;
    }
    if (a == 0) return k < 2 ? 1 : -1;
    if (a == 1) return (k == 0 || k == 2) ? 1 : -1;
    if (a == 2) return (k == 0 || k == 3) ? 1 : -1;
    return 0;
}

// Cell node with index ja along axis a and transverse node tt (the other
// axes, lowest first); node = j0 + NP j1 + NP^2 j2.
template <int D, int NP>
__host__ __device__ constexpr int sx_node(int a, int ja, int tt)
{
    int j[3] = {0, 0, 0};
    int r = tt;
    for (int b = 0; b < D; ++b) {
        if (b == a) continue;
        j[b] = r % NP;
        r /= NP;
    }
    j[a] = ja;
    return j[0] + NP * j[1] + NP * NP * j[2];
}

// Division by an invariant divisor d >= 1 for dividends below 2^31
// (Granlund and Montgomery, "Division by invariant integers using
// multiplication", 1994, the round-up multiplier): l = ceil(log2 d),
// m = floor(2^32 (2^l - d) / d) + 1, q = (mulhi(m, n) + n) >> l.
struct SxDiv {
    unsigned m;
    int l;
};

static inline SxDiv sx_div_make(int d)
{
    SxDiv r;
    int l = 0;
    while ((1LL << l) < d) ++l;
    r.l = l;
    r.m = (unsigned)((((1ULL << 32) * ((1ULL << l) - (unsigned long long)d)) / (unsigned long long)d) + 1);
    return r;
}

__device__ __forceinline__ int sx_div(int n, SxDiv d)
{
    return (int)(((unsigned long long)__umulhi(d.m, (unsigned)n) + (unsigned)n) >> d.l);
}

// Launch parameters of one sweep.  The block inverse, the cell weights and
// the face weights of every velocity travel in the parameter block, so the
// fully unrolled cell solve takes them as constant-bank operands.
template <int D, int P, typename T>
struct SxWave {
    static constexpr int NP = P + 1, NN = ipow(NP, D), TN = ipow(NP, D - 1), NV = D + 1;
    SxArgs S;
    int bpv;            // thread blocks per velocity
    int k0;             // first velocity of this launch
    SxDiv div_nsub, div_ns0, div_ns1;
    // The records are operands from the constant bank, and where they begin matters (56
    // unused bytes, without -> with: 2D p = 3 FP32 310 -> 255 us per step of 512^2 cells
    // (K = 1), 3D p = 2 FP32 3.25 -> 3.13 ms of 24^3, 3D p = 1 FP64 0.988 -> 0.966 of 32^3;
    // but the bricks 26.91 -> 27.04 of 128^3, 12 steps).
    int fill[D == 3 && P == 1 && sizeof(T) == 4 ? 0 : 14];
    T ainv[NV][NN * NN];
    T wcell[NN];
    T face[NV][D][TN];
};

// Prefetch rings of the sweep, filled by cp.async kSxRing - 1 waves ahead:
// per lane and wave, the cell's f^n (NN values) and its interface inflow
// along the stepping axis (TN values); per wave and boundary lane of a
// transverse axis, that axis' interface inflow (TN values).  Each lane owns
// NEP contiguous elements per variable and slot (NEP = NN + TN rounded up so
// that NEP / CW is odd: lanes then fall in distinct banks for scalar (CW = 1)
// and 16-byte (CW > 1) accesses).  The exchange of outflow faces between
// lanes uses the same rule with TN.
__host__ __device__ constexpr int sx_pad_odd(int n, int cw)
{
    return ((n + cw - 1) / cw) % 2 ? (n + cw - 1) / cw * cw : ((n + cw - 1) / cw + 1) * cw;
}

template <int D, int P, typename T>
struct SxRing {
    static constexpr int NN = ipow(P + 1, D), TN = ipow(P + 1, D - 1);
    static constexpr int C = 16 / (int)sizeof(T);
    static constexpr int CW = (NN % C == 0 && TN % C == 0) ? C : 1;
    static constexpr int NEP = sx_pad_odd(NN + TN, CW);   // f^n of the cell + inflow along DEP
    static constexpr int TNP = sx_pad_odd(TN, CW);
};
constexpr int kSxRing = 2;            // slots; waves in flight = kSxRing - 1

// Position of one lane in the stream of problems: q counts the lane's cells
// (q = wave - skew), od is the oriented coordinate along the stepping axis.
struct SxTrack {
    int q, od, i, pop;
    int s[3], g[3];
    bool valid;
};

template <int NN, typename T>
__device__ __forceinline__ void sx_st(T* p, const T* u)
{
    if constexpr ((NN * sizeof(T)) % 16 == 0) {
        if constexpr (sizeof(T) == 4) {
#pragma unroll
            for (int k = 0; k < NN / 4; ++k)
                reinterpret_cast<float4*>(p)[k] = make_float4(u[4 * k], u[4 * k + 1], u[4 * k + 2], u[4 * k + 3]);
        } else {
#pragma unroll
            for (int k = 0; k < NN / 2; ++k) reinterpret_cast<double2*>(p)[k] = make_double2(u[2 * k], u[2 * k + 1]);
        }
    } else {
#pragma unroll
        for (int i = 0; i < NN; ++i) p[i] = u[i];
    }
}

// N values from / to shared memory, 16 bytes at a time when VEC (the address
// is then 16-byte aligned and N a multiple of 16 / sizeof(T)).
template <int N, bool VEC, typename T>
__device__ __forceinline__ void sx_lds(const T* p, T* v)
{
    if constexpr (VEC && sizeof(T) == 4) {
#pragma unroll
        for (int k = 0; k < N / 4; ++k) {
            const float4 q = reinterpret_cast<const float4*>(p)[k];
            v[4 * k] = q.x;
            v[4 * k + 1] = q.y;
            v[4 * k + 2] = q.z;
            v[4 * k + 3] = q.w;
        }
    } else if constexpr (VEC) {
#pragma unroll
        for (int k = 0; k < N / 2; ++k) {
            const double2 q = reinterpret_cast<const double2*>(p)[k];
            v[2 * k] = q.x;
            v[2 * k + 1] = q.y;
        }
    } else {
#pragma unroll
        for (int i = 0; i < N; ++i) v[i] = p[i];
    }
}

template <int N, bool VEC, typename T>
__device__ __forceinline__ void sx_sts(T* p, const T* v)
{
    if constexpr (VEC && sizeof(T) == 4) {
#pragma unroll
        for (int k = 0; k < N / 4; ++k)
            reinterpret_cast<float4*>(p)[k] = make_float4(v[4 * k], v[4 * k + 1], v[4 * k + 2], v[4 * k + 3]);
    } else if constexpr (VEC) {
#pragma unroll
        for (int k = 0; k < N / 2; ++k) reinterpret_cast<double2*>(p)[k] = make_double2(v[2 * k], v[2 * k + 1]);
    } else {
#pragma unroll
        for (int i = 0; i < N; ++i) p[i] = v[i];
    }
}

// Transverse cell id of the face of axis a (the other axes, lowest first).
template <int D>
__device__ __forceinline__ int sx_face_cell(const SxArgs& S, int a, const int g[3])
{
    if (D == 2) return a == 0 ? g[1] : g[0];
    const int b1 = a == 0 ? 1 : 0, b2 = a == 2 ? 1 : 2;
    return g[b2] * S.n[b1] + g[b1];
}

template <int D, int KV>
__device__ __forceinline__ constexpr int sx_sg(int a)
{
    return a == 0 ? sx_sign(D, KV, 0) : (a == 1 ? sx_sign(D, KV, 1) : sx_sign(D, KV, 2));
}

// One velocity's part of a sweep (iterate it of eq. ibvp).  A thread block
// streams the problems (variable, subdomain) lb, lb + bpv, ... of velocity
// KV.  Its lanes are the subdomain's columns along the stepping axis DEP (the last axis with
// V_a != 0), indexed by the oriented transverse coordinates; lane o visits
// its column's cells one per wave, delayed by skew = sum of its oriented
// transverse coordinates, so that at every wave the cell of each lane has its
// upwind neighbours (Sec. 3.2) already done: along DEP the lane's own previous
// cell, along a transverse axis the previous wave of the neighbouring lane,
// which passes its outflow face through shared memory.  Consecutive
// problems follow each other in the column without a gap, so every lane is
// busy except during the first and last skew waves.  Cells on a subdomain's
// upwind boundary take their inflow from the previous iterate's traces (from
// f^n itself on iterate 1); cells on its downwind boundary write this
// iterate's traces.  The cell solve is the CN half step of eq. dg_imp in
// shifted form: with t = f^n at node 0,
//   f* = t + A^{-1} (W_cell (f^n - t) + sum_a nu_a E_a W_perp (tr_a - t)),
// which keeps constant states exactly.  The last iterate writes
// f^{n+1} = 2 f* - f^n in place.
template <int D, int P, int KV, typename T>
__device__ __forceinline__ void sx_sweep_velocity(const SxWave<D, P, T>& A, const int lb, T* xs, T* ring)
{
    constexpr int NP = P + 1, NN = ipow(NP, D), TN = ipow(NP, D - 1);
    using RG = SxRing<D, P, T>;
    constexpr int CW = RG::CW, NEP = RG::NEP, TNP = RG::TNP;
    constexpr int PF = kSxRing - 1;
    constexpr int DEP = D == 3 ? 2 : (KV == 0 ? 0 : 1);
    constexpr int TA0 = D == 3 ? 0 : 1 - DEP;
    constexpr int TA1 = D == 3 ? 1 : 0;          // only used when D == 3
    constexpr bool X0 = sx_sign(D, KV, TA0) != 0;
    constexpr bool X1 = D == 3 && sx_sign(D, KV, TA1) != 0;
    constexpr int SGD = sx_sign(D, KV, DEP);
    // node 0 receives face inflow iff some axis enters at index 0
    constexpr bool R0 = sx_sign(D, KV, 0) > 0 || sx_sign(D, KV, 1) > 0 || sx_sign(D, KV, 2) > 0;

    const SxArgs& S = A.S;
    const int tid = threadIdx.x, nt = blockDim.x;
    const int n0 = S.L[TA0], n1 = D == 3 ? S.L[TA1] : 1;
    const int Ld = S.L[DEP];
    const bool active = tid < n0 * n1;
    const int ot1 = D == 3 ? tid / n0 : 0, ot0 = tid - ot1 * n0;
    const int lt0 = sx_sign(D, KV, TA0) < 0 ? n0 - 1 - ot0 : ot0;
    const int lt1 = (D == 3 && sx_sign(D, KV, TA1) < 0) ? n1 - 1 - ot1 : ot1;
    const int skew = (X0 ? ot0 : 0) + (X1 ? ot1 : 0);
    const int maxskew = (X0 ? n0 - 1 : 0) + (X1 ? n1 - 1 : 0);
    const int nsub = S.NS[0] * S.NS[1] * S.NS[2];
    const int nprob = S.m * nsub;                // (variable, subdomain)
    const int nb = lb < nprob ? (nprob - lb + A.bpv - 1) / A.bpv : 0;
    const int span = nb * Ld;
    const int total = nb > 0 ? span + maxskew : 0;
    T* f = static_cast<T*>(S.f);

    auto advance = [&](SxTrack& t) {
        ++t.q;
        t.valid = false;
        if (t.q < 0 || t.q >= span) return;
        bool fresh = false;
        if (t.q == 0) {
            t.od = 0;
            t.i = 0;
            fresh = true;
        } else if (++t.od == Ld) {
            t.od = 0;
            ++t.i;
            fresh = true;
        }
        if (fresh) {
            const int pid = lb + t.i * A.bpv;
            const int v = sx_div(pid, A.div_nsub), s = pid - v * nsub;
            const int s12 = sx_div(s, A.div_ns0), s2 = sx_div(s12, A.div_ns1);
            t.pop = KV * S.m + v;
            t.s[0] = s - s12 * S.NS[0];
            t.s[1] = s12 - s2 * S.NS[1];
            t.s[2] = s2;
            t.g[TA0] = t.s[TA0] * S.L[TA0] + lt0;
            if (D == 3) t.g[TA1] = t.s[TA1] * S.L[TA1] + lt1;
            else t.g[2] = 0;
        }
        t.g[DEP] = t.s[DEP] * Ld + (SGD < 0 ? Ld - 1 - t.od : t.od);
        t.valid = active;
    };

    // interface inflow is needed on the upwind boundary of the subdomain
    auto at_inflow = [&](const SxTrack& t, int a) {
        return a == DEP ? t.od == 0 : (a == TA0 ? ot0 == 0 : ot1 == 0);
    };
    auto at_outflow = [&](const SxTrack& t, int a) {
        return a == DEP ? t.od == Ld - 1 : (a == TA0 ? ot0 == n0 - 1 : ot1 == n1 - 1);
    };
    // this lane's elements in ring slot r
    auto slot = [&](int r) -> T* { return ring + (r * nt + tid) * NEP; };
    // transverse inflow of boundary lane b of axis ax in slot r
    T* tring = ring + kSxRing * nt * NEP;
    const int nbm = D == 2 ? 1 : (n0 > n1 ? n0 : n1);
    auto tslot = [&](int r, int ax, int b) -> T* { return tring + ((r * 2 + ax) * nbm + b) * TNP; };
    const int bidx0 = ot1, bidx1 = ot0;          // boundary index of this lane on TA0 / TA1
    // exchange [parity][axis][lane][TNP]
    auto xslot = [&](int par, int ax) -> T* { return xs + ((par * 2 + ax) * nt + tid) * TNP; };

    // issue the copies of the wave tracked by t into ring slot r
    auto fetch = [&](const SxTrack& t, int r) {
        if (t.valid) {
            T* dst = slot(r);
            const int cell = (t.g[2] * S.n[1] + t.g[1]) * S.n[0] + t.g[0];
            const T* src = f + (long long)t.pop * S.nodes + (long long)cell * NN;
            if constexpr (CW > 1) {
#pragma unroll
                for (int e = 0; e < NN; e += CW) cp16_g2s(dst + e, src + e);
            } else {
#pragma unroll
                for (int e = 0; e < NN; ++e) cp_small_g2s<sizeof(T)>(dst + e, src + e);
            }
#pragma unroll
            for (int a = 0; a < D; ++a) {
                const int sg = sx_sg<D, KV>(a);
                if (sg == 0 || !at_inflow(t, a)) continue;
                T* dbase = a == DEP ? dst + NN : tslot(r, a == TA0 ? 0 : 1, a == TA0 ? bidx0 : bidx1);
                if (S.from_f) {
                    // iterate 0 of eq. ibvp: f^n on the outflow face of the upwind cell
                    int gu[3] = {t.g[0], t.g[1], t.g[2]};
                    gu[a] -= sg;
                    if (gu[a] < 0) gu[a] += S.n[a];
                    if (gu[a] >= S.n[a]) gu[a] -= S.n[a];
                    const T* up = f + (long long)t.pop * S.nodes
                        + (long long)((gu[2] * S.n[1] + gu[1]) * S.n[0] + gu[0]) * NN;
                    const int out = sg > 0 ? P : 0;
#pragma unroll
                    for (int tt = 0; tt < TN; ++tt)
                        cp_small_g2s<sizeof(T)>(dbase + tt, up + sx_node<D, NP>(a, out, tt));
                } else {
                    int sup = t.s[a] - sg;
                    if (sup < 0) sup += S.NS[a];
                    if (sup >= S.NS[a]) sup -= S.NS[a];
                    const T* tr = static_cast<const T*>(S.tr_in[a]) + ((long long)t.pop * S.NS[a] + sup) * S.glines[a]
                        + (long long)sx_face_cell<D>(S, a, t.g) * TN;
                    if constexpr (CW > 1) {
#pragma unroll
                        for (int tt = 0; tt < TN; tt += CW) cp16_g2s(dbase + tt, tr + tt);
                    } else {
#pragma unroll
                        for (int tt = 0; tt < TN; ++tt) cp_small_g2s<sizeof(T)>(dbase + tt, tr + tt);
                    }
                }
            }
        }
        cp_commit();
    };

    T pd[TN];                                   // own outflow face along DEP (previous wave)
#pragma unroll
    for (int tt = 0; tt < TN; ++tt) pd[tt] = T(0);

    auto compute = [&](int W, const SxTrack& t, int rs) {
        if (!t.valid) return;
        const int par = W & 1;
        const T* sl = slot(rs);
        // where each axis' inflow comes from: the interface (ring), the own
        // previous cell (registers) or the upwind lane (exchange)
        const T* isrc[3] = {nullptr, nullptr, nullptr};
        bool fromreg[3] = {false, false, false};
#pragma unroll
        for (int a = 0; a < D; ++a) {
            const int sg = sx_sg<D, KV>(a);
            if (sg == 0) continue;
            if (a == DEP) {
                if (at_inflow(t, a)) isrc[a] = sl + NN;
                else fromreg[a] = true;
            } else {
                const int ax = a == TA0 ? 0 : 1;
                isrc[a] = at_inflow(t, a) ? tslot(rs, ax, ax == 0 ? bidx0 : bidx1)
                                          : xslot(par ^ 1, ax) - (a == TA0 ? 1 : n0) * TNP;
            }
        }
        T u[NN];
        sx_lds<NN, (CW > 1)>(sl, u);
        const T tref = u[0];
        T r[NN];
        r[0] = T(0);
#pragma unroll
        for (int j = 1; j < NN; ++j) r[j] = A.wcell[j] * (u[j] - tref);
#pragma unroll
        for (int a = 0; a < D; ++a) {
            const int sg = sx_sg<D, KV>(a);
            if (sg == 0) continue;
            const int in = sg > 0 ? 0 : P;
            T tv[TN];
            if (a == DEP && fromreg[a]) {
#pragma unroll
                for (int tt = 0; tt < TN; ++tt) tv[tt] = pd[tt];
            } else {
                sx_lds<TN, (CW > 1)>(isrc[a], tv);
            }
#pragma unroll
            for (int tt = 0; tt < TN; ++tt) {
                const int j = sx_node<D, NP>(a, in, tt);
                r[j] = fma(A.face[KV][a][tt], tv[tt] - tref, r[j]);
            }
        }
        // x = A^{-1} r by columns: each step is NN independent FMAs
        T x[NN];
#pragma unroll
        for (int i = 0; i < NN; ++i) x[i] = R0 ? A.ainv[KV][i * NN] * r[0] : A.ainv[KV][i * NN + 1] * r[1];
#pragma unroll
        for (int j = R0 ? 1 : 2; j < NN; ++j)
#pragma unroll
            for (int i = 0; i < NN; ++i) x[i] = fma(A.ainv[KV][i * NN + j], r[j], x[i]);
#pragma unroll
        for (int i = 0; i < NN; ++i) x[i] += tref;
        // outflow faces: transverse ones to the next lanes, DEP kept here
#pragma unroll
        for (int a = 0; a < D; ++a) {
            const int sg = sx_sg<D, KV>(a);
            if (sg == 0) continue;
            const int out = sg > 0 ? P : 0;
            T o[TN];
#pragma unroll
            for (int tt = 0; tt < TN; ++tt) o[tt] = x[sx_node<D, NP>(a, out, tt)];
            if (a == DEP) {
#pragma unroll
                for (int tt = 0; tt < TN; ++tt) pd[tt] = o[tt];
            } else {
                sx_sts<TN, (CW > 1)>(xslot(par, a == TA0 ? 0 : 1), o);
            }
            if (!S.final_iter && at_outflow(t, a)) {
                T* tr = static_cast<T*>(S.tr_out[a]) + ((long long)t.pop * S.NS[a] + t.s[a]) * S.glines[a]
                    + (long long)sx_face_cell<D>(S, a, t.g) * TN;
                sx_st<TN>(tr, o);
            }
        }
        if (S.final_iter) {
            const int cell = (t.g[2] * S.n[1] + t.g[1]) * S.n[0] + t.g[0];
#pragma unroll
            for (int i = 0; i < NN; ++i) x[i] = fma(T(2), x[i], -u[i]);
            sx_st<NN>(f + (long long)t.pop * S.nodes + (long long)cell * NN, x);
        }
    };

    SxTrack tp, tc;
    tp.q = tc.q = -skew - 1;
    tp.od = tc.od = tp.i = tc.i = tp.pop = tc.pop = 0;
#pragma unroll
    for (int a = 0; a < 3; ++a) tp.s[a] = tc.s[a] = tp.g[a] = tc.g[a] = 0;
    tp.valid = tc.valid = false;
    for (int k = 0; k < PF; ++k) {
        advance(tp);
        fetch(tp, k);
    }
    for (int W = 0; W < total; ++W) {
        // with one wave in flight the prefetch position of the last wave is
        // this wave's: copy it rather than advance a second tracker
        if constexpr (PF == 1) tc = tp;
        advance(tp);
        fetch(tp, (W + PF) % kSxRing);             // wave W + PF
        cp_wait_group<PF>();                        // wave W has landed
        if constexpr (PF != 1) advance(tc);
        compute(W, tc, W % kSxRing);
        __syncthreads();
    }
    cp_wait_group<0>();
}

// One sweep over every population: blockIdx.x / bpv + k0 is the velocity.
// MAXT bounds the block size (the subdomain's columns), which bounds
// registers.
template <int D, int P, typename T, int MAXT>
__global__ void __launch_bounds__(MAXT) sx_wave_kernel(const __grid_constant__ SxWave<D, P, T> A)
{
    extern __shared__ __align__(128) unsigned char smem_raw[];
    T* xs = reinterpret_cast<T*>(smem_raw);
    const int k = A.k0 + (int)blockIdx.x / A.bpv, lb = (int)blockIdx.x % A.bpv;
    T* ring = xs + 4 * SxRing<D, P, T>::TNP * blockDim.x;
    if (k == 0) sx_sweep_velocity<D, P, 0, T>(A, lb, xs, ring);
    else if (k == 1) sx_sweep_velocity<D, P, 1, T>(A, lb, xs, ring);
    else if (k == 2) sx_sweep_velocity<D, P, 2, T>(A, lb, xs, ring);
    else if (D == 3) sx_sweep_velocity<D, P, 3, T>(A, lb, xs, ring);
}

// ---------------------------------------------------------------------------
// brick sweep: 3D, p = 1, FP32
// ---------------------------------------------------------------------------

// With one cell per lane and wave, four fifths of a warp's instructions were
// bookkeeping: positions, inflow selection, boundary lanes' branches (455 warp
// instructions per wave of 84 FMAs, 21 of 32 lanes active).  Here a lane takes a
// brick of 2 x 2 x 2 cells per wave, so that the bookkeeping is shared by
// eight solves, and a warp is a unit of its own: 32 / cols streams of
// problems, cols = (L0 / 2)(L1 / 2) lanes each, the brick columns of a
// subdomain along z.  The schedule is sx_sweep_velocity's on bricks: lane
// (ox, oy) runs ox + oy waves behind, so its upwind neighbours' outflow faces
// of the wave before are the ones it needs, and they come by shuffle; along z
// they are its own.  Nothing is shared between warps: no block barrier.
//   The cells' f^n arrive by cp.async, copied by the whole warp (8 lanes per half
// brick, so that every 32-byte sector is used): once the four cells of a half
// are solved, the next brick's half takes their place while the other half is
// solved, so one brick of shared memory per lane is enough.  The interface
// inflow of boundary lanes comes beside them, and the last iterate's f^{n+1}
// goes back the same way.  The cell solve is the one of sx_sweep_velocity, operation by
// operation: the results are bitwise the same.
//   Measured, D3Q4 128^3 cells, 8^3-cell subdomains: 201 us per launch (one
// velocity, one iterate) before, 146 now, 2.85 -> 2.17 ms per step.  Twelve warps
// fit per SM (137 registers); with two bricks per lane it was eight and 155 us,
// with the registers cut to 128 for sixteen 153 us.  1,550 warp instructions per
// wave, 920 of them the solves, are issued at 45% of the rate.
constexpr int kBrU = 68;              // shared-memory floats per lane: 64 values, an odd number of 16-byte words
constexpr int kBrF = 20;              // floats per interface face: 16 values, likewise

struct BrickShape {
    int bx, by, cols, nst;            // brick columns per axis, lanes per stream, streams per warp
    size_t smem;
};

__host__ __device__ inline BrickShape brick_shape(int L0, int L1)
{
    BrickShape b;
    b.bx = L0 / 2;
    b.by = L1 / 2;
    b.cols = b.bx * b.by;
    b.nst = b.cols > 0 && b.cols <= 32 ? 32 / b.cols : 0;
    b.smem = sizeof(float) * (size_t)(32 * kBrU + (32 + b.nst * (b.bx + b.by)) * kBrF);
    return b;
}

template <int KV>
__device__ __forceinline__ void sx_brick_velocity(const SxWave<3, 1, float>& A, const int lb, float* sm)
{
    constexpr int SG[3] = {sx_sign(3, KV, 0), sx_sign(3, KV, 1), sx_sign(3, KV, 2)};
    constexpr bool R0 = SG[0] > 0 || SG[1] > 0 || SG[2] > 0;
    const SxArgs& S = A.S;
    const BrickShape bs = brick_shape(S.L[0], S.L[1]);
    const int lane = threadIdx.x;
    const int str = lane / bs.cols, col = lane - str * bs.cols;
    const int oy = col / bs.bx, ox = col - oy * bs.bx;
    const bool active = str < bs.nst;
    const int bz = S.L[2] / 2, skew = ox + oy, maxskew = bs.bx + bs.by - 2;
    const int nsub = S.NS[0] * S.NS[1] * S.NS[2], nprob = S.m * nsub;
    const int nstreams = A.bpv * bs.nst, sid = lb * bs.nst + str;
    // problems of this stream; the warp runs as long as its first stream, which has the most
    const int mine = active && sid < nprob ? (nprob - sid + nstreams - 1) / nstreams : 0;
    const int most = lb * bs.nst < nprob ? (nprob - lb * bs.nst + nstreams - 1) / nstreams : 0;
    const int span = mine * bz, total = most > 0 ? most * bz + maxskew : 0;
    float* const f = static_cast<float*>(S.f);
    const int n0 = S.n[0], n01 = S.n[0] * S.n[1];

    float* const zin = sm + 32 * kBrU + lane * kBrF;
    float* const xin = sm + 32 * (kBrU + kBrF) + (str * bs.by + oy) * kBrF;
    float* const yin = sm + 32 * (kBrU + kBrF) + (bs.nst * bs.by + str * bs.bx + ox) * kBrF;

    // this lane's position: its brick's first cell, variable and subdomain
    struct Pos {
        int q, od, i, pop, s[3], g[3];
        bool valid;
    };
    auto advance = [&](Pos& t) {
        ++t.q;
        t.valid = t.q >= 0 && t.q < span;
        if (!t.valid) return;
        if (t.q == 0 || ++t.od == bz) {
            t.od = 0;
            if (t.q != 0) ++t.i;
            const int pid = sid + t.i * nstreams;
            const int v = sx_div(pid, A.div_nsub), s = pid - v * nsub;
            const int s12 = sx_div(s, A.div_ns0), s2 = sx_div(s12, A.div_ns1);
            t.pop = KV * S.m + v;
            t.s[0] = s - s12 * S.NS[0];
            t.s[1] = s12 - s2 * S.NS[1];
            t.s[2] = s2;
            t.g[0] = t.s[0] * S.L[0] + (SG[0] > 0 ? 2 * ox : S.L[0] - 2 - 2 * ox);
            t.g[1] = t.s[1] * S.L[1] + (SG[1] > 0 ? 2 * oy : S.L[1] - 2 - 2 * oy);
        }
        t.g[2] = t.s[2] * S.L[2] + (SG[2] > 0 ? 2 * t.od : S.L[2] - 2 - 2 * t.od);
    };
    auto offset = [&](const Pos& t) {
        return t.valid ? (long long)t.pop * S.nodes + (long long)(t.g[2] * n01 + t.g[1] * n0 + t.g[0]) * 8 : -1LL;
    };
    auto upper = [](long long v) { return (int)(v >> 32); };
    // the warp's half bricks (two cells along z: oriented half h), 8 lanes
    // each: lane c of 8 moves word c & 3 of row c / 4
    const int cq = lane & 7, cword = (cq & 3) * 4, crow = cq >> 2;
    auto each_word = [&](long long off, int h, auto&& go) {
        const int z = SG[2] > 0 ? h : 1 - h, src = cword + crow * n0 * 8 + z * n01 * 8;
#pragma unroll
        for (int r = 0; r < 8; ++r) {
            const int owner = 4 * r + (lane >> 3);
            const int lo = __shfl_sync(0xffffffffu, (int)off, owner), hi = __shfl_sync(0xffffffffu, upper(off), owner);
            const long long o = ((long long)hi << 32) | (unsigned)lo;
            if (o >= 0) go(f + o + src, sm + owner * kBrU + z * 32 + crow * 16 + cword);
        }
    };

    // interface inflow of one axis (2 x 2 cells, 4 values each), oriented order of the transverse cells
    auto inflow = [&](const Pos& t, int a, float* dst) {
        const int sg = SG[a], b1 = a == 0 ? 1 : 0, b2 = a == 2 ? 1 : 2;
#pragma unroll
        for (int c2 = 0; c2 < 2; ++c2)
#pragma unroll
            for (int c1 = 0; c1 < 2; ++c1) {
                const int g1 = t.g[b1] + (SG[b1] > 0 ? c1 : 1 - c1), g2 = t.g[b2] + (SG[b2] > 0 ? c2 : 1 - c2);
                float* const d = dst + (2 * c2 + c1) * 4;
                if (S.from_f) {
                    int g[3];
                    g[b1] = g1;
                    g[b2] = g2;
                    g[a] = t.g[a] + (sg > 0 ? -1 : 2);
                    if (g[a] < 0) g[a] += S.n[a];
                    if (g[a] >= S.n[a]) g[a] -= S.n[a];
                    const float* up = f + (long long)t.pop * S.nodes + (long long)(g[2] * n01 + g[1] * n0 + g[0]) * 8;
#pragma unroll
                    for (int tt = 0; tt < 4; ++tt) cp_small_g2s<4>(d + tt, up + sx_node<3, 2>(a, sg > 0 ? 1 : 0, tt));
                } else {
                    int sup = t.s[a] - sg;
                    if (sup < 0) sup += S.NS[a];
                    if (sup >= S.NS[a]) sup -= S.NS[a];
                    cp16_g2s(d, static_cast<const float*>(S.tr_in[a]) + ((long long)t.pop * S.NS[a] + sup) * S.glines[a] +
                                    (long long)(g2 * S.n[b1] + g1) * 4);
                }
            }
    };
    auto fetch = [&](const Pos& t, int h) {
        each_word(offset(t), h, [](float* g, float* d) { cp16_g2s(d, g); });
        if (h == 0 && t.valid) {
            if (ox == 0) inflow(t, 0, xin);
            if (oy == 0) inflow(t, 1, yin);
            if (t.od == 0) inflow(t, 2, zin);
        }
        cp_commit();
    };
    // outflow faces of a brick on the subdomain's downwind boundary
    auto trace = [&](const Pos& t, int a, const float (&w)[2][2][4]) {
        const int b1 = a == 0 ? 1 : 0, b2 = a == 2 ? 1 : 2;
        float* tr = static_cast<float*>(S.tr_out[a]) + ((long long)t.pop * S.NS[a] + t.s[a]) * S.glines[a];
#pragma unroll
        for (int c2 = 0; c2 < 2; ++c2)
#pragma unroll
            for (int c1 = 0; c1 < 2; ++c1) {
                const int g1 = t.g[b1] + (SG[b1] > 0 ? c1 : 1 - c1), g2 = t.g[b2] + (SG[b2] > 0 ? c2 : 1 - c2);
                sx_st<4>(tr + (long long)(g2 * S.n[b1] + g1) * 4, w[c2][c1]);
            }
    };

    // faces [c2][c1][4], the transverse cells in oriented order: inflow before
    // a cell's solve, its outflow after it
    float fx[2][2][4] = {}, fy[2][2][4] = {}, fz[2][2][4] = {};
    Pos tp, tc;
    tp.q = -skew - 1;
    tp.od = tp.i = tp.pop = 0;
    tp.valid = false;
#pragma unroll
    for (int a = 0; a < 3; ++a) tp.s[a] = tp.g[a] = 0;
    advance(tp);
    fetch(tp, 0);
    fetch(tp, 1);
    for (int W = 0; W < total; ++W) {
        tc = tp;
        advance(tp);
        // transverse inflow: the neighbour's faces of the wave before
#pragma unroll
        for (int c = 0; c < 16; ++c) {
            float* px = &fx[0][0][0] + c;
            float* py = &fy[0][0][0] + c;
            *px = __shfl_up_sync(0xffffffffu, *px, 1);
            *py = __shfl_up_sync(0xffffffffu, *py, bs.bx);
        }
#pragma unroll
        for (int k = 0; k < 2; ++k) {
            cp_wait_group<1>();           // half k has landed; the other half may be in flight
            __syncwarp();
            if (tc.valid) {
                if (k == 0) {
                    auto take = [&](const float* p, float (&w)[2][2][4]) {
#pragma unroll
                        for (int c = 0; c < 4; ++c) sx_lds<4, true>(p + 4 * c, &w[0][0][0] + 4 * c);
                    };
                    if (ox == 0) take(xin, fx);
                    if (oy == 0) take(yin, fy);
                    if (tc.od == 0) take(zin, fz);
                }
#pragma unroll
                for (int j = 0; j < 2; ++j)
#pragma unroll
                    for (int i = 0; i < 2; ++i) {
                        float* const uc = sm + lane * kBrU + (SG[2] > 0 ? k : 1 - k) * 32 +
                                          (SG[1] > 0 ? j : 1 - j) * 16 + (SG[0] > 0 ? i : 1 - i) * 8;
                        float u[8], r[8], x[8];
                        sx_lds<8, true>(uc, u);
                        const float tref = u[0];
                        r[0] = 0.0f;
#pragma unroll
                        for (int n = 1; n < 8; ++n) r[n] = A.wcell[n] * (u[n] - tref);
#pragma unroll
                        for (int a = 0; a < 3; ++a) {
                            const float* tv = a == 0 ? fx[k][j] : (a == 1 ? fy[k][i] : fz[j][i]);
#pragma unroll
                            for (int tt = 0; tt < 4; ++tt) {
                                const int n = sx_node<3, 2>(a, SG[a] > 0 ? 0 : 1, tt);
                                r[n] = fmaf(A.face[KV][a][tt], tv[tt] - tref, r[n]);
                            }
                        }
#pragma unroll
                        for (int n = 0; n < 8; ++n)
                            x[n] = R0 ? A.ainv[KV][n * 8] * r[0] : A.ainv[KV][n * 8 + 1] * r[1];
#pragma unroll
                        for (int c = R0 ? 1 : 2; c < 8; ++c)
#pragma unroll
                            for (int n = 0; n < 8; ++n) x[n] = fmaf(A.ainv[KV][n * 8 + c], r[c], x[n]);
#pragma unroll
                        for (int n = 0; n < 8; ++n) x[n] += tref;
#pragma unroll
                        for (int tt = 0; tt < 4; ++tt) {
                            fx[k][j][tt] = x[sx_node<3, 2>(0, SG[0] > 0 ? 1 : 0, tt)];
                            fy[k][i][tt] = x[sx_node<3, 2>(1, SG[1] > 0 ? 1 : 0, tt)];
                            fz[j][i][tt] = x[sx_node<3, 2>(2, SG[2] > 0 ? 1 : 0, tt)];
                        }
                        if (S.final_iter) {
#pragma unroll
                            for (int n = 0; n < 8; ++n) x[n] = fmaf(2.0f, x[n], -u[n]);
                            sx_sts<8, true>(uc, x);
                        }
                    }
                if (k == 1 && !S.final_iter) {
                    if (ox == bs.bx - 1) trace(tc, 0, fx);
                    if (oy == bs.by - 1) trace(tc, 1, fy);
                    if (tc.od == bz - 1) trace(tc, 2, fz);
                }
            }
            __syncwarp();                 // half k may be refilled; the last iterate's values are in it
            if (S.final_iter) {
                each_word(offset(tc), k, [](float* g, float* d) {
                    *reinterpret_cast<float4*>(g) = *reinterpret_cast<const float4*>(d);
                });
                __syncwarp();
            }
            fetch(tp, k);
        }
    }
    cp_wait_group<0>();
}

// One warp per block: blockIdx.x / bpv + k0 is the velocity.
__global__ void __launch_bounds__(32) sx_brick_kernel(const __grid_constant__ SxWave<3, 1, float> A)
{
    extern __shared__ __align__(128) unsigned char smem_raw[];
    float* sm = reinterpret_cast<float*>(smem_raw);
    const int k = A.k0 + (int)blockIdx.x / A.bpv, lb = (int)blockIdx.x % A.bpv;
    if (k == 0) sx_brick_velocity<0>(A, lb, sm);
    else if (k == 1) sx_brick_velocity<1>(A, lb, sm);
    else if (k == 2) sx_brick_velocity<2>(A, lb, sm);
    else sx_brick_velocity<3>(A, lb, sm);
}

// ---------------------------------------------------------------------------
// split sweep: 2D, FP32
// ---------------------------------------------------------------------------

// A 2D mesh has few problems (768 for 64 subdomains of the vortex), so a sweep
// is as long as its chain: 63 waves of one warp, 1,800 cycles each with the
// whole cell solve in the chain (57 us per iterate at p = 2).  But of
//   f* = t + A^{-1} (W_cell (f^n - t) + sum_a nu_a E_a W_perp (tr_a - t))
// the next cell needs only the outflow nodes, and the f^n part of those is known
// before the sweep starts.  So a step is
//   local   for every cell, t and A^{-1} W_cell (f^n - t) at the outflow nodes
//           (one record Z per population and cell), all cells at once -- only
//           after f was set: otherwise the step before has left them;
//   chain   K sweeps over the records: per cell 2 (p + 1) inflow values, a
//           (2p + 1) x 2(p + 1) matrix and 2p + 1 outflow values (p = 2: 30
//           FMAs instead of 87); the last one leaves the outflow values in Z;
//   finish  for every cell, the full solve with its final inflow, f^{n+1} =
//           2 f* - f^n, the relaxation and the next step's record, all cells
//           at once: f is read and written once.
// Both parts vanish for a constant state, so it is kept exactly, as in the
// one-kernel form.
//   Measured (20 steps with set-up and read-back, before -> now): 256^2 cells,
// p = 2 3.77 -> 2.18 ms; 378^2, 9-cell subdomains, p = 3 15.0 -> 5.6; 320 x 80,
// 40-cell subdomains, p = 3 6.7 -> 2.2; 384^2, 8-cell subdomains, p = 1 5.5 ->
// 2.5; 64^2, p = 1 1.87 -> 1.18.  What bounds it: the waves' latency (63 of them,
// three times a step) and the finish, 40 us cold, by its shared-memory traffic.
template <int P>
struct SxSplit {
    static constexpr int NP = P + 1, NN = NP * NP, TN = NP, NO = 2 * TN - 1, NI = 2 * TN;
    static constexpr int ZS = (NO + 1 + 3) / 4 * 4;      // floats per record: t, outflow nodes
    SxArgs S;
    float *Z, *Znext;                                    // records of this step, and of the next one
    int bpv;
    SxDiv div_nsub, div_ns0, div_n0, div_L0, div_L1;
    float gm[3][NO][NI];                                 // outflow node <- inflow value (axis DEP, then the other)
    float aw[3][NO][NN];                                 // outflow node <- f^n - t
    float ainv[3][NN * NN], wcell[NN], face[3][2][TN];
};

// Axis along which velocity k's chain runs, and the record's slot of each
// outflow node: the nodes of the face along that axis, then the rest of the other
// face (they share a corner).
__host__ __device__ constexpr int sp_dep(int k) { return k == 0 ? 0 : 1; }
__host__ __device__ constexpr int sp_out(int k, int a, int P) { return sx_sign(2, k, a) > 0 ? P : 0; }
template <int P>
__host__ __device__ constexpr int sp_slot(int k, int a, int tt)
{
    const int dep = sp_dep(k), od = sp_out(k, dep, P);
    if (a == dep) return tt;
    return tt == od ? sp_out(k, 1 - dep, P) : P + 1 + (tt < od ? tt : tt - 1);
}
template <int P>
__host__ __device__ constexpr int sp_node(int k, int slot)
{
    constexpr int NP = P + 1;
    const int dep = sp_dep(k), od = sp_out(k, dep, P), ot = sp_out(k, 1 - dep, P);
    if (slot < NP) return sx_node<2, NP>(dep, od, slot);
    const int r = slot - NP, tt = r < od ? r : r + 1;
    return sx_node<2, NP>(1 - dep, ot, tt);
}

template <int P>
__global__ void __launch_bounds__(64 * (P + 1)) sx_local_kernel(const __grid_constant__ SxSplit<P> A)
{
    using SP = SxSplit<P>;
    constexpr int NN = SP::NN, NO = SP::NO, ZS = SP::ZS, NNP = NN | 1, ZP = ZS + 1, NT = 32 * (NO + 1);
    __shared__ float u[32 * NNP], zr[32 * ZP];
    const int s = threadIdx.x >> 5, c = threadIdx.x & 31;          // warp: a slot; lanes: cells
    const long long cells = A.S.nodes / NN;
    const int pop = blockIdx.y, k = pop / A.S.m;
    const float* f = static_cast<const float*>(A.S.f) + (long long)pop * A.S.nodes;
    for (long long c0 = blockIdx.x * 32LL; c0 < cells; c0 += gridDim.x * 32LL) {
        const int nc = (int)(cells - c0 < 32 ? cells - c0 : 32);
        for (int e = threadIdx.x; e < nc * NN; e += NT) u[(e / NN) * NNP + e % NN] = f[c0 * NN + e];
        __syncthreads();
        const float t = u[c * NNP];
        float z = t;
        if (s > 0) {
            z = 0.0f;
#pragma unroll
            for (int j = 1; j < NN; ++j) z = fmaf(A.aw[k][s - 1][j], u[c * NNP + j] - t, z);
        }
        zr[c * ZP + s] = z;
        __syncthreads();
        float* Z = A.Z + ((long long)pop * cells + c0) * ZS;
        for (int e = threadIdx.x; e < nc * ZS; e += NT) Z[e] = zr[(e / ZS) * ZP + e % ZS];
        __syncthreads();
    }
}

// Problems that a block of nt lanes takes side by side on lanes of n0 columns
// each: as many as fit, while their transverse faces (2 Ld TN values each)
// stay within 32 KB.
__host__ __device__ inline int chain_groups(int nt, int n0, int Ld, int TN)
{
    const int fit = nt / n0, room = 4096 / (Ld * TN);
    return fit < 1 ? 1 : (fit <= room ? fit : (room < 1 ? 1 : room));
}

// One velocity's chain: the lanes and the skew of sx_sweep_velocity (D = 2) on
// records, problem after problem.  What a wave needs besides its record is
// moved out of the waves -- a problem's inflow along both axes is loaded before
// its first, its outflow traces are stored after its last -- because in a wave
// it is one lane's work that the whole warp waits for (with it in the waves they
// took 1,000 to 1,400 cycles).
template <int P, int KV>
__device__ __forceinline__ void sx_chain_velocity(const SxSplit<P>& A, const int lb, float* sm)
{
    using SP = SxSplit<P>;
    constexpr int NP = SP::NP, NN = SP::NN, TN = SP::TN, ZS = SP::ZS;
    constexpr int NEP = sx_pad_odd(ZS, 4), TNP = sx_pad_odd(TN, TN == 4 ? 4 : 1);
    constexpr int DEP = sp_dep(KV), TA = 1 - DEP, SGD = sx_sign(2, KV, DEP), SGT = sx_sign(2, KV, TA);
    constexpr bool X0 = SGT != 0;
    constexpr int NO = X0 ? SP::NO : TN, NI = X0 ? SP::NI : TN;
    const SxArgs& S = A.S;
    const int tid = threadIdx.x, nt = blockDim.x;
    const int n0 = S.L[TA], Ld = S.L[DEP];
    const int G = chain_groups(nt, n0, Ld, TN), grp = tid / n0, ln = tid - grp * n0;
    const int lt = SGT < 0 ? n0 - 1 - ln : ln;
    const int skew = X0 ? ln : 0, waves = Ld + (X0 ? n0 - 1 : 0);
    const int nsub = S.NS[0] * S.NS[1], nprob = S.m * nsub;
    const long long cells = S.nodes / NN;
    const float* f = static_cast<const float*>(S.f);
    float* const ring = sm;                                // [2][lane][NEP]
    float* const xs = ring + 2 * nt * NEP;                 // exchange [2][lane][TNP]
    float* const tin = xs + 2 * nt * TNP + grp * (2 * Ld * TN), *const tout = tin + Ld * TN;
    auto sync = [&]() {
        if (nt > 32) __syncthreads();
        else __syncwarp();
    };
    auto xslot = [&](int par) { return xs + (par * nt + tid) * TNP; };

    for (int base = lb * G; base < nprob; base += A.bpv * G) {
        const int pid = base + grp;
        const bool has = grp < G && pid < nprob;
        const int v = sx_div(has ? pid : 0, A.div_nsub), sub = (has ? pid : 0) - v * nsub;
        int s[2];
        s[1] = sx_div(sub, A.div_ns0);
        s[0] = sub - s[1] * S.NS[0];
        const int pop = KV * S.m + v, gt = s[TA] * n0 + lt;
        auto along = [&](int od) { return s[DEP] * Ld + (SGD < 0 ? Ld - 1 - od : od); };
        // value tt of the inflow across axis a's interface at transverse cell gc
        auto inflow = [&](int a, int gc, int tt) {
            const int sg = a == DEP ? SGD : SGT;
            if (S.from_f) {
                // iterate 0 of eq. ibvp: f^n on the outflow face of the upwind cell
                int g = s[a] * S.L[a] + (sg > 0 ? -1 : S.L[a]);
                if (g < 0) g += S.n[a];
                if (g >= S.n[a]) g -= S.n[a];
                const int cell = a == 0 ? gc * S.n[0] + g : g * S.n[0] + gc;
                return f[(long long)pop * S.nodes + (long long)cell * NN + sx_node<2, NP>(a, sg > 0 ? P : 0, tt)];
            }
            int sup = s[a] - sg;
            if (sup < 0) sup += S.NS[a];
            if (sup >= S.NS[a]) sup -= S.NS[a];
            return static_cast<const float*>(S.tr_in[a])[((long long)pop * S.NS[a] + sup) * S.glines[a] +
                                                          (long long)gc * TN + tt];
        };
        float pd[TN];                                      // outflow face along DEP of the wave before
#pragma unroll
        for (int tt = 0; tt < TN; ++tt) pd[tt] = has ? inflow(DEP, gt, tt) : 0.0f;
        if (X0 && has)
            for (int e = ln; e < Ld * TN; e += n0) tin[e] = inflow(TA, along(e / TN), e % TN);
        const int c0 = DEP == 0 ? gt * S.n[0] + along(0) : along(0) * S.n[0] + gt;
        float* const z0 = A.Z + ((long long)pop * cells + c0) * ZS;
        const long long zstep = (long long)SGD * (DEP == 0 ? 1 : S.n[0]) * ZS;
        auto fetch = [&](int W) {
            const int q = W - skew;
            if (has && q >= 0 && q < Ld) {
                float* d = ring + ((W & 1) * nt + tid) * NEP;
                const float* src = z0 + q * zstep;
#pragma unroll
                for (int e = 0; e < ZS; e += 4) cp16_g2s(d + e, src + e);
            }
            cp_commit();
        };
        fetch(0);
        sync();                                            // tin is there for the group's first lane
        for (int W = 0; W < waves; ++W) {
            fetch(W + 1);
            cp_wait_group<1>();
            const int q = W - skew;
            if (has && q >= 0 && q < Ld) {
                float z[ZS], g[NI], o[NO];
                sx_lds<ZS, true>(ring + ((W & 1) * nt + tid) * NEP, z);
#pragma unroll
                for (int tt = 0; tt < TN; ++tt) g[tt] = pd[tt] - z[0];
                if constexpr (X0) {
                    const float* src = ln == 0 ? tin + q * TN : xslot((W & 1) ^ 1) - TNP;
#pragma unroll
                    for (int tt = 0; tt < TN; ++tt) g[TN + tt] = src[tt] - z[0];
                }
                // the differences to t first, t last: summed onto t, every term would
                // round like t itself (64^2 cells, p = 1: 55.9 -> 57.8 us per step)
#pragma unroll
                for (int sl = 0; sl < NO; ++sl) o[sl] = fmaf(A.gm[KV][sl][0], g[0], z[1 + sl]);
#pragma unroll
                for (int j = 1; j < NI; ++j)
#pragma unroll
                    for (int sl = 0; sl < NO; ++sl) o[sl] = fmaf(A.gm[KV][sl][j], g[j], o[sl]);
#pragma unroll
                for (int sl = 0; sl < NO; ++sl) o[sl] += z[0];
#pragma unroll
                for (int tt = 0; tt < TN; ++tt) pd[tt] = o[tt];
                if constexpr (X0) {
                    float* d = ln == n0 - 1 ? tout + q * TN : xslot(W & 1);
#pragma unroll
                    for (int tt = 0; tt < TN; ++tt) d[tt] = o[sp_slot<P>(KV, TA, tt)];
                }
                if (S.final_iter) {
#pragma unroll
                    for (int sl = 0; sl < NO; ++sl) z[1 + sl] = o[sl];
                    sx_st<ZS>(z0 + q * zstep, z);
                }
            }
            sync();
        }
        if (!S.final_iter && has) {
            float* tr = static_cast<float*>(S.tr_out[DEP]) + ((long long)pop * S.NS[DEP] + s[DEP]) * S.glines[DEP] +
                        (long long)gt * TN;
#pragma unroll
            for (int tt = 0; tt < TN; ++tt) tr[tt] = pd[tt];
            if constexpr (X0) {
                float* tx = static_cast<float*>(S.tr_out[TA]) + ((long long)pop * S.NS[TA] + s[TA]) * S.glines[TA];
                for (int e = ln; e < Ld * TN; e += n0) tx[(long long)along(e / TN) * TN + e % TN] = tout[e];
            }
        }
        sync();                                            // tin and tout may be filled again
    }
    cp_wait_group<0>();
}

template <int P, int MAXT>
__global__ void __launch_bounds__(MAXT) sx_chain_kernel(const __grid_constant__ SxSplit<P> A)
{
    extern __shared__ __align__(128) unsigned char smem_raw[];
    float* sm = reinterpret_cast<float*>(smem_raw);
    const int k = (int)blockIdx.x / A.bpv, lb = (int)blockIdx.x % A.bpv;
    if (k == 0) sx_chain_velocity<P, 0>(A, lb, sm);
    else if (k == 1) sx_chain_velocity<P, 1>(A, lb, sm);
    else sx_chain_velocity<P, 2>(A, lb, sm);
}

// (the velocities with a transverse inflow run along y on lanes along x)
template <int P>
static size_t chain_smem(int nt, const int* L)
{
    constexpr int TN = P + 1, NEP = sx_pad_odd(SxSplit<P>::ZS, 4), TNP = sx_pad_odd(TN, TN == 4 ? 4 : 1);
    return sizeof(float) * ((size_t)2 * nt * (NEP + TNP) + (size_t)chain_groups(nt, L[0], L[1], TN) * 2 * L[1] * TN);
}

// Relaxation of one node's populations with the d + 1 velocity equilibria:
// M_{k,v} = sum_j Minv[k][j] rhs_j, rhs = (W_v, Q^1_v, ..., Q^d_v) (eq. maxwell_def).
template <int D, int SYS, typename T>
__device__ __forceinline__ void sx_relax_node(const SxArgs& S, T* fk)
{
    constexpr int M = nvars(D, SYS);
    constexpr int NV = D + 1;
    const RelaxK<T>& RK = relax_k<T>(S.rx);
    auto minv = [&](int i, int j) -> T {
        if constexpr (sizeof(T) == 4) return S.minvf[i * NV + j];
        else return S.minv[i * NV + j];
    };
    T W[M];
#pragma unroll
    for (int v = 0; v < M; ++v) {
        Acc<T> acc;
#pragma unroll
        for (int kk = 0; kk < NV; ++kk) acc.add(fk[kk * M + v]);
        W[v] = acc.s;
    }
    T Q[D][M];
    if (SYS == kAdvection) {
#pragma unroll
        for (int a = 0; a < D; ++a) Q[a][0] = RK.adv[a] * W[0];
    } else {
        const T inv = T(1) / W[0];
        T ke = 0;
#pragma unroll
        for (int b = 0; b < D; ++b) ke = fma(W[1 + b], W[1 + b], ke);
        const T pr = RK.gm1 * (W[1 + D] - T(0.5) * ke * inv);
#pragma unroll
        for (int a = 0; a < D; ++a) {
            const T ua = W[1 + a] * inv;
            Q[a][0] = W[1 + a];
#pragma unroll
            for (int b = 0; b < D; ++b) Q[a][1 + b] = W[1 + b] * ua + (b == a ? pr : T(0));
            Q[a][1 + D] = (W[1 + D] + pr) * ua;
        }
    }
#pragma unroll
    for (int kk = 0; kk < NV; ++kk)
#pragma unroll
        for (int v = 0; v < M; ++v) {
            T mk = minv(kk, 0) * W[v];
#pragma unroll
            for (int a = 0; a < D; ++a) mk = fma(minv(kk, 1 + a), Q[a][v], mk);
            T& fv = fk[kk * M + v];
            fv = S.rx.two ? fma(T(2), mk, -fv) : RK.omega * mk + RK.om1 * fv;
        }
}

// Threads: node-major over 32 cells, so that a warp's node, and with it every
// coefficient, is uniform.
template <int P, int SYS>
__global__ void __launch_bounds__(32 * (P + 1) * (P + 1)) sx_finish_kernel(const __grid_constant__ SxSplit<P> A)
{
    using SP = SxSplit<P>;
    constexpr int NP = SP::NP, NN = SP::NN, TN = SP::TN, ZS = SP::ZS, NNP = NN | 1, NT = 32 * NN;
    constexpr int M = nvars(2, SYS), NPOP = 3 * M;
    extern __shared__ __align__(128) unsigned char smem_raw[];
    float* const u = reinterpret_cast<float*>(smem_raw);         // [pop][cell][NNP]
    float* const r = u + NPOP * 32 * NNP;                         // [pop][node][cell]
    float* const tr = r + NPOP * NN * 32;                         // [pop][axis][face node][cell]
    const SxArgs& S = A.S;
    const int n = threadIdx.x >> 5, c = threadIdx.x & 31;
    const long long cells = S.nodes / NN;
    float* const f = static_cast<float*>(S.f);
    for (long long c0 = blockIdx.x * 32LL; c0 < cells; c0 += gridDim.x * 32LL) {
        const int nc = (int)(cells - c0 < 32 ? cells - c0 : 32);
        // (every load by cp.async: a dozen loops of loads waited for one by one
        // took most of the kernel's time, 44 us for 256^2 cells at p = 2)
        if ((int)threadIdx.x < nc * NN) {
#pragma unroll
            for (int pop = 0; pop < NPOP; ++pop)
                cp_small_g2s<4>(u + (pop * 32 + threadIdx.x / NN) * NNP + threadIdx.x % NN,
                                f + (long long)pop * S.nodes + c0 * NN + threadIdx.x);
        }
        for (int e = threadIdx.x; e < NPOP * 2 * 32; e += NT) {
            const int cc = e & 31, a = (e >> 5) & 1, pop = e >> 6, k = pop / M, sg = sx_sign(2, k, a);
            if (sg == 0 || cc >= nc) continue;
            const int cell = (int)c0 + cc, gy = sx_div(cell, A.div_n0), gx = cell - gy * S.n[0];
            const int ga = a == 0 ? gx : gy, sub = sx_div(ga, a == 0 ? A.div_L0 : A.div_L1), la = ga - sub * S.L[a];
            float* const d = tr + (pop * 2 + a) * TN * 32 + cc;
            if (la == (sg > 0 ? 0 : S.L[a] - 1)) {
                int sup = sub - sg;
                if (sup < 0) sup += S.NS[a];
                if (sup >= S.NS[a]) sup -= S.NS[a];
                const float* p = static_cast<const float*>(S.tr_in[a]) + ((long long)pop * S.NS[a] + sup) * S.glines[a] +
                                 (long long)(a == 0 ? gy : gx) * TN;
#pragma unroll
                for (int tt = 0; tt < TN; ++tt) cp_small_g2s<4>(d + tt * 32, p + tt);
            } else {
                const float* p = A.Z + ((long long)pop * cells + cell - (a == 0 ? sg : sg * S.n[0])) * ZS + 1;
#pragma unroll
                for (int tt = 0; tt < TN; ++tt) cp_small_g2s<4>(d + tt * 32, p + sp_slot<P>(k, a, tt));
            }
        }
        cp_commit();
        cp_wait_all();
        __syncthreads();
        const int jx = n % NP, jy = n / NP;
#pragma unroll
        for (int k = 0; k < 3; ++k)
#pragma unroll
            for (int v = 0; v < M; ++v) {
                const int pop = k * M + v;
                const float t = u[(pop * 32 + c) * NNP];
                float x = n == 0 ? 0.0f : A.wcell[n] * (u[(pop * 32 + c) * NNP + n] - t);
#pragma unroll
                for (int a = 0; a < 2; ++a) {
                    const int sg = sx_sign(2, k, a);
                    if (sg == 0 || (a == 0 ? jx : jy) != (sg > 0 ? 0 : P)) continue;
                    const int tt = a == 0 ? jy : jx;
                    x = fmaf(A.face[k][a][tt], tr[((pop * 2 + a) * TN + tt) * 32 + c] - t, x);
                }
                r[(pop * NN + n) * 32 + c] = x;
            }
        __syncthreads();
        float fk[NPOP];
#pragma unroll
        for (int k = 0; k < 3; ++k)
#pragma unroll
            for (int v = 0; v < M; ++v) {
                const int pop = k * M + v;
                float x = A.ainv[k][n * NN] * r[pop * NN * 32 + c];
#pragma unroll
                for (int j = 1; j < NN; ++j) x = fmaf(A.ainv[k][n * NN + j], r[(pop * NN + j) * 32 + c], x);
                // 2 (t + x) - f^n, without rounding f* = t + x in between
                const float t = u[(pop * 32 + c) * NNP], un = u[(pop * 32 + c) * NNP + n];
                fk[pop] = fmaf(2.0f, x, fmaf(2.0f, t, -un));
            }
        sx_relax_node<2, SYS, float>(S, fk);
        __syncthreads();
#pragma unroll
        for (int pop = 0; pop < NPOP; ++pop) u[(pop * 32 + c) * NNP + n] = fk[pop];
        __syncthreads();
        if ((int)threadIdx.x < nc * NN) {
#pragma unroll
            for (int pop = 0; pop < NPOP; ++pop)
                f[(long long)pop * S.nodes + c0 * NN + threadIdx.x] =
                    u[(pop * 32 + threadIdx.x / NN) * NNP + threadIdx.x % NN];
        }
        // the next step's records while f^{n+1} is here (sx_local_kernel)
        float* const zr = r;                                      // [pop][cell][ZS + 1]
        constexpr int NO = SP::NO, ZP = ZS + 1;
        static_assert(ZP <= NN + 2 * TN, "the records fit where the right-hand sides and faces were");
        if (n <= NO) {
#pragma unroll
            for (int k = 0; k < 3; ++k)
#pragma unroll
                for (int v = 0; v < M; ++v) {
                    const int pop = k * M + v;
                    const float* const uc = u + (pop * 32 + c) * NNP;
                    float acc = 0.0f;
                    if (n > 0)
#pragma unroll
                        for (int j = 1; j < NN; ++j) acc = fmaf(A.aw[k][n - 1][j], uc[j] - uc[0], acc);
                    zr[(pop * 32 + c) * ZP + n] = n > 0 ? acc : uc[0];
                }
        }
        __syncthreads();
        for (int pop = 0; pop < NPOP; ++pop)
            for (int e = threadIdx.x; e < nc * ZS; e += NT)
                A.Znext[((long long)pop * cells + c0) * ZS + e] = zr[(pop * 32 + e / ZS) * ZP + e % ZS];
        __syncthreads();
    }
}

template <int D, int SYS, typename T>
__global__ void sx_relax_kernel(const __grid_constant__ SxArgs S)
{
    constexpr int NPOP = (D + 1) * nvars(D, SYS);
    T* f = static_cast<T*>(S.f);
    for (long long i = blockIdx.x * (long long)blockDim.x + threadIdx.x; i < S.nodes;
         i += (long long)gridDim.x * blockDim.x) {
        T fk[NPOP];
#pragma unroll
        for (int p = 0; p < NPOP; ++p) fk[p] = f[(long long)p * S.nodes + i];
        sx_relax_node<D, SYS>(S, fk);
#pragma unroll
        for (int p = 0; p < NPOP; ++p) f[(long long)p * S.nodes + i] = fk[p];
    }
}

// f = M(W) for the d + 1 sets (initialisation), FP64 in; the arithmetic is
// that of kin_init.cuh.  md / mf: the inverse moment matrix in FP64 / as pairs.
template <int NV>
struct SxInit {
    InitArgs A;
    double md[NV * NV];
    F2 mf[NV * NV];
};

template <int D, int SYS, typename T>
__global__ void __launch_bounds__(256) sx_init_kernel(const __grid_constant__ SxInit<D + 1> S,
                                                      const double* __restrict__ Wd, T* __restrict__ f)
{
    constexpr int M = nvars(D, SYS);
    constexpr int NV = D + 1;
    const long long nodes = S.A.nodes;
    for (long long i = blockIdx.x * (long long)blockDim.x + threadIdx.x; i < nodes;
         i += (long long)gridDim.x * blockDim.x) {
        init_node<D, SYS, T>(Wd, nodes, i, S.A.fast, [&](const auto& W) {
            using V = std::remove_cv_t<std::remove_reference_t<decltype(W[0])>>;
            V Q[D][M];
            float worst = init_flux<D, SYS, V>(init_k<V>(S.A), W, Q);
#pragma unroll
            for (int kk = 0; kk < NV; ++kk)
#pragma unroll
                for (int v = 0; v < M; ++v) {
                    auto mi = [&](int j) {
                        if constexpr (std::is_same<V, double>::value) return S.md[kk * NV + j];
                        else return S.mf[kk * NV + j];
                    };
                    V mk = mi(0) * W[v];
                    float mag = init_mag(mk);
#pragma unroll
                    for (int a = 0; a < D; ++a) {
                        const V q = mi(1 + a) * Q[a][v];
                        mk = mk + q;
                        mag += init_mag(q);
                    }
                    init_put<SYS>(f[(long long)(kk * M + v) * nodes + i], mk, mag, worst);
                }
            return worst >= 0.0f;
        });
    }
}

// ---------------------------------------------------------------------------
// launchers
// ---------------------------------------------------------------------------

cudaError_t sx_launch_setup(const SxSetupArgs& a, cudaStream_t st)
{
    sx_setup_kernel<<<1, 32, 0, st>>>(a);
    return cudaGetLastError();
}

static int sx_grid(long long n)
{
    long long g = (n + 255) / 256;
    if (g > 152 * 8) g = 152 * 8;
    return (int)(g < 1 ? 1 : g);
}

constexpr int kSxNarrow = 256;     // block sizes up to this use the register-rich instance

template <int D, int P, typename T>
static const void* wave_fn(int nt)
{
    return nt <= kSxNarrow ? (const void*)sx_wave_kernel<D, P, T, kSxNarrow> : (const void*)sx_wave_kernel<D, P, T, 1024>;
}

template <typename T>
static const void* wave_pick(int dim, int degree, int nt)
{
    if (dim == 2) {
        if (degree == 1) return wave_fn<2, 1, T>(nt);
        if (degree == 2) return wave_fn<2, 2, T>(nt);
        if (degree == 3) return wave_fn<2, 3, T>(nt);
    } else if (dim == 3) {
        if (degree == 1) return wave_fn<3, 1, T>(nt);
        if (degree == 2) return wave_fn<3, 2, T>(nt);
    }
    return nullptr;
}

static int sx_lanes(const SxArgs& a)
{
    if (a.dim == 2) return a.L[0] > a.L[1] ? a.L[0] : a.L[1];
    return a.L[0] * a.L[1];
}

// boundary lanes per transverse axis, at most (the larger transverse extent
// over the velocities' lane layouts)
static int sx_boundary_lanes(const SxArgs& a)
{
    if (a.dim == 2) return 1;
    return a.L[0] > a.L[1] ? a.L[0] : a.L[1];
}

template <int D, int P, typename T>
static size_t wave_smem_of(int nt, int nbm)
{
    using RG = SxRing<D, P, T>;
    // exchange [2 parities][2 axes][nt][TNP] + ring [kSxRing][nt][NEP]
    // + transverse inflow [kSxRing][2 axes][nbm][TNP]
    return (((size_t)4 * RG::TNP + (size_t)kSxRing * RG::NEP) * nt + (size_t)kSxRing * 2 * nbm * RG::TNP) * sizeof(T);
}

template <typename T>
static size_t wave_smem(int dim, int degree, int nt, int nbm)
{
    if (dim == 2) {
        if (degree == 1) return wave_smem_of<2, 1, T>(nt, nbm);
        if (degree == 2) return wave_smem_of<2, 2, T>(nt, nbm);
        if (degree == 3) return wave_smem_of<2, 3, T>(nt, nbm);
    } else if (dim == 3) {
        if (degree == 1) return wave_smem_of<3, 1, T>(nt, nbm);
        if (degree == 2) return wave_smem_of<3, 2, T>(nt, nbm);
    }
    return 0;
}

int sx_sweep_shape(const SxArgs& a, int prec, SxPlan* plan)
{
    const int nt = (sx_lanes(a) + 31) / 32 * 32;
    const void* fn = prec == 1 ? wave_pick<float>(a.dim, a.degree, nt) : wave_pick<double>(a.dim, a.degree, nt);
    const int nbm = sx_boundary_lanes(a);
    const size_t sm = prec == 1 ? wave_smem<float>(a.dim, a.degree, nt, nbm) : wave_smem<double>(a.dim, a.degree, nt, nbm);
    if (!fn || nt > 1024 || sm > 227 * 1024) return 0;
    plan->threads = nt;
    plan->smem = sm;
    return 1;
}

cudaError_t sx_sweep_plan(const SxArgs& a, int prec, SxPlan* plan)
{
    if (!sx_sweep_shape(a, prec, plan)) return cudaErrorInvalidValue;
    int dev = 0, nsm = 0;
    cudaError_t e = cudaGetDevice(&dev);
    if (e == cudaSuccess) e = cudaDeviceGetAttribute(&nsm, cudaDevAttrMultiProcessorCount, dev);
    if (e != cudaSuccess) return e;
    // Bricks: subdomains of whole 2 x 2 x 2 bricks with at most a warp of brick
    // columns, and enough of them that 16 warps per SM have work -- a brick wave
    // is eight cells long, and with few warps its latency shows (12 steps, one
    // cell against bricks: 22 warps per SM, 48^3 cells in 6^3 subdomains, 5.5 ms
    // against 4.0; 7 per SM, 40 x 40 x 48 cells, 2.8 against 4.1).  True of up to 10
    // columns; with 11 to 16 bricks are faster from about 96 warps per SM on and with 17 to 32
    // from 108 (us per step, one cell against bricks: 8^3 cells, 343 subdomains 302 and 454,
    // 729 707 and 717, 1331 1123 and 945; 12 x 10 x 8 cells, 180 307 and 533, 729 1157 and 1059).
    const bool even = a.dim == 3 && a.degree == 1 && a.L[0] % 2 == 0 && a.L[1] % 2 == 0 && a.L[2] % 2 == 0;
    const BrickShape bs = brick_shape(a.L[0], a.L[1]);
    const long long all = (long long)a.nvel * a.m * a.NS[0] * a.NS[1] * a.NS[2];
    plan->brick = prec == 1 && even && bs.nst > 0 && all >= 16LL * nsm * bs.nst;
    if (plan->brick) {
        plan->threads = 32;
        plan->smem = bs.smem;
    }
    const void* fn = (const void*)sx_brick_kernel;
    if (!plan->brick)
        fn = prec == 1 ? wave_pick<float>(a.dim, a.degree, plan->threads)
                       : wave_pick<double>(a.dim, a.degree, plan->threads);
    // (the brick kernel's shared memory stays below 48 KB)
    e = plan->brick ? cudaFuncSetAttribute(fn, cudaFuncAttributePreferredSharedMemoryCarveout, 100)
                    : allow_dynamic_smem(fn, plan->smem);
    if (e != cudaSuccess) return e;
    int occ = 0;
    e = cudaOccupancyMaxActiveBlocksPerMultiprocessor(&occ, fn, plan->threads, plan->smem);
    if (e != cudaSuccess) return e;
    if (occ < 1) return cudaErrorInvalidConfiguration;
    // one resident wave of blocks, each streaming ceil(problems / blocks)
    // problems.  When one velocity's problems alone fill that wave, the
    // velocities go in separate launches (an SM then runs one velocity's
    // code at a time); otherwise one launch takes them all.
    const int nst = plan->brick ? bs.nst : 1;                  // problem streams per block
    const int nprob = (a.m * a.NS[0] * a.NS[1] * a.NS[2] + nst - 1) / nst;
    const int slots = occ * nsm;
    plan->split = nprob >= slots;
    int b = plan->split ? slots : slots / a.nvel;
    if (b < 1) b = 1;
    if (b > nprob) b = nprob;
    const int per = (nprob + b - 1) / b;
    plan->bpv = (nprob + per - 1) / per;
    plan->occupancy = occ;
    return cudaSuccess;
}

template <int D, int P, typename T>
static cudaError_t wave_launch(const SxArgs& a, const double* hrec, int rstride, const SxPlan& plan,
                               cudaStream_t st)
{
    using WA = SxWave<D, P, T>;
    static_assert(sizeof(WA) <= 32000, "sweep parameters exceed the kernel parameter limit");
    constexpr int NN = WA::NN, TN = WA::TN, NV = WA::NV;
    WA w;
    memset(&w, 0, sizeof w);
    w.S = a;
    w.bpv = plan.bpv;
    w.k0 = 0;
    w.div_nsub = sx_div_make(a.NS[0] * a.NS[1] * a.NS[2]);
    w.div_ns0 = sx_div_make(a.NS[0]);
    w.div_ns1 = sx_div_make(a.NS[1]);
    for (int k = 0; k < NV; ++k) {
        const double* rec = hrec + (size_t)k * rstride;
        for (int e = 0; e < NN * NN; ++e) w.ainv[k][e] = (T)rec[e];
        for (int ax = 0; ax < D; ++ax)
            for (int t = 0; t < TN; ++t) w.face[k][ax][t] = (T)rec[NN * NN + NN + ax * TN + t];
    }
    for (int j = 0; j < NN; ++j) w.wcell[j] = (T)hrec[NN * NN + j];
    const void* fn = wave_fn<D, P, T>(plan.threads);
    if constexpr (D == 3 && P == 1 && sizeof(T) == 4)
        if (plan.brick) fn = (const void*)sx_brick_kernel;
    void* p[] = {&w};
    if (!plan.split)
        return cudaLaunchKernel(fn, dim3(a.nvel * plan.bpv), dim3(plan.threads), p, plan.smem, st);
    for (int k = 0; k < a.nvel; ++k) {
        w.k0 = k;
        const cudaError_t e = cudaLaunchKernel(fn, dim3(plan.bpv), dim3(plan.threads), p, plan.smem, st);
        if (e != cudaSuccess) return e;
    }
    return cudaSuccess;
}

// ---- split sweep (2D, FP32): one step from f^n to f^{n+1} ----
template <int P>
static cudaError_t split_step(SxArgs a, const double* hrec, int rstride, const SxPlan& plan, float* Z, float* Znext,
                              bool ready, int iters, void* const (*tr)[3], cudaStream_t st)
{
    using SP = SxSplit<P>;
    constexpr int NN = SP::NN, TN = SP::TN, NO = SP::NO, NP = SP::NP;
    static_assert(sizeof(SP) <= 32000, "parameters exceed the kernel parameter limit");
    SP w;
    memset(&w, 0, sizeof w);
    w.Z = Z;
    w.Znext = Znext;
    w.bpv = plan.split_bpv;
    w.div_nsub = sx_div_make(a.NS[0] * a.NS[1]);
    w.div_ns0 = sx_div_make(a.NS[0]);
    w.div_n0 = sx_div_make(a.n[0]);
    w.div_L0 = sx_div_make(a.L[0]);
    w.div_L1 = sx_div_make(a.L[1]);
    for (int j = 0; j < NN; ++j) w.wcell[j] = (float)hrec[NN * NN + j];
    for (int k = 0; k < 3; ++k) {
        const double* rec = hrec + (size_t)k * rstride;
        const double* fc = rec + NN * NN + NN;
        for (int e = 0; e < NN * NN; ++e) w.ainv[k][e] = (float)rec[e];
        for (int ax = 0; ax < 2; ++ax)
            for (int t = 0; t < TN; ++t) w.face[k][ax][t] = (float)fc[ax * TN + t];
        const bool both = sx_sign(2, k, 1 - sp_dep(k)) != 0;
        for (int s = 0; s < (both ? NO : TN); ++s) {
            const int n = sp_node<P>(k, s);
            for (int j = 0; j < NN; ++j) w.aw[k][s][j] = (float)(rec[n * NN + j] * rec[NN * NN + j]);
            for (int q = 0; q < (both ? 2 : 1); ++q) {
                const int ax = q == 0 ? sp_dep(k) : 1 - sp_dep(k);
                for (int t = 0; t < TN; ++t)
                    w.gm[k][s][q * TN + t] =
                        (float)(rec[n * NN + sx_node<2, NP>(ax, sx_sign(2, k, ax) > 0 ? 0 : P, t)] * fc[ax * TN + t]);
            }
        }
    }
    w.S = a;
    const long long groups = (a.nodes / NN + 31) / 32;
    const unsigned gx = (unsigned)(groups < 1024 ? groups : 1024);
    cudaError_t e = cudaSuccess;
    if (!ready) {
        sx_local_kernel<P><<<dim3(gx, a.npop), 64 * (P + 1), 0, st>>>(w);
        e = cudaGetLastError();
    }
    const void* chain = plan.threads <= 64 ? (const void*)sx_chain_kernel<P, 64> : (const void*)sx_chain_kernel<P, 1024>;
    void* p[] = {&w};
    for (int it = 1; it <= iters && e == cudaSuccess; ++it) {
        for (int ax = 0; ax < 3; ++ax) {
            w.S.tr_in[ax] = tr[(it - 1) & 1][ax];
            w.S.tr_out[ax] = tr[it & 1][ax];
        }
        w.S.from_f = it == 1 && iters > 1;
        w.S.final_iter = it == iters;
        e = cudaLaunchKernel(chain, dim3(3 * w.bpv), dim3(plan.threads), p, plan.split_smem, st);
    }
    const size_t fsm = sizeof(float) * (size_t)a.npop * 32 * ((NN | 1) + NN + 2 * TN);
    const unsigned fg = (unsigned)(groups < 152 * 16 ? groups : 152 * 16);
    const void* fin = a.system == kEuler ? (const void*)sx_finish_kernel<P, kEuler>
                                         : (const void*)sx_finish_kernel<P, kAdvection>;
    if (e == cudaSuccess) e = cudaLaunchKernel(fin, dim3(fg), dim3(32 * NN), p, fsm, st);
    return e;
}

template <int P>
static cudaError_t split_plan(const SxArgs& a, SxPlan* plan)
{
    constexpr int NN = SxSplit<P>::NN, TN = SxSplit<P>::TN;
    const void* chain = plan->threads <= 64 ? (const void*)sx_chain_kernel<P, 64> : (const void*)sx_chain_kernel<P, 1024>;
    plan->split_smem = chain_smem<P>(plan->threads, a.L);
    // (set once to a constant where the default 48 KB would not do: contexts
    // of different sizes share the functions)
    int occ = 0, dev = 0, nsm = 0;
    cudaError_t e = cudaSuccess;
    if (plan->split_smem > 48 * 1024)
        e = cudaFuncSetAttribute(chain, cudaFuncAttributeMaxDynamicSharedMemorySize, 227 * 1024);
    constexpr size_t most = sizeof(float) * 12 * 32 * ((NN | 1) + NN + 2 * TN);       // Euler's 12 populations
    if (e == cudaSuccess && most > 48 * 1024 && a.system == kEuler)
        e = cudaFuncSetAttribute((const void*)sx_finish_kernel<P, kEuler>, cudaFuncAttributeMaxDynamicSharedMemorySize,
                                 (int)most);
    if (e == cudaSuccess)
        e = cudaOccupancyMaxActiveBlocksPerMultiprocessor(&occ, chain, plan->threads, plan->split_smem);
    if (e == cudaSuccess) e = cudaGetDevice(&dev);
    if (e == cudaSuccess) e = cudaDeviceGetAttribute(&nsm, cudaDevAttrMultiProcessorCount, dev);
    if (e != cudaSuccess) return e;
    const int G = std::min(chain_groups(plan->threads, a.L[0], a.L[1], TN),
                           chain_groups(plan->threads, a.L[1], a.L[0], TN));
    const int nprob = (a.m * a.NS[0] * a.NS[1] + G - 1) / G;
    int b = occ * nsm / 3;
    b = b < 1 ? 1 : (b > nprob ? nprob : b);
    const int per = (nprob + b - 1) / b;
    plan->split_bpv = (nprob + per - 1) / per;
    return cudaSuccess;
}

cudaError_t sx_split_plan(const SxArgs& a, SxPlan* plan)
{
    return a.degree == 1 ? split_plan<1>(a, plan) : (a.degree == 2 ? split_plan<2>(a, plan) : split_plan<3>(a, plan));
}

size_t sx_split_bytes(const SxArgs& a)
{
    const int zs = a.degree == 1 ? SxSplit<1>::ZS : (a.degree == 2 ? SxSplit<2>::ZS : SxSplit<3>::ZS);
    return 2 * sizeof(float) * (size_t)a.npop * (size_t)(a.nodes / a.nn) * zs;
}

cudaError_t sx_split_step(const SxArgs& a, const double* hrec, int rstride, const SxPlan& plan, void* Z, int parity,
                          int ready, int iters, void* const (*tr)[3], cudaStream_t st)
{
    const size_t half = sx_split_bytes(a) / 2 / sizeof(float);
    float* z = static_cast<float*>(Z) + (parity ? half : 0);
    float* zn = static_cast<float*>(Z) + (parity ? 0 : half);
    if (a.degree == 1) return split_step<1>(a, hrec, rstride, plan, z, zn, ready, iters, tr, st);
    if (a.degree == 2) return split_step<2>(a, hrec, rstride, plan, z, zn, ready, iters, tr, st);
    return split_step<3>(a, hrec, rstride, plan, z, zn, ready, iters, tr, st);
}

template <typename T>
static cudaError_t wave_dispatch(const SxArgs& a, const double* hrec, int rstride, const SxPlan& plan,
                                 cudaStream_t st)
{
    if (a.dim == 2) {
        if (a.degree == 1) return wave_launch<2, 1, T>(a, hrec, rstride, plan, st);
        if (a.degree == 2) return wave_launch<2, 2, T>(a, hrec, rstride, plan, st);
        if (a.degree == 3) return wave_launch<2, 3, T>(a, hrec, rstride, plan, st);
    } else if (a.dim == 3) {
        if (a.degree == 1) return wave_launch<3, 1, T>(a, hrec, rstride, plan, st);
        if (a.degree == 2) return wave_launch<3, 2, T>(a, hrec, rstride, plan, st);
    }
    return cudaErrorInvalidValue;
}

cudaError_t sx_launch_sweep(const SxArgs& a, int prec, const double* hrec, int rstride, const SxPlan& plan,
                            cudaStream_t st)
{
    return prec == 1 ? wave_dispatch<float>(a, hrec, rstride, plan, st)
                     : wave_dispatch<double>(a, hrec, rstride, plan, st);
}

cudaError_t sx_launch_trace0(const SxArgs& a, int prec, cudaStream_t st)
{
    const int g = sx_grid(a.trace_total);
    if (prec == 1) sx_trace0_kernel<float><<<g, 256, 0, st>>>(a);
    else sx_trace0_kernel<double><<<g, 256, 0, st>>>(a);
    return cudaGetLastError();
}

template <int D, int SYS, typename T>
static void init_go(const SxArgs& a, const double* W, int g, cudaStream_t st)
{
    SxInit<D + 1> S;
    S.A = init_args(a.nodes, a.dim, a.lambda, a.gamma, a.adv);
    for (int i = 0; i < (D + 1) * (D + 1); ++i) {
        S.md[i] = a.minv[i];
        S.mf[i] = f2_make(a.minv[i]);
    }
    sx_init_kernel<D, SYS, T><<<g, 256, 0, st>>>(S, W, static_cast<T*>(a.f));
}

template <typename T>
static cudaError_t relax_dispatch(const SxArgs& a, cudaStream_t st, bool init, const double* W)
{
    const int g = sx_grid(a.nodes);
#define KIN_SX(DD, SY)                                                                     \
    if (a.dim == DD && a.system == SY) {                                                   \
        if (init) init_go<DD, SY, T>(a, W, g, st);                      \
        else sx_relax_kernel<DD, SY, T><<<g, 256, 0, st>>>(a);                             \
        return cudaGetLastError();                                                         \
    }
    KIN_SX(2, kAdvection)
    KIN_SX(2, kEuler)
    KIN_SX(3, kAdvection)
    KIN_SX(3, kEuler)
#undef KIN_SX
    return cudaErrorInvalidValue;
}

cudaError_t sx_launch_relax(const SxArgs& a, int prec, cudaStream_t st)
{
    return prec == 1 ? relax_dispatch<float>(a, st, false, nullptr) : relax_dispatch<double>(a, st, false, nullptr);
}

cudaError_t sx_launch_init(const SxArgs& a, const double* W, int prec, cudaStream_t st)
{
    return prec == 1 ? relax_dispatch<float>(a, st, true, W) : relax_dispatch<double>(a, st, true, W);
}

}  // namespace kin
