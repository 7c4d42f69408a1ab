// Per-step right-hand side (FIR epilogue) and near-field solve (Eq. MOTInversion).
//
//   rhs_m  = E_{n,m} - P_{n-1,m},
//   P_{n-1,m} = T(1)/eps_m J_{n-1,m} + sum_{l=1}^{L-1} delta_l J_{n-l,m} - chi_m (G * J)_hist,m
// with T(1) = 1/2 (Sec. 2.3 reading) and the FIR taps delta_l of Sec. 6.1.
//
// Z_0^delta = diag(T(0)/eps + delta_0) - diag(chi) G_0 couples each voxel to its 26
// neighbours when c dt = h (Sec. 5.2).  Scaled by diag(1/chi) it is symmetric positive
// definite on the voxels with chi > 0 (D_0 = Z_0 in the PDSA, Eq. Dn): the system is A x = b,
// A = diag((T(0)/eps + delta_0)/chi) - G_0 and b = rhs/chi, solved by iterative refinement with
// Chebyshev iterations in FP32 (k_cg) from a fit of the earlier solutions.  Voxels with eps = 1
// (chi = 0) carry J = rhs / (T(0) + delta_0), which is zero for the zero initial state.  The
// solve is one cooperative kernel: on grids whose tiles all fit the GPU its blocks exchange words
// with their neighbours, on larger ones they meet at grid barriers (bounded waits either way: one
// that runs out ends the kernel with a timeout flag).  It stops at ||b - A x|| <= tol ||b|| or
// after max_iter iterations.
#include "mot_internal.cuh"

#include <type_traits>

#include <algorithm>
#include <cmath>

namespace {

constexpr int NT = 256;
constexpr int MAXTAPS = 64;
constexpr int MAXCHEB = 64;

__constant__ double c_stencil[27 * 6];   // G_0(e) for e in {-1,0,1}^3, order xx yy zz xy xz yz
// FIR taps delta_0 .. delta_{n-1} of a context, passed by value to the kernels that
// read them (several contexts with different taps may be live at once)
struct Taps {
    double d[MAXTAPS];
    int n;
};
inline Taps taps_of(const mot_ctx* c) {
    Taps t;
    for (int l = 0; l < MAXTAPS; ++l) t.d[l] = l < c->n_taps ? c->taps[l] : 0.0;
    t.n = c->n_taps;
    return t;
}

// ring slot of J_{n-l}: (s0 - l) mod jring, s0 = n mod jring, 0 <= l < jring
__device__ __forceinline__ long long jslot(int s0, int l, int jring, long long stride) {
    int sl = s0 - l;
    if (sl < 0) sl += jring;
    return (long long)sl * stride;
}

// ---------------------------------------------------------------- start of the solve
// The solve of step n starts from x0 = sum_{i=1}^{F} c_i x_{n-i}, the coefficients being
// the least-squares fit of the previous right-hand side by the F before it,
//     min || b_{n-1} - sum_i c_i b_{n-1-i} ||,        A x_{n-i} = b_{n-i},
// applied one step later.  The right-hand sides of a band-limited march change
// smoothly, so the fit of one step serves the next (start residual 1.7 times that of the
// fit of b_n itself), and nothing of the fit is on the step's critical path: what forms b_n
// also forms the dot products <b_n, b_{n-i}> while it holds the values, and one block
// of the solve kernel sums them, updates the Gram matrix of the ring and solves the F x F
// system while the others iterate.  F = 6: relative start residual 3e-6 on the eps_r = 12
// sphere in a pulse that rises smoothly from rest, 1e-4 .. 1e-3 within 100 steps of an
// abrupt onset, against 7e-3 .. 3e-2 for the quadratic extrapolation (4 vectors: 30 and 5
// times more, 12: 2 times less).
// The extrapolation remains where there is nothing to fit: fewer than four solved steps
// since the march state was reset, or a fit that leaves more than kFitPoor.
constexpr int kFit = mot::kFitVectors;
constexpr int kSlots = kFit + 1;           // ring of right-hand sides
constexpr int kSums = mot::kFitSums;       // <b,b>, <b,b_{n-i}>
constexpr double kFitPoor = 0.05;          // largest ||b - fit||^2 / ||b||^2 that is used
constexpr double kFitPivot = 1e-13;        // relative pivot below which a vector is dropped

struct FitRecord {
    double c[kFit];
    float cf[kFit];    // rounded to FP32
    int use;           // 0: quadratic extrapolation
    int e;             // 2^e is near 1 / rms(b)
};
struct FitState {      // device, zeroed with the march state
    FitRecord rec[2];                  // step n reads rec[n & 1]; its solve writes the other
    double gram[kSlots * kSlots];      // <b_i, b_j> by ring slot
    // the scale that a solve had to find by FP64 sums (an excitation beyond FP32's range at the
    // scale before it: 1e19 times larger or 1e-23), kWide + e, for the step after it; else 0.  The
    // epilogue's own sums overflowed, so that the record alone would never find it, and every step
    // of such a march would start from the extrapolation and form its sums twice
    int wide[2];
};
constexpr int kWide = 1 << 16;
__device__ __forceinline__ int scale_of(const FitState& f, int step) {
    const int w = f.wide[step & 1];
    return w ? w - kWide : f.rec[step & 1].e;
}
static_assert(sizeof(FitState) <= sizeof(double) * mot::kFitWords, "fit state size");

// 2^e, |e| <= 1000 (double) / 120 (float)
__device__ __forceinline__ double pow2d(int e) { return __hiloint2double((1023 + e) << 20, 0); }
__device__ __forceinline__ float pow2f(int e) { return __int_as_float((127 + e) << 23); }
// (double)v by integer operations: a conversion holds the sub-partition like any FP64 instruction
__device__ __forceinline__ double widen(float v) {
    const unsigned u = __float_as_uint(v), m = u & 0x7fffffffu;
    if (m - 0x00800000u >= 0x7f000000u && m != 0u) return (double)v;    // denormal, Inf, NaN
    const unsigned hi = m ? (m >> 3) + 0x38000000u : 0u;
    return __hiloint2double((int)((u & 0x80000000u) | hi), (int)(m << 29));
}
__device__ __forceinline__ double widen(double v) { return v; }
__device__ __forceinline__ bool is_zero(double v) { return (__double_as_longlong(v) << 1) == 0; }

// b ring slot of step n - i, s0 = n mod kSlots
__device__ __forceinline__ int fslot(int s0, int i) {
    const int sl = s0 - i;
    return sl < 0 ? sl + kSlots : sl;
}

// per-voxel factors precomputed at setup (no FP64 divisions in the step):
//   f[0][m] = T(1)/eps_m = 0.5/eps_m, f[1][m] = 1/chi_m (0 if chi_m = 0),
//   f[2][m] = 1/(T(0)/eps_m + delta_0) (used where chi_m = 0), f[3][m] = chi_m
struct EpiArgs {
    long long M;
    const double* f;
    const double* En;      // AoS excitation (forward; may be null) or dO/dJ (adjoint)
    const void* hist;      // (G * J)_hist, SoA
    double* Jring;
    int s0, jring;
    Taps tp;
    int n, bs, nv;         // step, its ring slot, valid (x, b) pairs before it
    double* b64;           // FP64: right-hand side ring [kSlots][3][M]
    float2* xb;            // FP32-history: (x, b) ring [kSlots][3][M], b its high part
    float* bl;             //   low part of b_n [3][M]
    float4* x0;            //   x0 for the neighbours' reads
    double* rhs;           // adjoint: rhs on vacuum voxels (k_adj_vacuum)
    double* out;           // AoS J_n (vacuum voxels written here, the others by the solve) or null
    const FitState* fit;
    double* part;          // [kSums][blocks] partial sums
    double* nrm;           // [blocks] |x|^2 off the active set
    bool adj;
};

// a thread's sums over its voxels: <b, b>, <b, b_{n-i}> and |x|^2 off the active set
template <typename R> struct EpiSums {
    typedef typename std::conditional<std::is_same<R, float>::value, float, double>::type D;
    D bb = 0, dots[kFit];
    double xin = 0.0;
    __device__ EpiSums() {
#pragma unroll
        for (int i = 0; i < kFit; ++i) dots[i] = 0;
    }
};
// what a step's voxels share: the start's coefficients and the scale of the FP32 sums
template <typename R> struct EpiFit {
    typename EpiSums<R>::D c[kFit];
    bool use;
    float scf;
    __device__ EpiFit(const EpiArgs& a) {
        const FitRecord& rec = a.fit->rec[a.n & 1];
        use = rec.use != 0;
        scf = std::is_same<R, float>::value ? pow2f(scale_of(*a.fit, a.n)) : 1.f;
#pragma unroll
        for (int i = 0; i < kFit; ++i)
            if constexpr (std::is_same<R, float>::value) c[i] = use ? rec.cf[i] : extrapolation(i);
            else c[i] = use ? rec.c[i] : extrapolation(i);
    }
    __device__ static constexpr float extrapolation(int i) {
        return i == 0 ? 3.f : i == 1 ? -3.f : i == 2 ? 1.f : 0.f;
    }
};

// Right-hand side and start of one voxel, its three components: the AoS excitation row and
// the factors are read once and coalesced.  All loads of a voxel come before its stores (the
// new slot Jn lies in the same ring the loads read from).  adj: the adjoint march.
// Returns whether the voxel is active; x0: its start (FP32-history, for the neighbours).
// Bound by FP64 issue: an FP64 instruction holds its sub-partition for 64 cycles, so the
// terms are arranged for few of them (b = ((e - g1 j1) - delta_2 j2 ..) / chi + hist: three
// per component with FIR3), vacuum voxels with nothing but zeros in them take none, there
// is no division (scales are powers of two), and FP32-history forms its dot products in
// FP32: it keeps x and b of earlier steps as floats, which only shape the start and the
// fit; the residual of the start that is stored is formed in float pairs.
template <typename R>
__device__ __forceinline__ bool epi_voxel(const EpiArgs& a, bool adj, const EpiFit<R>& fit,
                                          long long m, EpiSums<R>& sum, float4& x0v) {
    constexpr bool DF = std::is_same<R, float>::value;
    const long long M = a.M, st = 3 * M;
    const R* hist = static_cast<const R*>(a.hist);
    const double* r1 = a.Jring + jslot(a.s0, 1, a.jring, st);
    const double* r2 = a.Jring + jslot(a.s0, 2, a.jring, st);
    double* Jn = a.Jring + jslot(a.s0, 0, a.jring, st);
    const double d1 = a.tp.n > 1 ? a.tp.d[1] : 0.0, d2 = a.tp.n > 2 ? a.tp.d[2] : 0.0;
    const double f0 = a.f[m], ichi = a.f[M + m];
    const bool active = !is_zero(ichi);
    double t[3], j1[3], j2[3] = {0.0, 0.0, 0.0};
    bool zero = true;
#pragma unroll
    for (int k = 0; k < 3; ++k) {
        const long long i = k * M + m;
        t[k] = a.En ? a.En[m * 3 + k] : 0.0;
        j1[k] = r1[i];
        if (a.tp.n > 2) j2[k] = r2[i];
        zero = zero && is_zero(t[k]) && is_zero(j1[k]) && is_zero(j2[k]);
    }
    // the vectors of the earlier steps and the history, requested before the first of them is
    // used (one trip to L2 instead of one per step: 14 -> 5 thousand cycles a voxel)
    R hv[3];
    typename std::conditional<DF, float2, double>::type w[kFit][3];
    if (active || adj) {
#pragma unroll
        for (int k = 0; k < 3; ++k) hv[k] = hist[k * M + m];
    }
    if (active) {
#pragma unroll
        for (int i = 0; i < kFit; ++i)
#pragma unroll
            for (int k = 0; k < 3; ++k) {
                if constexpr (DF) {
                    w[i][k] = make_float2(0.f, 0.f);
                    if (i < a.nv) w[i][k] = a.xb[(long long)fslot(a.bs, i + 1) * st + k * M + m];
                } else {
                    w[i][k] = 0.0;
                    if (i < a.nv) w[i][k] = a.b64[(long long)fslot(a.bs, i + 1) * st + k * M + m];
                }
            }
    }
    if (!active && zero && a.tp.n <= 3) {      // vacuum at rest
#pragma unroll
        for (int k = 0; k < 3; ++k) {
            if (adj) a.rhs[k * M + m] = widen(hv[k]);
            Jn[k * M + m] = 0.0;
            if (!adj && a.out) a.out[m * 3 + k] = 0.0;
        }
        return false;
    }
    const double g1 = f0 + d1;
#pragma unroll
    for (int k = 0; k < 3; ++k) {
        t[k] -= g1 * j1[k];
        t[k] -= d2 * j2[k];
    }
    for (int l = 3; l < a.tp.n; ++l) {
        const double* rl = a.Jring + jslot(a.s0, l, a.jring, st);
#pragma unroll
        for (int k = 0; k < 3; ++k) t[k] -= a.tp.d[l] * rl[k * M + m];
    }
    if (!active) {
        const double f2 = a.f[2 * M + m];
#pragma unroll
        for (int k = 0; k < 3; ++k) {
            if (adj) {
                // the solve's iterate must vanish off the active set; vacuum voxels
                // get their lambda after the solve (k_adj_post), when mu is known
                a.rhs[k * M + m] = t[k] + widen(hv[k]);
                Jn[k * M + m] = 0.0;
            } else {
                const double x = t[k] * f2;     // chi = 0: no field term
                Jn[k * M + m] = x;
                if (a.out) a.out[m * 3 + k] = x;
                sum.xin += x * x;
            }
        }
        return false;
    }
    double b[3];
#pragma unroll
    for (int k = 0; k < 3; ++k) {
        const double h = widen(hv[k]);
        b[k] = adj ? t[k] + h : t[k] * ichi + h;
    }
    if constexpr (DF) {
        float bh[3], xs[3] = {0.f, 0.f, 0.f};
#pragma unroll
        for (int k = 0; k < 3; ++k) {
            bh[k] = (float)b[k];
            a.bl[k * M + m] = (float)(b[k] - widen(bh[k]));
            sum.bb += (bh[k] * fit.scf) * (bh[k] * fit.scf);
        }
#pragma unroll
        for (int i = 0; i < kFit; ++i) {
            if (i >= a.nv) continue;
#pragma unroll
            for (int k = 0; k < 3; ++k) {
                xs[k] += fit.c[i] * w[i][k].x;
                sum.dots[i] += (bh[k] * fit.scf) * (w[i][k].y * fit.scf);
            }
        }
        if (!fit.use) {   // quadratic extrapolation from the FP64 ring
            const double* q2 = a.Jring + jslot(a.s0, 2, a.jring, st);
            const double* q3 = a.Jring + jslot(a.s0, 3, a.jring, st);
#pragma unroll
            for (int k = 0; k < 3; ++k) {
                const double x0 = 3.0 * j1[k] - 3.0 * q2[k * M + m] + q3[k * M + m];
                xs[k] = (float)(adj ? a.f[3 * M + m] * x0 : x0);
            }
        }
        float2* v0 = a.xb + (long long)a.bs * st + m;
#pragma unroll
        for (int k = 0; k < 3; ++k) v0[k * M] = make_float2(xs[k], bh[k]);
        x0v = make_float4(xs[0], xs[1], xs[2], 0.f);
    } else {
        double x0[3] = {0.0, 0.0, 0.0}, wx[kFit][3];
        const int nx = fit.use ? a.nv : 3;
#pragma unroll
        for (int i = 0; i < kFit; ++i)
#pragma unroll
            for (int k = 0; k < 3; ++k) {
                wx[i][k] = j1[k];
                if (i > 0 && i < nx)
                    wx[i][k] = a.Jring[jslot(a.s0, i + 1, a.jring, st) + k * M + m];
            }
#pragma unroll
        for (int i = 0; i < kFit; ++i) {
            if (i >= a.nv) continue;
#pragma unroll
            for (int k = 0; k < 3; ++k) sum.dots[i] += b[k] * w[i][k];
        }
#pragma unroll
        for (int i = 0; i < kFit; ++i) {
            if (i >= nx) continue;
#pragma unroll
            for (int k = 0; k < 3; ++k) x0[k] += fit.c[i] * wx[i][k];
        }
        double* b0 = a.b64 + (long long)a.bs * st;
        const double chi = adj ? a.f[3 * M + m] : 1.0;
#pragma unroll
        for (int k = 0; k < 3; ++k) {
            sum.bb += b[k] * b[k];
            b0[k * M + m] = b[k];
            Jn[k * M + m] = adj ? chi * x0[k] : x0[k];
        }
    }
    return true;
}

// A warp's sums of the kSums values, added up lane against lane with the values dealt out on
// the way: 4 + 2 + 1 + 1 + 1 additions for eight values instead of five each.  Lane 4 q
// returns the sum of value q.
template <typename R>
__device__ __forceinline__ typename EpiSums<R>::D epi_warp_sums(const EpiSums<R>& sum) {
    typedef typename EpiSums<R>::D D;
    static_assert(kSums <= 8, "three exchange steps deal out eight values");
    D v[8];
#pragma unroll
    for (int q = 0; q < 8; ++q) v[q] = q == 0 ? sum.bb : q <= kFit ? sum.dots[q - 1] : (D)0;
    const int lane = threadIdx.x & 31;
#pragma unroll
    for (int o = 16, n = 4; o >= 4; o >>= 1, n >>= 1) {
        const bool up = (lane & o) != 0;
#pragma unroll
        for (int q = 0; q < 4; ++q)
            if (q < n) {
                const D keep = up ? v[q + n] : v[q], send = up ? v[q] : v[q + n];
                v[q] = keep + __shfl_xor_sync(0xffffffffu, send, o);
            }
    }
    D r = v[0];
    r += __shfl_xor_sync(0xffffffffu, r, 2);
    r += __shfl_xor_sync(0xffffffffu, r, 1);
    return r;
}
// A block's sums: the warps' in shared memory (stash), a barrier of the block, then one warp,
// whose lane q < kSums returns the sum of value q.  FP32-history sums stay scaled by 4^e
// (fit_block unscales the totals).
template <typename R, int NTH> using EpiRed = typename EpiSums<R>::D[NTH / 32][8];
template <typename R, int NTH>
__device__ __forceinline__ void epi_stash(EpiRed<R, NTH>& red, const EpiSums<R>& sum) {
    const typename EpiSums<R>::D r = epi_warp_sums<R>(sum);
    if ((threadIdx.x & 3) == 0) red[threadIdx.x >> 5][(threadIdx.x & 31) >> 2] = r;
}
template <typename R, int NTH>
__device__ __forceinline__ double epi_block_sum(const EpiRed<R, NTH>& red) {
    const int q = threadIdx.x & 7;
    typename EpiSums<R>::D v = red[0][q];
#pragma unroll
    for (int w = 1; w < NTH / 32; ++w) v += red[w][q];
    return (double)v;
}
// |x|^2 off the active set, the block's share
__device__ __forceinline__ void epi_vacuum_norm(double xin, double* out) {
    __shared__ double redx[NT / 32];
    if (!__syncthreads_or(!is_zero(xin))) {
        if (threadIdx.x == 0) *out = 0.0;
        return;
    }
    for (int o = 16; o > 0; o >>= 1) xin += __shfl_down_sync(0xffffffffu, xin, o);
    if ((threadIdx.x & 31) == 0) redx[threadIdx.x >> 5] = xin;
    __syncthreads();
    if (threadIdx.x == 0) {
        double v = 0.0;
        for (int w = 0; w < (int)blockDim.x / 32; ++w) v += redx[w];
        *out = v;
    }
}

// The epilogue of grids whose solve keeps its vectors in memory (resident solves form the
// right-hand side of their own tile themselves, see k_cg): one thread per voxel.  104^3
// sphere, solve phase with it: 414 -> 376 us with the loads of a voxel requested together and
// eight instead of eleven FP64 instructions a component.
template <typename R, bool ADJ>
__global__ void __launch_bounds__(NT) k_epilogue(const __grid_constant__ EpiArgs a) {
    pdl_trigger();
    pdl_wait();
    const EpiFit<R> fit(a);
    EpiSums<R> sum;
    for (long long m = (long long)blockIdx.x * blockDim.x + threadIdx.x; m < a.M;
         m += (long long)gridDim.x * blockDim.x) {
        float4 x0;
        const bool active = epi_voxel<R>(a, ADJ, fit, m, sum, x0);
        if (std::is_same<R, float>::value && active) a.x0[m] = x0;
    }
    __shared__ EpiRed<R, NT> red;
    epi_stash<R, NT>(red, sum);
    __syncthreads();
    if (threadIdx.x < kSums)
        a.part[(long long)threadIdx.x * gridDim.x + blockIdx.x] = epi_block_sum<R, NT>(red);
    epi_vacuum_norm(sum.xin, a.nrm + blockIdx.x);
}

struct CGArgs {
    long long M;
    int noff[27];         // neighbour e = (ez+1)*9 + (ey+1)*3 + (ex+1): m offset ex + U ey + U V ez
    const int* act;       // active voxels (chi > 0)
    const int* nmask;     // per active voxel: bit e set if neighbour e (0..26) is in the grid
    long long nact;
    int U, V, W;
    const int* tiles;     // origins (x | y << 10 | z << 20) of the tiles with active voxels
    int ntiles;
    const int* halo;      // resident tiles: halo voxels (k_halo_list)
    int nw;               // worker blocks; block nw sums the dot products and fits
    double* x;            // J_n slot (in/out), SoA [3][M]
    double* out;          // AoS J_n or null
    const double* b;      // FP64: rhs / chi, SoA (this step's ring slot)
    const float* diag32;  // A's diagonal (T(0)/eps + delta_0)/chi, FP32 copy
    const double* diag;
    float4* r;            // FP32 inner vectors, one float4 (x, y, z, 0) per voxel
    float4* p;
    float4* q;
    float4* e;
    // FP32-history: (x, b) of this step, SoA; low parts of b; the low parts of the diagonal
    // (its high parts are diag32); the start for the neighbours' reads, and the low parts of
    // x in later refinements
    float2* xb;
    const float* bl;
    const float* diag_lo;
    float4* xl;
    double* red;          // [2][nw] FP64 partial sums: wide residual sums
    float4* red4;         // [2][nw] exchanged partial sums (values, sequence number)
    float tol;            // outer tolerance, relative to ||b||
    float inv_theta;      // Chebyshev: 1 / theta, theta = (lmin + lmax) / 2
    int n_cheb;           // most Chebyshev iterations per refinement (<= MAXCHEB)
    float inv_log2_rate;  // 1 / log2 of the Chebyshev convergence rate (< 0)
    float c1[MAXCHEB];    // d_{k+1} = c1[k] d_k + c2[k] r_{k+1}
    float c2[MAXCHEB];
    int max_iter;         // cap on total inner iterations
    int max_outer;
    int step;             // time index n (for the status record)
    int* status;          // [0] inner its, [1] flags, [2] first bad step, [3] total its
    unsigned* bar;        // [0], [1] arrivals at the grid barriers of even and odd launches,
                          // [2] abort
    int parity;           // of this launch; its block 0 clears the other's arrival words
    long long bar_budget; // longest wait at one barrier, SM clock cycles
    double* nrm;          // [nred] |x|^2 of every block of this step
    const double* nrm_prev;   // of the step before, added up by the fit block into
    double* norm_prev;        // ||x||^2 of that step (null: none to do)
    int nred, prev_step;
    const int* vac;       // resident: voxels outside every tile, taken by the blocks past nw
    int nvac, nvb;
    FitState* fit;
    const double* part;   // epilogue's partial sums [kSums][nepi]
    float4* part4;        // resident: those of the solve's blocks (value, tag seq) [kSums][nw]
    int nepi;
    int bs, nv;           // ring slot of b_n, valid pairs before it
    unsigned seq;         // first sequence number of this launch's exchanges
};

__constant__ float c_st32[27 * 6];   // FP32 copy of c_stencil
__constant__ float c_stl[27 * 6];    // c_stencil - c_st32 rounded to FP32 (double-float low parts)
// the 13 neighbours e > 13 pair with their mirrors 26 - e; G_0(-e) = G_0(e)

// Neighbour pair EP, 26 - EP of the 27-point stencil (G_0(-e) = G_0(e), so the pair's
// values are summed first).  Off-diagonal component (a, b) is zero unless both offset
// coordinates a and b are nonzero (parity), so face pairs take 3 products, edge pairs
// 5 and corner pairs 9.  FULL: every neighbour in the grid (no mask tests).
template <int EP, bool FULL, typename R, typename V>
__device__ __forceinline__ void stencil_pair(const R* __restrict__ S, V&& load, int mask,
                                             R& o0, R& o1, R& o2) {
    constexpr int EM = 26 - EP;
    constexpr int ex = EP % 3 - 1, ey = (EP / 3) % 3 - 1, ez = EP / 9 - 1;
    R sx = 0, sy = 0, sz = 0;
    if (FULL || (mask & (1 << EP))) load(std::integral_constant<int, EP>(), sx, sy, sz);
    if (FULL || (mask & (1 << EM))) load(std::integral_constant<int, EM>(), sx, sy, sz);
    const R* P = S + EP * 6;
    o0 -= P[0] * sx;
    o1 -= P[1] * sy;
    o2 -= P[2] * sz;
    if constexpr (ex != 0 && ey != 0) { o0 -= P[3] * sy; o1 -= P[3] * sx; }
    if constexpr (ex != 0 && ez != 0) { o0 -= P[4] * sz; o2 -= P[4] * sx; }
    if constexpr (ey != 0 && ez != 0) { o1 -= P[5] * sz; o2 -= P[5] * sy; }
}

template <bool FULL, typename R, typename V>
__device__ __forceinline__ void stencil_pairs(const R* __restrict__ S, V&& load, int mask, R& o0,
                                              R& o1, R& o2) {
    stencil_pair<14, FULL>(S, load, mask, o0, o1, o2);
    stencil_pair<15, FULL>(S, load, mask, o0, o1, o2);
    stencil_pair<16, FULL>(S, load, mask, o0, o1, o2);
    stencil_pair<17, FULL>(S, load, mask, o0, o1, o2);
    stencil_pair<18, FULL>(S, load, mask, o0, o1, o2);
    stencil_pair<19, FULL>(S, load, mask, o0, o1, o2);
    stencil_pair<20, FULL>(S, load, mask, o0, o1, o2);
    stencil_pair<21, FULL>(S, load, mask, o0, o1, o2);
    stencil_pair<22, FULL>(S, load, mask, o0, o1, o2);
    stencil_pair<23, FULL>(S, load, mask, o0, o1, o2);
    stencil_pair<24, FULL>(S, load, mask, o0, o1, o2);
    stencil_pair<25, FULL>(S, load, mask, o0, o1, o2);
    stencil_pair<26, FULL>(S, load, mask, o0, o1, o2);
}

constexpr int kAllNeighbours = (1 << 27) - 1;

// f(std::integral_constant<int, E>) for the 13 pairs E = 14 .. 26
template <int B, int E> struct UnrollPairs {
    template <typename F> __device__ __forceinline__ static void run(F&& f) {
        f(std::integral_constant<int, B>());
        UnrollPairs<B + 1, E>::run(f);
    }
};
template <int E> struct UnrollPairs<E, E> {
    template <typename F> __device__ __forceinline__ static void run(F&&) {}
};
typedef UnrollPairs<14, 27> Unroll13;

// (A x)_m in FP64 for an active voxel: centre + 13 symmetric pairs
__device__ __forceinline__ void applyA64(const CGArgs& a, const double* __restrict__ x, int m,
                                         int mask, double o[3]) {
    const long long M = a.M;
    const double* S0 = c_stencil + 13 * 6;
    const double d = a.diag[m];
    double o0 = (d - S0[0]) * x[m], o1 = (d - S0[1]) * x[M + m], o2 = (d - S0[2]) * x[2 * M + m];
    auto load = [&](auto e, double& sx, double& sy, double& sz) {
        const int m2 = m + a.noff[decltype(e)::value];
        sx += x[m2];
        sy += x[M + m2];
        sz += x[2 * M + m2];
    };
    if (mask == kAllNeighbours) stencil_pairs<true>(c_stencil, load, mask, o0, o1, o2);
    else stencil_pairs<false>(c_stencil, load, mask, o0, o1, o2);
    o[0] = o0; o[1] = o1; o[2] = o2;
}

// ---- double-float residual (FP32-history mode)
// A value is a pair hi + lo of floats (about 48 significant bits).  Error-free
// transformations in FP32 with round-to-nearest intrinsics (never contracted into
// FMAs): Knuth's two-sum gives s + e = a + b exactly, and fma(a, b, -a*b) is the exact
// error of the product a*b.  Products keep the hi*lo cross terms and drop lo*lo; sums
// are accumulated without renormalising the low part.  GB300 issues FP64 at about 1/64
// of the FP32 rate, so a residual in these terms costs far fewer issue slots than in
// FP64, at a relative accuracy (~1e-14) four orders below the FP32-history tolerance.
__device__ __forceinline__ void df_two_sum(float a, float b, float& s, float& e) {
    s = __fadd_rn(a, b);
    const float bb = __fsub_rn(s, a);
    e = __fadd_rn(__fsub_rn(a, __fsub_rn(s, bb)), __fsub_rn(b, bb));
}
// (oh, ol) -= (sh + sl) (xh + xl)
__device__ __forceinline__ void df_msub(float sh, float sl, float xh, float xl, float& oh,
                                        float& ol) {
    const float p = __fmul_rn(sh, xh);
    const float pe = __fadd_rn(__fmaf_rn(sh, xh, -p), __fmaf_rn(sh, xl, __fmul_rn(sl, xh)));
    float s, e;
    df_two_sum(oh, -p, s, e);
    oh = s;
    ol = __fadd_rn(ol, __fsub_rn(e, pe));
}
__device__ __forceinline__ void df_split(double v, float& h, float& l) {
    h = (float)v;
    l = (float)(v - (double)h);
}

// (oh, ol) -= G_0 (x_e + x_-e), the pair of neighbours ah + al and bh + bl; COUPLED: with the
// couplings of the components (exactly zero on the three axis pairs)
template <bool PAIR, bool COUPLED>
__device__ __forceinline__ void stencil_pair_df(int e, const float4& ah, const float4& al,
                                                const float4& bh, const float4& bl, float* oh,
                                                float* ol) {
    float sh[3], sl[3];
    df_two_sum(ah.x, bh.x, sh[0], sl[0]);
    df_two_sum(ah.y, bh.y, sh[1], sl[1]);
    df_two_sum(ah.z, bh.z, sh[2], sl[2]);
    if constexpr (PAIR) {
        sl[0] = __fadd_rn(sl[0], __fadd_rn(al.x, bl.x));
        sl[1] = __fadd_rn(sl[1], __fadd_rn(al.y, bl.y));
        sl[2] = __fadd_rn(sl[2], __fadd_rn(al.z, bl.z));
    }
    const float* H = c_st32 + e * 6;
    const float* L = c_stl + e * 6;
    df_msub(H[0], L[0], sh[0], sl[0], oh[0], ol[0]);
    df_msub(H[1], L[1], sh[1], sl[1], oh[1], ol[1]);
    df_msub(H[2], L[2], sh[2], sl[2], oh[2], ol[2]);
    if constexpr (COUPLED) {      // (an edge pair has one of the three, a corner pair all)
        if (H[3] != 0.f) {
            df_msub(H[3], L[3], sh[1], sl[1], oh[0], ol[0]);
            df_msub(H[3], L[3], sh[0], sl[0], oh[1], ol[1]);
        }
        if (H[4] != 0.f) {
            df_msub(H[4], L[4], sh[2], sl[2], oh[0], ol[0]);
            df_msub(H[4], L[4], sh[0], sl[0], oh[2], ol[2]);
        }
        if (H[5] != 0.f) {
            df_msub(H[5], L[5], sh[2], sl[2], oh[1], ol[1]);
            df_msub(H[5], L[5], sh[1], sl[1], oh[2], ol[2]);
        }
    }
}

// r = b - A x at an active voxel in double-float, rounded to FP32.  dh, dl: its diagonal;
// bh, bl: its b pair; load(o, vh, vl): the voxel at halo offset o, HX and HXY the halo's
// strides.  A loop over the neighbour pairs: the pass runs once or twice a step, and written
// out (1200 instructions a voxel, 19 KB) it waited for its own code.
template <bool PAIR, int HX, int HXY, typename V>
__device__ __forceinline__ float4 residual_df_at(float dh, float dl, const float* bh,
                                                 const float* bl, V&& load) {
    float oh[3] = {0.f, 0.f, 0.f}, ol[3] = {0.f, 0.f, 0.f};   // o = A x
    const float* H0 = c_st32 + 13 * 6;
    const float* L0 = c_stl + 13 * 6;
    // centre block: (d - G_0(0)) x; G_0(0) is diagonal (parity)
    float4 c4, cl4 = make_float4(0.f, 0.f, 0.f, 0.f);
    load(0, c4, cl4);
    const float ch[3] = {c4.x, c4.y, c4.z};
    const float cl[3] = {PAIR ? cl4.x : 0.f, PAIR ? cl4.y : 0.f, PAIR ? cl4.z : 0.f};
#pragma unroll
    for (int k = 0; k < 3; ++k) {
        df_msub(-dh, -dl, ch[k], cl[k], oh[k], ol[k]);
        df_msub(H0[k], L0[k], ch[k], cl[k], oh[k], ol[k]);
    }
    // o = (d - G_0(0)) x - sum_pairs G_0(e) (x_e + x_-e) = A x
    auto pair = [&](int e, int o, auto coupled) {
        float4 ah, al, gh, gl;
        load(o, ah, al);
        load(-o, gh, gl);
        stencil_pair_df<PAIR, decltype(coupled)::value>(e, ah, al, gh, gl, oh, ol);
    };
    pair(14, 1, std::false_type());
    pair(16, HX, std::false_type());
    pair(22, HXY, std::false_type());
#pragma unroll 1
    for (int e = 15; e < 27; ++e) {
        if (e == 16 || e == 22) continue;
        pair(e, (e / 9 - 1) * HXY + ((e / 3) % 3 - 1) * HX + e % 3 - 1, std::true_type());
    }
    float r[3];
#pragma unroll
    for (int k = 0; k < 3; ++k) {
        float s, e;
        df_two_sum(bh[k], -oh[k], s, e);
        r[k] = __fadd_rn(s, __fadd_rn(__fsub_rn(bl[k], ol[k]), e));
    }
    return make_float4(r[0], r[1], r[2], 0.f);
}

// ---------------------------------------------------------------- tiles
// The FP32 passes run on tiles of the grid.  A pass stages the tile of d_k with a
// one-voxel halo (zero outside the grid) in shared memory, then every active voxel updates
//   e += d_k, r -= A d_k, d_{k+1} = c1 d_k + c2 r.
// Inactive voxels (diag = 0) hold zeros in every vector and are skipped.
// A thread takes VPT voxels next to each other along z, so that the planes of the stencil
// that they share are read from shared memory once (apply_column).  Tiles of 8 x 4 x 4,
// 8 x 4 x 8 and 8 x 8 x 8 voxels on 128 threads (VPT = 1, 2, 4): the smallest whose tiles all
// find a block of their own on the GPU, which then keeps e, r, d and the diagonal in
// registers for the whole solve and fetches only the halo in a pass; grids with more tiles
// than that take 8 x 8 x 8 on 256 threads with the vectors in memory (solve_shape).  Solve
// phase with the 8 x 4 x 4 tile resident or in memory only, and now: 133 x 27 x 21 150 ->
// 115 us, 48^3 cube 150 -> 109, 56^3 sphere 172 -> 106, 64^3 cube 280 -> 182; in memory, 88^3
// cube 411 -> 391, sphere 365 -> 321 (three blocks per SM instead of two: 375 and 341).
template <int X, int Y, int Z, int V> struct TileShape {
    static constexpr int TX = X, TY = Y, TZ = Z, VPT = V, NTH = X * Y * Z / V;
    static constexpr int HX = X + 2, HY = Y + 2, HZ = Z + 2, HALO = HX * HY * HZ;
    static_assert(NTH % 32 == 0 && Z % V == 0, "tile shape");
    // position of the thread's first voxel; voxel v of it lies v further along z
    __device__ static void local(int& lx, int& ly, int& lz) {
        lx = threadIdx.x % TX;
        ly = (threadIdx.x / TX) % TY;
        lz = threadIdx.x / (TX * TY) * VPT;
    }
    __device__ static int hidx(int lx, int ly, int lz) { return ((lz + 1) * HY + ly + 1) * HX + lx + 1; }
};
typedef TileShape<8, 4, 4, 1> Tile1;
typedef TileShape<8, 4, 8, 2> Tile2;
typedef TileShape<8, 8, 8, 4> Tile4;
typedef TileShape<8, 8, 8, 2> TileMem;   // vectors in memory

__device__ __forceinline__ unsigned ld_acquire_gpu(const unsigned* p) {
    unsigned v;
    asm volatile("ld.acquire.gpu.global.u32 %0, [%1];\n" : "=r"(v) : "l"(p) : "memory");
    return v;
}

// asynchronous 16-byte global -> shared copy; zero-fills the destination when !valid
__device__ __forceinline__ void cp_async16(void* dst, const void* src, bool valid) {
    const unsigned d = (unsigned)__cvta_generic_to_shared(dst);
    asm volatile("cp.async.cg.shared.global [%0], [%1], 16, %2;\n" ::"r"(d), "l"(src),
                 "r"(valid ? 16 : 0));
}
__device__ __forceinline__ void cp_async_commit() {
    asm volatile("cp.async.commit_group;\n" ::: "memory");
}
__device__ __forceinline__ void cp_async_wait1() {   // all but the newest group landed
    asm volatile("cp.async.wait_group 1;\n" ::: "memory");
}
__device__ __forceinline__ void cp_async_wait0() {   // every group landed
    asm volatile("cp.async.wait_group 0;\n" ::: "memory");
}

// halo (zero outside the grid) of v around the tile with origin `org`
template <class T>
__device__ __forceinline__ void load_halo(const CGArgs& a, const float4* __restrict__ v,
                                          float4* buf, int org) {
    const long long UV = (long long)a.U * a.V;
    const int x0 = org & 1023, y0 = (org >> 10) & 1023, z0 = org >> 20;
    for (int h = threadIdx.x; h < T::HALO; h += T::NTH) {
        const int hx = h % T::HX, hy = (h / T::HX) % T::HY, hz = h / (T::HX * T::HY);
        const int x = x0 + hx - 1, y = y0 + hy - 1, z = z0 + hz - 1;
        const bool in = x >= 0 && x < a.U && y >= 0 && y < a.V && z >= 0 && z < a.W;
        cp_async16(&buf[h], in ? v + ((long long)z * UV + (long long)y * a.U + x) : v, in);
    }
}

// A d at the thread's VPT voxels (one above the other, the first at halo position hc), for
// their diagonals dg; c: d itself.  The 27 points of a voxel are three planes of 3 x 3, and a
// plane's sums serve the voxels below, in and above it.  With the element's parities (even
// in each offset on the diagonal; (a, b) odd in d_a and d_b) a plane contributes
//   U  to the voxel in it, E + O to the one below and E - O to the one above:
// per component the centre, the sums over x+-1, y+-1 and the four corners, the corners'
// alternating sum (xy), and the x- and y-odd differences (xz, yz, in O).  31 additions and
// 36 multiply-adds a plane against 39 and 75 for a voxel on its own, and 9 (VPT + 2) / VPT
// shared loads a voxel instead of 27.
template <class T>
__device__ __forceinline__ void apply_column(const float4* sb, int hc, const float* dg, float4* c,
                                             float (*o)[3]) {
    constexpr int V = T::VPT;
    const float* G = c_st32;
    constexpr int C0 = 13 * 6, X1 = 14 * 6, Y1 = 16 * 6, XY = 17 * 6, Z1 = 22 * 6, XZ = 23 * 6,
                  YZ = 25 * 6, XYZ = 26 * 6;        // (1,0,0), (0,1,0), (1,1,0), (0,0,1), ...
#pragma unroll
    for (int v = 0; v < V; ++v) o[v][0] = o[v][1] = o[v][2] = 0.f;
#pragma unroll
    for (int p = -1; p <= V; ++p) {
        const float4* q = sb + hc + p * (T::HX * T::HY);
        const float4 m0 = q[0], xm = q[-1], xp = q[1], ym = q[-T::HX], yp = q[T::HX];
        const float4 mm = q[-T::HX - 1], pm = q[-T::HX + 1], mp = q[T::HX - 1], pp = q[T::HX + 1];
        // corner sums: all, alternating, x-odd, y-odd (first index x)
        const float ax = pp.x + mp.x, bx = pp.x - mp.x, cx = pm.x + mm.x, dx = pm.x - mm.x;
        const float ay = pp.y + mp.y, by = pp.y - mp.y, cy = pm.y + mm.y, dy = pm.y - mm.y;
        const float az = pp.z + mp.z, bz = pp.z - mp.z, cz = pm.z + mm.z, dz = pm.z - mm.z;
        const float Scx = ax + cx, Ax = bx - dx, Cxx = bx + dx;
        const float Scy = ay + cy, Ay = by - dy, Cyy = ay - cy;
        const float Scz = az + cz, Cxz = bz + dz, Cyz = az - cz;
        const float Sxx = xp.x + xm.x, Syx = yp.x + ym.x, Dxx = xp.x - xm.x;
        const float Sxy = xp.y + xm.y, Syy = yp.y + ym.y, Dyy = yp.y - ym.y;
        const float Sxz = xp.z + xm.z, Syz = yp.z + ym.z, Dxz = xp.z - xm.z, Dyz = yp.z - ym.z;
        const float Ex = G[Z1] * m0.x + G[XZ] * Sxx + G[YZ] * Syx + G[XYZ] * Scx + G[XYZ + 3] * Ay;
        const float Ey = G[Z1 + 1] * m0.y + G[XZ + 1] * Sxy + G[YZ + 1] * Syy + G[XYZ + 1] * Scy +
                         G[XYZ + 3] * Ax;
        const float Ez = G[Z1 + 2] * m0.z + G[XZ + 2] * Sxz + G[YZ + 2] * Syz + G[XYZ + 2] * Scz;
        const float Ox = G[XZ + 4] * Dxz + G[XYZ + 4] * Cxz;
        const float Oy = G[YZ + 5] * Dyz + G[XYZ + 5] * Cyz;
        const float Oz = G[XZ + 4] * Dxx + G[XYZ + 4] * Cxx + G[YZ + 5] * Dyy + G[XYZ + 5] * Cyy;
        if (p >= 0 && p < V) {
            c[p] = m0;
            o[p][0] += (dg[p] - G[C0]) * m0.x;
            o[p][1] += (dg[p] - G[C0 + 1]) * m0.y;
            o[p][2] += (dg[p] - G[C0 + 2]) * m0.z;
            o[p][0] -= G[X1] * Sxx + G[Y1] * Syx + G[XY] * Scx + G[XY + 3] * Ay;
            o[p][1] -= G[X1 + 1] * Sxy + G[Y1 + 1] * Syy + G[XY + 1] * Scy + G[XY + 3] * Ax;
            o[p][2] -= G[X1 + 2] * Sxz + G[Y1 + 2] * Syz + G[XY + 2] * Scz;
        }
        if (p >= 1) {                 // the voxel below: this plane is at +z of it
            o[p - 1][0] -= Ex + Ox;
            o[p - 1][1] -= Ey + Oy;
            o[p - 1][2] -= Ez + Oz;
        }
        if (p + 1 < V) {              // the voxel above
            o[p + 1][0] -= Ex - Ox;
            o[p + 1][1] -= Ey - Oy;
            o[p + 1][2] -= Ez - Oz;
        }
    }
}

// voxel index of the thread's voxel v in the tile at org, -1 if outside the grid
template <class T>
__device__ __forceinline__ long long tile_voxel(const CGArgs& a, int org, int v) {
    int lx, ly, lz;
    T::local(lx, ly, lz);
    const int x = (org & 1023) + lx, y = ((org >> 10) & 1023) + ly, z = (org >> 20) + lz + v;
    if (x >= a.U || y >= a.V || z >= a.W) return -1;
    return ((long long)z * a.V + y) * a.U + x;
}

// One Chebyshev iteration over the tiles of this block with all vectors in memory (e = d_0
// on the first iteration, so e needs no clearing).  The halo of the next tile is copied
// into the other shared buffer while the current one is computed, and each thread loads
// its voxels' own e, r and diagonal before waiting for the halo.  LAST: adds |r|^2.
template <class T>
__device__ __forceinline__ void cheb_pass_tiled(const CGArgs& a, const float4* __restrict__ dk,
                                                float4* __restrict__ dn, float c1, float c2,
                                                bool first, bool last, float4 (*sd)[T::HALO],
                                                float& rr_p) {
    int tile = blockIdx.x;
    if (tile < a.ntiles) load_halo<T>(a, dk, sd[0], a.tiles[tile]);
    cp_async_commit();
    for (int it = 0; tile < a.ntiles; ++it, tile += a.nw) {
        const int next = tile + a.nw;
        if (next < a.ntiles) load_halo<T>(a, dk, sd[(it + 1) & 1], a.tiles[next]);
        cp_async_commit();
        const int org = a.tiles[tile];
        long long mv[T::VPT];
        float dgv[T::VPT];
        float4 ev[T::VPT], rv[T::VPT];
#pragma unroll
        for (int v = 0; v < T::VPT; ++v) {
            const long long m = tile_voxel<T>(a, org, v);
            mv[v] = -1;
            dgv[v] = m >= 0 ? a.diag32[m] : 0.f;
            if (dgv[v] != 0.f) {
                mv[v] = m;
                ev[v] = first ? make_float4(0.f, 0.f, 0.f, 0.f) : a.e[m];
                rv[v] = a.r[m];
            }
        }
        cp_async_wait1();
        __syncthreads();
        const float4* sb = sd[it & 1];
        int lx, ly, lz;
        T::local(lx, ly, lz);
        float4 cv[T::VPT];
        float o[T::VPT][3];
        apply_column<T>(sb, T::hidx(lx, ly, lz), dgv, cv, o);
#pragma unroll
        for (int v = 0; v < T::VPT; ++v) {
            if (mv[v] < 0) continue;
            const float4 c = cv[v];
            float4 e = ev[v], r = rv[v];
            e.x += c.x; e.y += c.y; e.z += c.z;
            r.x -= o[v][0]; r.y -= o[v][1]; r.z -= o[v][2];
            const long long m = mv[v];
            a.e[m] = e;
            a.r[m] = r;
            if (last) rr_p += r.x * r.x + r.y * r.y + r.z * r.z;
            dn[m] = make_float4(c1 * c.x + c2 * r.x, c1 * c.y + c2 * r.y, c1 * c.z + c2 * r.z, 0.f);
        }
        __syncthreads();
    }
}

// A block's one tile, resident for the whole solve: each thread's e, r, d and diagonal in
// registers, the tile of d_k in shared memory.  Neighbouring blocks exchange d through
// global memory without a grid barrier: a voxel's d is one 16-byte word whose fourth lane
// is the sequence number of its iteration, stored and loaded as a unit, and a block waits
// for exactly the words of its halo (bounded, like the grid barrier).  An iteration then
// costs one store-to-load trip through L2 instead of fence, counter, poll and halo load.
// d_k lives in p for even and q for odd k; a block overwrites d_k with d_{k+2} only after
// it has seen d_{k+1} of its neighbours, which they store after reading d_k.
template <class T> struct Resident {
    static constexpr int SHELL = T::HALO - T::TX * T::TY * T::TZ;
    static constexpr int HPT = (SHELL + T::NTH - 1) / T::NTH;   // halo voxels per thread
    int m[T::VPT];           // voxel index, -1: none or inactive
    float dg[T::VPT];
    float4 e[T::VPT], r[T::VPT], d[T::VPT];
    int hm[HPT], hs[HPT];    // halo voxels: index (-1: none, stays zero) and shared position
    // position h of the shell of the HX x HY x HZ box: two z faces, then the rings between
    __device__ static void shell(int h, int& hx, int& hy, int& hz) {
        constexpr int FACE = T::HX * T::HY, RING = FACE - T::TX * T::TY;
        if (h < 2 * FACE) {
            hz = h < FACE ? 0 : T::HZ - 1;
            hx = (h % FACE) % T::HX;
            hy = (h % FACE) / T::HX;
        } else {
            const int k = h - 2 * FACE, q = k % RING;
            hz = 1 + k / RING;
            if (q < 2 * T::HX) { hy = q < T::HX ? 0 : T::HY - 1; hx = q % T::HX; }
            else { hy = 1 + (q - 2 * T::HX) / 2; hx = ((q - 2 * T::HX) & 1) ? T::HX - 1 : 0; }
        }
    }
};

template <class T>
__device__ __forceinline__ void resident_init(const CGArgs& a, Resident<T>& t, float4 (*sd)[T::HALO]) {
    typedef Resident<T> RT;
#pragma unroll
    for (int v = 0; v < T::VPT; ++v) {
        t.m[v] = -1;
        t.dg[v] = 0.f;
    }
#pragma unroll
    for (int i = 0; i < RT::HPT; ++i) t.hm[i] = t.hs[i] = -1;
    if ((int)blockIdx.x >= a.ntiles) return;
    const int org = a.tiles[blockIdx.x];
#pragma unroll
    for (int v = 0; v < T::VPT; ++v) {
        const long long m = tile_voxel<T>(a, org, v);
        t.dg[v] = m >= 0 ? a.diag32[m] : 0.f;
        if (t.dg[v] != 0.f) t.m[v] = (int)m;
    }
#pragma unroll
    for (int i = 0; i < RT::HPT; ++i) {
        const int h = threadIdx.x + i * T::NTH;
        if (h >= RT::SHELL) continue;
        int hx, hy, hz;
        RT::shell(h, hx, hy, hz);
        t.hs[i] = (hz * T::HY + hy) * T::HX + hx;
        t.hm[i] = a.halo[(long long)blockIdx.x * (RT::HPT * T::NTH) + h];
        sd[0][t.hs[i]] = sd[1][t.hs[i]] = make_float4(0.f, 0.f, 0.f, 0.f);
    }
}

// halo list of every tile (setup): the voxel of each shell position, -1 where the tile does
// not need it: outside the grid, inactive, or with no active voxel of the tile next to it.
// The last condition makes the waits mutual (a block waits only for words of blocks that
// wait for its own), which is what keeps a word from being overwritten while it is awaited.
template <class T>
__global__ void k_halo_list(const int* __restrict__ tiles, const float* __restrict__ diag32, int U,
                            int V, int W, int* __restrict__ halo) {
    typedef Resident<T> RT;
    const int org = tiles[blockIdx.x];
    const int x0 = org & 1023, y0 = (org >> 10) & 1023, z0 = org >> 20;
    for (int h = threadIdx.x; h < RT::HPT * T::NTH; h += blockDim.x) {
        int found = -1;
        if (h < RT::SHELL) {
            int hx, hy, hz;
            RT::shell(h, hx, hy, hz);
            const int x = x0 + hx - 1, y = y0 + hy - 1, z = z0 + hz - 1;
            const long long m = ((long long)z * V + y) * U + x;
            if (x >= 0 && x < U && y >= 0 && y < V && z >= 0 && z < W && diag32[m] != 0.f)
                for (int e = 0; e < 27; ++e) {
                    const int nx = x + e % 3 - 1, ny = y + (e / 3) % 3 - 1, nz = z + e / 9 - 1;
                    if (nx < x0 || nx >= min(x0 + T::TX, U) || ny < y0 || ny >= min(y0 + T::TY, V) ||
                        nz < z0 || nz >= min(z0 + T::TZ, W))
                        continue;
                    if (diag32[((long long)nz * V + ny) * U + nx] != 0.f) found = (int)m;
                }
        }
        halo[(long long)blockIdx.x * (RT::HPT * T::NTH) + h] = found;
    }
}

// 16-byte loads and stores that are single-copy atomic (data and sequence number together)
__device__ __forceinline__ float4 ld_word(const float4* p) {
    unsigned long long lo, hi;
    asm volatile("{\n.reg .b128 t;\nld.relaxed.gpu.global.b128 t, [%2];\nmov.b128 {%0, %1}, t;\n}"
                 : "=l"(lo), "=l"(hi) : "l"(p) : "memory");
    return make_float4(__uint_as_float((unsigned)lo), __uint_as_float((unsigned)(lo >> 32)),
                       __uint_as_float((unsigned)hi), __uint_as_float((unsigned)(hi >> 32)));
}
__device__ __forceinline__ void st_word(float4* p, float4 v) {
    const unsigned long long lo = (unsigned long long)__float_as_uint(v.x) |
                                  ((unsigned long long)__float_as_uint(v.y) << 32);
    const unsigned long long hi = (unsigned long long)__float_as_uint(v.z) |
                                  ((unsigned long long)__float_as_uint(v.w) << 32);
    asm volatile("{\n.reg .b128 t;\nmov.b128 t, {%1, %2};\nst.relaxed.gpu.global.b128 [%0], t;\n}"
                 ::"l"(p), "l"(lo), "l"(hi) : "memory");
}

// a wait that ran out of its budget: abort word and timeout flag, as grid_barrier
__device__ __forceinline__ void wait_failed(const CGArgs& a) {
    atomicExch(a.bar + 2, 1u);
    atomicOr(a.status + 1, 4);
    atomicCAS(a.status + 2, 0, a.step);
}

// Puts the tile's halo words of `src` tagged `tag` into sb; false on a timed-out wait
template <class T>
__device__ __forceinline__ int halo_words(const CGArgs& a, const float4* src, unsigned tag,
                                          const Resident<T>& t, float4* sb) {
    typedef Resident<T> RT;
    int ok = 1;
    float4 h[RT::HPT];
#pragma unroll
    for (int i = 0; i < RT::HPT; ++i)
        if (t.hm[i] >= 0) h[i] = ld_word(src + t.hm[i]);
#pragma unroll
    for (int i = 0; i < RT::HPT; ++i) {
        if (t.hm[i] < 0 || __float_as_uint(h[i].w) == tag) continue;
        const long long t0 = clock64();
        for (int spin = 1;; ++spin) {
            h[i] = ld_word(src + t.hm[i]);
            if (__float_as_uint(h[i].w) == tag) break;
            if ((spin & 255) != 0) continue;
            if (ld_acquire_gpu(a.bar + 2) != 0u) { ok = 0; break; }
            if (clock64() - t0 > a.bar_budget) { wait_failed(a); ok = 0; break; }
        }
    }
#pragma unroll
    for (int i = 0; i < RT::HPT; ++i)
        if (t.hm[i] >= 0) sb[t.hs[i]] = h[i];
    return ok;
}

// One iteration on the resident tile: waits for the halo words tagged seq + k (with RFIRST
// the first iteration starts from r instead, complete in memory: d_0 = r / theta).  Returns
// false on a timed-out wait.
template <class T, bool RFIRST>
__device__ __forceinline__ bool cheb_pass_resident(const CGArgs& a, int k, unsigned seq, bool last,
                                                   float4 (*sd)[T::HALO], Resident<T>& t,
                                                   float& rr_p) {
    typedef Resident<T> RT;
    if ((int)blockIdx.x >= a.ntiles) return true;
    const float4* dk = (k & 1) ? a.q : a.p;
    float4* dn = (k & 1) ? a.p : a.q;
    float4* sb = sd[k & 1];
    int ok = 1;
    int lx, ly, lz;
    T::local(lx, ly, lz);
#pragma unroll
    for (int v = 0; v < T::VPT; ++v)
        sb[T::hidx(lx, ly, lz + v)] = t.m[v] >= 0 ? t.d[v] : make_float4(0.f, 0.f, 0.f, 0.f);
    if (RFIRST && k == 0) {
        float4 h[RT::HPT];
#pragma unroll
        for (int i = 0; i < RT::HPT; ++i)
            if (t.hm[i] >= 0) {
                h[i] = __ldcg(a.r + t.hm[i]);
                h[i].x *= a.inv_theta; h[i].y *= a.inv_theta; h[i].z *= a.inv_theta;
            }
#pragma unroll
        for (int i = 0; i < RT::HPT; ++i)
            if (t.hm[i] >= 0) sb[t.hs[i]] = h[i];
    } else {
        ok = halo_words<T>(a, dk, seq, t, sb);
    }
    if (!__syncthreads_and(ok)) return false;
    float4 cv[T::VPT];
    float o[T::VPT][3];
    apply_column<T>(sb, T::hidx(lx, ly, lz), t.dg, cv, o);
#pragma unroll
    for (int v = 0; v < T::VPT; ++v) {
        if (t.m[v] < 0) continue;
        const float4 c = cv[v];
        float4 &e = t.e[v], &r = t.r[v];
        e.x += c.x; e.y += c.y; e.z += c.z;
        r.x -= o[v][0]; r.y -= o[v][1]; r.z -= o[v][2];
        if (last) {
            rr_p += r.x * r.x + r.y * r.y + r.z * r.z;
        } else {
            const float c1 = a.c1[k], c2 = a.c2[k];
            t.d[v] = make_float4(c1 * c.x + c2 * r.x, c1 * c.y + c2 * r.y, c1 * c.z + c2 * r.z,
                                 __uint_as_float(seq + 1u));
            st_word(dn + t.m[v], t.d[v]);
        }
    }
    return true;
}

// Partial sums of a thread: |r|^2 and |b|^2 scaled by 4^e in FP32, or (wide) unscaled in FP64.
// They only steer the iteration; in FP32 they are at most 40 roundings, 1.2e-6 of a norm, off
// (thread, warp, block and grid sums in turn), less than the allowance kDrift and kNear make.
struct Sums {
    float rr, bb;
    double rrw, bbw;
    __device__ void add_r(const float* r, bool wide, float sc) {
        if (wide) rrw += (double)r[0] * r[0] + (double)r[1] * r[1] + (double)r[2] * r[2];
        rr += (r[0] * sc) * (r[0] * sc) + (r[1] * sc) * (r[1] * sc) + (r[2] * sc) * (r[2] * sc);
    }
};

// Double-float residual pass on the tiles (FP32-history): the start is in xl; later (PAIR) x
// is in q (high) and xl (low); zero on inactive voxels.  Leaves r scaled by sc = 2^e and the
// first Chebyshev direction d_0 = r / theta of the active voxels: resident tiles keep them
// and send d_0 out as the words of iteration 0, the others store both.
template <class T, bool PAIR, bool RES>
__device__ __forceinline__ bool residual_df_tiled(const CGArgs& a, float4 (*sd)[T::HALO], float sc,
                                                  bool wide, Sums& sum, Resident<T>& res,
                                                  unsigned seq, unsigned xtag, bool own) {
    const long long M = a.M;
    for (int tile = blockIdx.x; tile < a.ntiles; tile += a.nw) {
        const int org = a.tiles[tile];
        constexpr bool words = RES && !PAIR;
        int ok = 1;
        if constexpr (!words) {
            load_halo<T>(a, PAIR ? a.q : a.xl, sd[0], org);
            if (PAIR) load_halo<T>(a, a.xl, sd[1], org);
            cp_async_commit();
        }
        long long mv[T::VPT];
        float dhv[T::VPT], dlv[T::VPT], bh[T::VPT][3], bl[T::VPT][3];
#pragma unroll
        for (int v = 0; v < T::VPT; ++v) {
            const long long m = tile_voxel<T>(a, org, v);
            mv[v] = -1;
            dhv[v] = m >= 0 ? a.diag32[m] : 0.f;
            if (dhv[v] != 0.f) {
                mv[v] = m;
                dlv[v] = a.diag_lo[m];
#pragma unroll
                for (int k = 0; k < 3; ++k) {
                    bh[v][k] = a.xb[k * M + m].y;
                    bl[v][k] = a.bl[k * M + m];
                }
            }
        }
        if constexpr (words) {
            if (!own) {
                int lx, ly, lz;
                T::local(lx, ly, lz);
#pragma unroll
                for (int v = 0; v < T::VPT; ++v)
                    sd[0][T::hidx(lx, ly, lz + v)] =
                        mv[v] >= 0 ? __ldcg(a.xl + mv[v]) : make_float4(0.f, 0.f, 0.f, 0.f);
            }
            ok = halo_words<T>(a, a.xl, xtag, res, sd[0]);
        } else {
            cp_async_wait0();
        }
        if (!__syncthreads_and(ok)) return false;
#pragma unroll
        for (int v = 0; v < T::VPT; ++v) {
            if (mv[v] < 0) continue;
            int lx, ly, lz;
            T::local(lx, ly, lz);
            const int hc = T::hidx(lx, ly, lz + v);
            auto load = [&](int o, float4& vh, float4& vl) {
                vh = sd[0][hc + o];
                if constexpr (PAIR) vl = sd[1][hc + o];
            };
            const float4 r4 = residual_df_at<PAIR, T::HX, T::HX * T::HY>(dhv[v], dlv[v], bh[v], bl[v], load);
            const float rv[3] = {r4.x, r4.y, r4.z};
            sum.add_r(rv, wide, sc);
            const float* h = bh[v];
            if (wide) sum.bbw += (double)h[0] * h[0] + (double)h[1] * h[1] + (double)h[2] * h[2];
            sum.bb += (h[0] * sc) * (h[0] * sc) + (h[1] * sc) * (h[1] * sc) + (h[2] * sc) * (h[2] * sc);
            const float4 r = make_float4(r4.x * sc, r4.y * sc, r4.z * sc, 0.f);
            const float4 d = make_float4(r.x * a.inv_theta, r.y * a.inv_theta, r.z * a.inv_theta,
                                         __uint_as_float(seq));
            if constexpr (RES) {
                res.r[v] = r;
                res.d[v] = d;
                st_word(a.p + mv[v], d);
            } else {
                a.r[mv[v]] = r;
                a.p[mv[v]] = d;
            }
        }
        __syncthreads();
    }
    return true;
}

// block-wide sum of two values; result valid in every thread
template <int NTH>
__device__ __forceinline__ void block_sum2(double& a, double& b) {
    __shared__ double sh[2][NTH / 32];
    for (int o = 16; o > 0; o >>= 1) {
        a += __shfl_down_sync(0xffffffffu, a, o);
        b += __shfl_down_sync(0xffffffffu, b, o);
    }
    const int lane = threadIdx.x & 31, wid = threadIdx.x >> 5;
    __syncthreads();
    if (lane == 0) { sh[0][wid] = a; sh[1][wid] = b; }
    __syncthreads();
    double s0 = 0.0, s1 = 0.0;
#pragma unroll
    for (int k = 0; k < NTH / 32; ++k) { s0 += sh[0][k]; s1 += sh[1][k]; }
    a = s0;
    b = s1;
}

// sum of nb per-block partials, computed by warp 0 (fixed order: identical in every
// block) and broadcast through shared memory
__device__ __forceinline__ double grid_total(const double* red, int nb) {
    __shared__ double s_tot;
    if (threadIdx.x < 32) {
        double v0 = 0.0, v1 = 0.0, v2 = 0.0, v3 = 0.0;   // four independent loads in flight
        int k = threadIdx.x;
        for (; k + 96 < nb; k += 128) {
            v0 += __ldcg(red + k);
            v1 += __ldcg(red + k + 32);
            v2 += __ldcg(red + k + 64);
            v3 += __ldcg(red + k + 96);
        }
        for (; k < nb; k += 32) v0 += __ldcg(red + k);
        double v = (v0 + v1) + (v2 + v3);
        for (int o = 16; o > 0; o >>= 1) v += __shfl_down_sync(0xffffffffu, v, o);
        if (threadIdx.x == 0) s_tot = v;
    }
    __syncthreads();
    const double r = s_tot;
    __syncthreads();
    return r;
}

// Sums over the worker blocks without a grid barrier: a block publishes its two partial
// sums and a sequence number as one 16-byte word, and every block adds all words in the
// same order once they carry that number (bounded waits).  Two sets of words alternate: a
// block publishes to a set again only after it has collected the other, which every block
// publishes after it has read the first.
template <int NTH>
__device__ __forceinline__ void publish(const CGArgs& a, int set, unsigned tag, float v0, float v1) {
    __shared__ float sh[2][NTH / 32];
    for (int o = 16; o > 0; o >>= 1) {
        v0 += __shfl_down_sync(0xffffffffu, v0, o);
        v1 += __shfl_down_sync(0xffffffffu, v1, o);
    }
    if ((threadIdx.x & 31) == 0) { sh[0][threadIdx.x >> 5] = v0; sh[1][threadIdx.x >> 5] = v1; }
    __syncthreads();
    if (threadIdx.x == 0) {
        v0 = v1 = 0.f;
#pragma unroll
        for (int k = 0; k < NTH / 32; ++k) { v0 += sh[0][k]; v1 += sh[1][k]; }
        st_word(a.red4 + set * a.nw + blockIdx.x, make_float4(v0, v1, 0.f, __uint_as_float(tag)));
    }
}
template <int NTH>
__device__ __forceinline__ bool collect(const CGArgs& a, int set, unsigned tag, float& v0, float& v1) {
    __shared__ float sh[2][NTH / 32];
    int ok = 1;
    v0 = v1 = 0.f;
    for (int b = threadIdx.x; b < a.nw; b += NTH) {
        const float4* p = a.red4 + set * a.nw + b;
        float4 w = ld_word(p);
        if (__float_as_uint(w.w) != tag) {
            const long long t0 = clock64();
            for (int spin = 1;; ++spin) {
                w = ld_word(p);
                if (__float_as_uint(w.w) == tag) break;
                if ((spin & 255) != 0) continue;
                if (ld_acquire_gpu(a.bar + 2) != 0u) { ok = 0; break; }
                if (clock64() - t0 > a.bar_budget) { wait_failed(a); ok = 0; break; }
            }
        }
        v0 += w.x;
        v1 += w.y;
    }
    for (int o = 16; o > 0; o >>= 1) {
        v0 += __shfl_xor_sync(0xffffffffu, v0, o);
        v1 += __shfl_xor_sync(0xffffffffu, v1, o);
    }
    if ((threadIdx.x & 31) == 0) { sh[0][threadIdx.x >> 5] = v0; sh[1][threadIdx.x >> 5] = v1; }
    if (!__syncthreads_and(ok)) return false;
    v0 = v1 = 0.f;
#pragma unroll
    for (int k = 0; k < NTH / 32; ++k) { v0 += sh[0][k]; v1 += sh[1][k]; }
    return true;
}

// Grid-wide barrier of a cooperative launch (every block resident) with a bounded wait.
// Each block's thread 0 publishes the block's writes, arrives on a counter that only
// grows, and waits until the arrivals of this barrier are complete (n per barrier): one
// round trip to the counter after the last arrival.  The counter is zero at launch: the
// launch before, which uses another one, clears it.  A wait longer than
// `budget` SM clock cycles (a block that never arrives) sets the abort word and the
// timeout flag (4) in status[1] with the step in status[2]; blocks that see the abort word
// leave at once.  Returns false when the caller must return: the kernel ends without
// touching the solution any further.
__device__ bool grid_barrier(unsigned* bar, unsigned* abort, unsigned n, unsigned& target,
                             long long budget, int* status, int step) {
    int ok = 1;
    target += n;
    __syncthreads();
    if (threadIdx.x == 0) {
        __threadfence();
        atomicAdd(bar, 1u);
        if ((int)(ld_acquire_gpu(bar) - target) < 0) {
            const long long t0 = clock64();
            for (int spin = 1; (int)(ld_acquire_gpu(bar) - target) < 0; ++spin) {
                if ((spin & 63) != 0) continue;
                if (ld_acquire_gpu(abort) != 0u) { ok = 0; break; }
                if (clock64() - t0 > budget) {
                    atomicExch(abort, 1u);
                    atomicOr(status + 1, 4);
                    atomicCAS(status + 2, 0, step);
                    ok = 0;
                    break;
                }
            }
        }
        __threadfence();
    }
    return __syncthreads_and(ok) != 0;
}

// for i = t0, t0 + gs, ... < n: U indices per round, ld(i) for all of them before
// st(i, value) for any (the loads of a round are independent requests in flight)
template <int U, typename Ld, typename St>
__device__ __forceinline__ void grid_loop(long long t0, long long n, long long gs, Ld&& ld,
                                          St&& st) {
    for (long long i0 = t0; i0 < n; i0 += U * gs) {
        decltype(ld(0LL)) v[U];
#pragma unroll
        for (int u = 0; u < U; ++u)
            if (i0 + u * gs < n) v[u] = ld(i0 + u * gs);
#pragma unroll
        for (int u = 0; u < U; ++u)
            if (i0 + u * gs < n) st(i0 + u * gs, v[u]);
    }
}

// Check of the barrier's bounded wait: every block passes `rounds` barriers, except the
// block `absent` (>= 0), which returns at once; the others' wait then runs out.
// w[1] flags, w[2] the round of a timeout, w[4..7] the barrier, w[8] blocks that
// passed every round.
__global__ void __launch_bounds__(NT) k_barrier_check(int* w, long long budget, int rounds,
                                                      int absent) {
    if ((int)blockIdx.x == absent) return;
    unsigned target = 0;
    for (int r = 1; r <= rounds; ++r)
        if (!grid_barrier(reinterpret_cast<unsigned*>(w + 4),
                          reinterpret_cast<unsigned*>(w + 6), gridDim.x, target, budget, w, r))
            return;
    if (threadIdx.x == 0) atomicAdd(w + 8, 1);
}

// status: 1 not converged, 2 NaN or Inf; the first such step
__device__ __forceinline__ void bad_step(int* status, int flag, int step) {
    atomicOr(status + 1, flag);
    const int old = atomicCAS(status + 2, 0, step);
    if (old > step) atomicMin(status + 2, step);
}

// ||x||^2 of a step from its blocks' shares (one warp, fixed order), checked
__device__ __forceinline__ void norm_total(const double* p, int n, double* out, int* status,
                                           int step) {
    double v0 = 0.0, v1 = 0.0, v2 = 0.0, v3 = 0.0;   // four independent loads in flight
    int k = threadIdx.x;
    for (; k + 96 < n; k += 128) {
        v0 += __ldcg(p + k);
        v1 += __ldcg(p + k + 32);
        v2 += __ldcg(p + k + 64);
        v3 += __ldcg(p + k + 96);
    }
    for (; k < n; k += 32) v0 += __ldcg(p + k);
    double v = (v0 + v1) + (v2 + v3);
    for (int o = 16; o > 0; o >>= 1) v += __shfl_down_sync(0xffffffffu, v, o);
    if (threadIdx.x != 0) return;
    *out = v;
    if (!(v == v) || v > 1e300) bad_step(status, 2, step);
}

// The least-squares fit of b_n by b_{n-1} .. b_{n-nv} (one block): sums the
// partial dot products in a fixed order, updates the Gram matrix of the ring and solves
// the normal equations by a Cholesky factorisation in ring order, newest first (a vector
// whose remainder after the newer ones is below kFitPivot of its square is left out).
// The matrix is scaled to unit diagonal.  Lane i of warp 0 holds row i.
template <bool DF, bool RES> __device__ void fit_block(const CGArgs& a) {
    __shared__ double t[kSums];
    const int lane = threadIdx.x & 31, nwarp = blockDim.x >> 5;
    for (int q = threadIdx.x >> 5; q < kSums; q += nwarp) {
        double v = 0.0;
        if constexpr (RES) {
            // sent by this launch's blocks (bounded wait)
            const float4* p = a.part4 + (long long)q * a.nw;
            const long long t0 = clock64();
            for (int k = lane; k < a.nw; k += 32) {
                float4 w = ld_word(p + k);
                for (int spin = 1; __float_as_uint(w.w) != a.seq; ++spin) {
                    if ((spin & 255) == 0) {
                        if (ld_acquire_gpu(a.bar + 2) != 0u) break;
                        if (clock64() - t0 > a.bar_budget) { wait_failed(a); break; }
                    }
                    w = ld_word(p + k);
                }
                v += __hiloint2double(__float_as_int(w.y), __float_as_int(w.x));
            }
        } else {
            const double* p = a.part + (long long)q * a.nepi;
            for (int k = lane; k < a.nepi; k += 32) v += p[k];
        }
        for (int o = 16; o > 0; o >>= 1) v += __shfl_down_sync(0xffffffffu, v, o);
        // FP32-history sums are scaled by 4^e of this step
        const double un = DF ? pow2d(-2 * scale_of(*a.fit, a.step)) : 1.0;
        if (lane == 0) t[q] = v * un;
    }
    __syncthreads();
    if (threadIdx.x >= 32) return;
    double* gram = a.fit->gram;
    const int s0 = a.bs, si = fslot(s0, min(lane, kFit - 1) + 1);
    const bool row = lane < kFit && lane < a.nv;
    double A[kFit], L[kFit], rs[kFit];
    const double bb = t[0];
    const double dii = row ? gram[si * kSlots + si] : 0.0;
    const double s = row && dii > 0.0 && dii < 1e300 ? rsqrt(dii) : 0.0;
#pragma unroll
    for (int j = 0; j < kFit; ++j) {
        A[j] = row && j < a.nv ? gram[si * kSlots + fslot(s0, j + 1)] : 0.0;
        A[j] *= s * __shfl_sync(0xffffffffu, s, j);
    }
    double g = row ? t[1 + lane] * s : 0.0, y = 0.0, yy = 0.0;
#pragma unroll
    for (int j = 0; j < kFit; ++j) {
        const double v = __shfl_sync(0xffffffffu, A[j], j);
        rs[j] = v > kFitPivot ? rsqrt(v) : 0.0;
        L[j] = lane >= j ? A[j] * rs[j] : 0.0;
#pragma unroll
        for (int k = j + 1; k < kFit; ++k) A[k] -= L[j] * __shfl_sync(0xffffffffu, L[j], k);
        const double yj = __shfl_sync(0xffffffffu, g, j) * rs[j];
        if (lane == j) y = yj;
        g -= L[j] * yj;
        yy += yj * yj;
    }
    double c = 0.0;
#pragma unroll
    for (int j = kFit - 1; j >= 0; --j) {
        const double cj = __shfl_sync(0xffffffffu, y, j) * rs[j];
        if (lane == j) c = cj * s;
#pragma unroll
        for (int k = 0; k < j; ++k) {
            const double ljk = __shfl_sync(0xffffffffu, L[k], j);
            if (lane == k) y -= ljk * cj;
        }
    }
    double mag = fabs(c);
    for (int o = 4; o > 0; o >>= 1) mag = fmax(mag, __shfl_xor_sync(0xffffffffu, mag, o));
    FitRecord& rec = a.fit->rec[(a.step + 1) & 1];
    if (lane < kFit) {
        rec.c[lane] = c;
        rec.cf[lane] = (float)c;
    }
    if (lane == 0) {
        // a poor or degenerate fit (also NaN anywhere in it) falls back to extrapolation
        rec.use = a.nv >= 3 && bb > 0.0 && bb - yy <= kFitPoor * bb && mag < 1e4;
        // 2^e near 1 / rms(b), from the exponents alone
        const double mean = bb / (3.0 * (double)a.nact);
        const int lim = DF ? 120 : 500, ex = ((__double2hiint(mean) >> 20) & 2047) - 1023;
        rec.e = mean > 0.0 && ex < 1024 ? max(-lim, min(lim, -(ex >> 1))) : 0;
        gram[s0 * kSlots + s0] = bb;
    }
    if (row) {
        gram[s0 * kSlots + si] = t[1 + lane];
        gram[si * kSlots + s0] = t[1 + lane];
    }
}

// r = b - A x in FP64 at the active voxels, scaled by sc and rounded to FP32, with (not RES)
// d_0 = r / theta; adds |r|^2 (and |b|^2 on the first pass) to the thread's sums.
// Where there are fewer active voxels than lanes on the GPU (SPLIT), a warp takes one
// component of its 32 voxels: the pass is bound by the FP64 chain of a voxel, and three
// warps on three sub-partitions run a third of it each.  Warps are dealt to the blocks in
// turn, so that few voxels spread over many SMs.
template <int C>
__device__ __forceinline__ double applyA64_row(const CGArgs& a, const double* __restrict__ x, int m,
                                               int mask) {
    const long long M = a.M;
    constexpr int C1 = C == 0 ? 1 : 0, C2 = C == 2 ? 1 : 2;      // the other two components
    constexpr int K1 = C == 2 ? 4 : 3;                           // coupling (C, C1)
    constexpr int K2 = C == 0 ? 4 : 5;                           // coupling (C, C2)
    double o = (a.diag[m] - c_stencil[13 * 6 + C]) * x[C * M + m];
    double o1 = 0.0;
    Unroll13::run([&](auto ec) {
        constexpr int E = decltype(ec)::value;
        constexpr int d[3] = {E % 3 - 1, (E / 3) % 3 - 1, E / 9 - 1};
        const bool inp = mask & (1 << E), inm = mask & (1 << (26 - E));
        const long long mp = m + a.noff[E], mm = m + a.noff[26 - E];
        o -= c_stencil[E * 6 + C] * ((inp ? x[C * M + mp] : 0.0) + (inm ? x[C * M + mm] : 0.0));
        if constexpr (d[C] != 0 && d[C1] != 0)
            o1 -= c_stencil[E * 6 + K1] * ((inp ? x[C1 * M + mp] : 0.0) + (inm ? x[C1 * M + mm] : 0.0));
        if constexpr (d[C] != 0 && d[C2] != 0)
            o1 -= c_stencil[E * 6 + K2] * ((inp ? x[C2 * M + mp] : 0.0) + (inm ? x[C2 * M + mm] : 0.0));
    });
    return o + o1;
}

template <bool SPLIT, bool RES>
__device__ __forceinline__ void residual64(const CGArgs& a, int e, bool first, bool wide, Sums& sum) {
    const long long M = a.M;
    const double sc = pow2d(e);
    const int lane = threadIdx.x & 31;
    const long long warp = (long long)(threadIdx.x >> 5) * a.nw + blockIdx.x;
    const long long warps = (long long)(blockDim.x >> 5) * a.nw;
    // one component: sums of the scaled values, r in FP32
    auto part = [&](double b, double r) {
        const float rs = (float)(r * sc);
        sum.rr += rs * rs;
        if (first) {
            const float bs = (float)(b * sc);
            sum.bb += bs * bs;
        }
        if (wide) { sum.rrw += r * r; sum.bbw += b * b; }
        return rs;
    };
    if constexpr (SPLIT) {
        const long long groups = (a.nact + 31) / 32;
        float* rf = reinterpret_cast<float*>(a.r);
        float* pf = reinterpret_cast<float*>(a.p);
        for (long long w = warp; w < 3 * groups; w += warps) {
            const int c = (int)(w / groups);
            const long long i = (w % groups) * 32 + lane;
            if (i >= a.nact) continue;
            const int m = a.act[i], mask = a.nmask[i];
            double o;
            if (c == 0) o = applyA64_row<0>(a, a.x, m, mask);
            else if (c == 1) o = applyA64_row<1>(a, a.x, m, mask);
            else o = applyA64_row<2>(a, a.x, m, mask);
            const double b = a.b[c * M + m];
            const float rs = part(b, b - o);
            rf[4LL * m + c] = rs;
            if (!RES) pf[4LL * m + c] = rs * a.inv_theta;
        }
    } else {
        for (long long i = warp * 32 + lane; i < a.nact; i += warps * 32) {
            const int m = a.act[i];
            double o[3];
            applyA64(a, a.x, m, a.nmask[i], o);
            float rs[3];
#pragma unroll
            for (int k = 0; k < 3; ++k) {
                const double b = a.b[k * M + m];
                rs[k] = part(b, b - o[k]);
            }
            a.r[m] = make_float4(rs[0], rs[1], rs[2], 0.f);
            if (!RES)
                a.p[m] = make_float4(rs[0] * a.inv_theta, rs[1] * a.inv_theta, rs[2] * a.inv_theta, 0.f);
        }
    }
}

// The solve of one step.  Resident tiles (RES) first form the right-hand side and the start of
// their own voxels (epi_voxel); in FP32-history the start goes to the neighbours as tagged
// words like the iteration's d, in FP64 a grid barrier follows, because the FP64 residual
// deals the voxels out anew.  Blocks past nw take the voxels outside every tile.  The norm
// of a step is added up beside the next one's solve, not by the last block to finish.
// Against an epilogue of its own and a last block (solve phase of a step): 9^3 sphere
// FP32-history 43.2 -> 35.5 us, 32^3 52.6 -> 40.9, 133 x 27 x 21 116 -> 95, 8^3 FP64 49.9 -> 45.0
// (36.9, 44.4, 102 and 46.8 with the aims of `need` below, two iterations more).
// What remains of the 9^3 solve, thousands of cycles: right-hand side 13, residual 11, two
// iterations beside the sums 5, the sums 1, eleven iterations 25, x and its norm 4.
//
// Mixed-precision iterative refinement from x0: residual r = b - A x (FP64, or
// double-float in FP32-history mode, DF), FP32 Chebyshev iterations for A e = r, x += e.
// One fused pass and one grid barrier per iteration (apply to d_k, update e, r, d_{k+1}; d
// is double-buffered because neighbours read d_k during the pass).  The iteration's own
// residual (r is carried, r -= A d_k in FP32) differs from that of x + e by a few FP32
// roundings of the *start* residual, so once it is below the tolerance with kDrift of the
// start residual added, the step is done without forming b - A x again; otherwise the next
// refinement starts from a new true residual.  All blocks take identical decisions because
// every block sums the same per-block partials in the same order.
//   RES: a block has at most one tile (see Resident; no grid barrier in the iteration).  In
//     FP32-history the first two iterations run while the sums of the residual are still
//     on their way: at least three are made anyway, and x is not touched by them.
//   SPLIT: FP64 residual by components (see residual64).
// The scalars that steer the iteration are FP32 numbers scaled by powers of two (an FP64
// square root, logarithm and division for every warp cost 4 to 7 us of a 45 us solve).  Sums
// that leave FP32's range at the scale of the step before (wide) are formed again in FP64,
// which gives the new scale.
// kDrift: the carried residual was at most 2.9e-7 of the start residual away from that of
// x + e in 32,000 refinements of 3 to 64 iterations (cubes, cores, films and noise, eps_r 1.001
// to 1000, spectral intervals 3 to 10,000 wide, rough and smooth residuals): the width comes from
// the diagonal, which scales a voxel's error with its own residual, not from G_0.
constexpr float kDrift = 1e-6f;
constexpr float kFloor = 1e-6f;
// A refinement aims at a tenth of the tolerance but may fall short of it by kFloor; what it then
// leaves just below the tolerance (half of the FP64 steps of a field that the fit follows to 1e-7)
// would be 5 times the usual error.  One more refinement of three iterations or so follows.
constexpr float kNear = 0.2f;
// sequence numbers that a residual and two iterations whose results are dropped may have used
constexpr unsigned kAborted = 4;

template <bool DF, class T, bool RES, bool SPLIT>
__global__ void __launch_bounds__(T::NTH, RES ? 4 : 2)
k_cg(const __grid_constant__ CGArgs a, const __grid_constant__ EpiArgs ep) {
    typedef typename std::conditional<DF, float, double>::type R;
    __shared__ __align__(16) float4 sd[2][T::HALO];      // tile halos of the passes
    pdl_trigger();                       // (launched as an ordinary, cooperative kernel)
    if ((int)blockIdx.x == a.nw) {       // the fit for the next step, beside the solve
        if (a.norm_prev && threadIdx.x < 32)
            norm_total(a.nrm_prev, a.nred, a.norm_prev, a.status, a.prev_step);
        fit_block<DF, RES>(a);
        return;
    }
    if constexpr (RES) {
        if ((int)blockIdx.x > a.nw) {    // voxels outside every tile
            const EpiFit<R> fit(ep);
            EpiSums<R> sum;
            float4 none;
            for (int i = ((int)blockIdx.x - a.nw - 1) * T::NTH + threadIdx.x; i < a.nvac;
                 i += a.nvb * T::NTH)
                epi_voxel<R>(ep, ep.adj, fit, a.vac[i], sum, none);
            epi_vacuum_norm(sum.xin, a.nrm + blockIdx.x - 1);
            return;
        }
    }
    if (blockIdx.x == 0 && threadIdx.x == 0) a.bar[a.parity ^ 1] = 0u;
    unsigned target = 0, seq = a.seq, tag = a.seq, xtag = a.seq;
    int set = 0;
    auto gsync = [&] {
        return grid_barrier(a.bar + a.parity, a.bar + 2, a.nw, target, a.bar_budget, a.status, a.step);
    };
    const long long M = a.M;
    const long long t0 = (long long)blockIdx.x * T::NTH + threadIdx.x;
    const long long gs = (long long)a.nw * T::NTH;
    const int nb = a.nw;
    double* red0 = a.red;
    double* red1 = a.red + nb;
    Resident<T> res;
    double xin = 0.0;                    // |x|^2 of the tile's vacuum voxels
    __shared__ EpiRed<R, T::NTH> fitred;
    bool fit_due = RES;                  // the block's sums for the fit are still to be sent
    auto fit_sums = [&] {
        if constexpr (RES) {
            if (!fit_due) return;
            fit_due = false;
            if (threadIdx.x >= T::NTH - 32 && (threadIdx.x & 31) < kSums) {
                const double v = epi_block_sum<R, T::NTH>(fitred);
                st_word(a.part4 + (threadIdx.x & 31) * nb + blockIdx.x,
                        make_float4(__int_as_float(__double2loint(v)),
                                    __int_as_float(__double2hiint(v)), 0.f, __uint_as_float(a.seq)));
            }
        }
    };
    if constexpr (RES) {
        const EpiFit<R> fit(ep);
        resident_init<T>(a, res, sd);
        // right-hand side and start of the tile's voxels
        EpiSums<R> sum;
        if ((int)blockIdx.x < a.ntiles) {
            const int org = a.tiles[blockIdx.x];
            int lx, ly, lz;
            T::local(lx, ly, lz);
#pragma unroll 1
            for (int v = 0; v < T::VPT; ++v) {
                const long long m = tile_voxel<T>(a, org, v);
                float4 x0 = make_float4(0.f, 0.f, 0.f, 0.f);
                if (m >= 0 && epi_voxel<R>(ep, ep.adj, fit, m, sum, x0) && DF) {
                    x0.w = __uint_as_float(xtag);
                    st_word(a.xl + m, x0);
                }
                if (DF) sd[0][T::hidx(lx, ly, lz + v)] = x0;
            }
        }
        xin = sum.xin;
        epi_stash<R, T::NTH>(fitred, sum);
        // the zeros of the shells before a pass writes halos over them; FP64: the start and b
        // before other blocks read them
        if constexpr (DF) {
            __syncthreads();
            fit_sums();
        } else if (!gsync()) {
            return;
        }
    }
    float bb = 0.f, rr = 0.f;            // scaled by 4^e0 and 4^e
    double xx = 0.0;                     // |x|^2 of the block's share, once x is stored
    int e = scale_of(*a.fit, a.step), e0 = e;
    int its = 0, outer = 0, wides = 0;
    bool first = true, wide = false, converged = false, nonfinite = false, zero = false;
    bool stored = false;     // x is in a.x; else DF's start is in xb only
    bool own = true;         // sd[0] holds the tile's start
    bool rescaled = false;   // e0 comes from FP64 sums
    bool polished = false;   // a residual that met the tolerance is being refined (kNear)
    // f(voxel, its correction e) over the block's share of the active voxels
    auto each = [&](auto&& f) {
        if constexpr (RES) {
#pragma unroll
            for (int v = 0; v < T::VPT; ++v)
                if (res.m[v] >= 0) f(res.m[v], res.e[v], v);
        } else {
            struct ME { int m; float4 e; };
            grid_loop<4>(t0, a.nact, gs,
                [&](long long i) {
                    ME v;
                    v.m = a.act[i];
                    v.e = a.e[v.m];
                    return v;
                },
                [&](long long, const ME& v) { f(v.m, v.e, 0); });
        }
    };
    while (true) {
        // ---- residual, scaled by 2^e
        Sums sum = {0.f, 0.f, 0.0, 0.0};
        if constexpr (DF) {
            if (!(stored ? residual_df_tiled<T, true, RES>(a, sd, pow2f(e), wide, sum, res, seq, xtag, own)
                         : residual_df_tiled<T, false, RES>(a, sd, pow2f(e), wide, sum, res, seq, xtag, own)))
                return;
            own = false;
        } else {
            residual64<SPLIT, RES>(a, e, first, wide, sum);
        }
        if (wide) {                      // sums in FP64: the true scale, or none
            block_sum2<T::NTH>(sum.rrw, sum.bbw);
            if (threadIdx.x == 0) { red0[blockIdx.x] = sum.rrw; red1[blockIdx.x] = sum.bbw; }
            if (!gsync()) return;
            const double rw = grid_total(red0, nb), bw = grid_total(red1, nb);
            if (!(rw <= 1e300) || !(bw <= 1e300)) { nonfinite = true; break; }
            if (bw == 0.0) { zero = converged = true; break; }
            int ex = 0;
            frexp(sqrt(first ? bw : rw), &ex);
            e = max(-(DF ? 120 : 500), min(DF ? 120 : 500, -ex));
            if (first) {
                e0 = e;
                rescaled = true;
            }
            wide = false;
            seq += kAborted;
            if (!gsync()) return;
            continue;
        }
        publish<T::NTH>(a, set, ++tag, sum.rr, sum.bb);
        float rr_p = 0.f;
        constexpr bool early = RES && DF;     // iterate while the sums travel
        bool ran2 = false;
        if constexpr (RES) {
#pragma unroll
            for (int v = 0; v < T::VPT; ++v) res.e[v] = make_float4(0.f, 0.f, 0.f, 0.f);
        }
        if (early && !stored) {
            for (int k = 0; k < 2; ++k)
                if (!cheb_pass_resident<T, false>(a, k, seq + k, false, sd, res, rr_p)) return;
            ran2 = true;
        } else {
            fit_sums();
            if (!gsync()) return;        // r complete (with x as pairs: q read by all)
        }
        float b_tot;
        if (!collect<T::NTH>(a, set, tag, rr, b_tot)) return;
        set ^= 1;
        if (first) bb = b_tot;
        const float sb = sqrtf(bb), goal = a.tol * sb * pow2f(max(-120, min(120, e - e0))),
                    have = sqrtf(rr);
        // a NaN or Inf in the sums, a vanishing right-hand side or a scale far off
        const bool off = !(rr <= 1e14f) || (first && !(bb >= 1e-10f && bb <= 1e14f)) ||
                         (!first && have > goal && rr < 1e-30f);
        const bool odd = off && ++wides <= 3;      // (the FP64 sums settle it the first time)
        if (!odd && !(rr <= 1e30f)) { nonfinite = true; break; }
        if (!odd && have <= goal) {
            // a residual formed anew that lies near the tolerance is refined once more
            if (polished || have <= kNear * goal || outer >= a.max_outer || its >= a.max_iter) {
                converged = true;
                break;
            }
            polished = true;
        }
        if (odd || (first && rr > bb)) {
            if (!odd) {
                // a start worse than none (an abrupt change of the excitation): from zero
                each([&](long long m, const float4&, int) {
#pragma unroll
                    for (int k = 0; k < 3; ++k) {
                        if (DF) a.xb[k * M + m].x = 0.f;
                        else a.x[k * M + m] = 0.0;
                    }
                    if (DF) st_word(a.xl + m, make_float4(0.f, 0.f, 0.f, __uint_as_float(xtag + 1u)));
                });
                ++xtag;
                first = false;
            }
            wide = odd;
            seq += kAborted;
            if (!gsync()) return;
            continue;
        }
        first = false;
        if (outer >= a.max_outer || its >= a.max_iter) break;
        // ---- Chebyshev: iterations for the reduction still needed, never asking for more
        // than FP32 can deliver in one refinement (kFloor), and below the tolerance: what a step
        // leaves adds up along smooth modes.  FP64 at a hundredth instead of a tenth: 7 x 8 x 9
        // cube, eps_r 30, 1.1e-13 -> 3.3e-14 from the exact march, 9^3 sphere 4.7e-14 -> 1.8e-14, 8^3
        // cube 2.0e-14 -> 6.5e-15, for two iterations of 30.  FP32-history at a tenth instead of 0.8: 24^3
        // cube 9.6e-7 -> 9.1e-7 from FP64, 66 x 27 x 21 noise 1.35e-6 -> 1.29e-6, the errors of
        // 10 and 100 times smaller tolerances, for two iterations of 15
        const float need = fmaxf((DF ? 0.1f : 0.01f) * (goal - kDrift * have) / have, kFloor);
        const int n_it = min(a.n_cheb, max(3, (int)ceilf(log2f(0.5f * need) * a.inv_log2_rate)));
        if constexpr (RES) {
            if constexpr (!DF) {
#pragma unroll
                for (int v = 0; v < T::VPT; ++v) {
                    if (res.m[v] < 0) continue;
                    const float4 r = __ldcg(a.r + res.m[v]);
                    res.r[v] = r;
                    res.d[v] = make_float4(r.x * a.inv_theta, r.y * a.inv_theta, r.z * a.inv_theta, 0.f);
                }
            }
            for (int k = ran2 ? 2 : 0; k < n_it; ++k)
                if (!cheb_pass_resident<T, !DF>(a, k, seq + k, k == n_it - 1, sd, res, rr_p)) return;
            seq += n_it;
        } else {
            float4* dk = a.p;
            float4* dn = a.q;
            for (int k = 0; k < n_it; ++k) {
                cheb_pass_tiled<T>(a, dk, dn, a.c1[k], a.c2[k], k == 0, k == n_it - 1, sd, rr_p);
                if (k < n_it - 1 && !gsync()) return;
                float4* tmp = dk; dk = dn; dn = tmp;
            }
        }
        its += n_it;
        ++outer;
        publish<T::NTH>(a, set, ++tag, rr_p, 0.f);
        if (!RES && !gsync()) return;    // the update deals the voxels out by list
        // ---- x += e / 2^e (DF: the float start becomes an FP64 x)
        const double back = pow2d(-e);
        xx = 0.0;
        each([&](long long m, const float4& d, int) {
            const float ec[3] = {d.x, d.y, d.z};
#pragma unroll
            for (int k = 0; k < 3; ++k) {
                double x = DF && !stored ? widen(a.xb[k * M + m].x) : a.x[k * M + m];
                x += back * widen(ec[k]);
                a.x[k * M + m] = x;
                if (a.out) a.out[m * 3 + k] = x;
                if (DF) a.xb[k * M + m].x = (float)x;
                xx += x * x;
            }
        });
        stored = true;
        float left, dummy;
        if (!collect<T::NTH>(a, set, tag, left, dummy)) return;
        set ^= 1;
        left = sqrtf(left);
        if (left + kDrift * have <= goal) { converged = true; break; }
        if (!(left <= 1e14f)) { nonfinite = true; break; }
        // ---- not there yet: a new residual (DF: of x as float pairs)
        e = max(-(DF ? 120 : 500), min(DF ? 120 : 500,
                e - (((__float_as_int(fmaxf(left, 1e-37f)) >> 23) & 255) - 127)));
        if constexpr (DF) {
            if (!gsync()) return;        // q: every block is done with its halo words
            each([&](long long m, const float4&, int) {
                float4 h, l;
                df_split(a.x[m], h.x, l.x);
                df_split(a.x[M + m], h.y, l.y);
                df_split(a.x[2 * M + m], h.z, l.z);
                h.w = 0.f;
                l.w = __uint_as_float(a.seq + 1023u);    // no launch's tag of a start
                a.q[m] = h;
                a.xl[m] = l;
            });
        }
        if (!gsync()) return;
    }
    // ---- an x not stored yet, and its norm.  NaN or Inf in the right-hand side or the
    // start: no iteration can help; J_n is returned as NaN so that the monitor and the
    // caller see it
    if (!stored || nonfinite) {
        xx = 0.0;
        each([&](long long m, const float4&, int) {
#pragma unroll
            for (int k = 0; k < 3; ++k) {
                double x = DF && !stored ? widen(a.xb[k * M + m].x) : a.x[k * M + m];
                if (zero) x = 0.0;
                if (nonfinite) x = __longlong_as_double(0x7ff8000000000000LL);
                a.x[k * M + m] = x;
                if (a.out) a.out[m * 3 + k] = x;
                if (DF) a.xb[k * M + m].x = (float)x;
                xx += x * x;
            }
        });
    }
    fit_sums();
    xx += xin;
    __shared__ double shx[T::NTH / 32];
    for (int o = 16; o > 0; o >>= 1) xx += __shfl_down_sync(0xffffffffu, xx, o);
    if ((threadIdx.x & 31) == 0) shx[threadIdx.x >> 5] = xx;
    __syncthreads();
    if (threadIdx.x != 0) return;
#pragma unroll
    for (int w = 1; w < T::NTH / 32; ++w) xx += shx[w];
    a.nrm[blockIdx.x] = xx;
    if (blockIdx.x == 0) {
        a.fit->wide[(a.step + 1) & 1] = rescaled ? kWide + e0 : 0;
        a.status[0] = its;
        a.status[3] += its;
        const int flag = nonfinite ? 2 : converged ? 0 : 1;
        if (flag) bad_step(a.status, flag, a.step);
    }
}

// ||x||^2 of a march's last step (the others are added up beside the solve that follows)
__global__ void k_norm_total(const double* nrm, int n, double* out, int* status, int step) {
    norm_total(nrm, n, out, status, step);
}

__global__ void k_from_aos(const double* __restrict__ in, long long M, double* __restrict__ x) {
    const long long i = (long long)blockIdx.x * blockDim.x + threadIdx.x;
    if (i >= 3 * M) return;
    const long long m = i / 3;
    const int c = (int)(i % 3);
    x[c * M + m] = in[i];
}

// ---------------------------------------------------------------- adjoint march
// In adjoint time tau = N + 1 - n the ring holds lambda.  With mu = chi lambda,
//   Z_0^T lambda_n = g_n - sum_{l>=1} Z_l^T lambda_{n+l},
//   Z_l^T lambda = (T(l)/eps + delta_l) lambda - G_l * (chi lambda)      (G_l^T = G_l),
// and Z_0^T lambda = A mu with the same symmetric A as the forward solve (k_epilogue with
// ADJ: b = rhs on active voxels, the start in terms of mu).
// lambda = mu / chi on active voxels; on vacuum voxels (chi = 0) the row of Z_0^T reads
// (T(0) + delta_0) lambda_m - (G_0 * mu)_m = rhs_m, so lambda_m = (rhs_m + (G_0 * mu)_m)
// / (T(0) + delta_0).  Gradient accumulation on active voxels:
//   dO/dchi_m += lambda_n,m . (1/chi_m) sum_l (T(l) + delta_l) J_{n-l,m}
// (the chi-derivative of row m of the forward system, simplified with that row's own
// equation), and optional AoS output of lambda_n.  Two launches: the first turns mu
// into lambda on active voxels only after the second has read mu around vacuum ones.
__global__ void k_adj_vacuum(long long M, int U, int V, int W, const double* __restrict__ f,
                             const double* __restrict__ mu, const double* __restrict__ rhs,
                             double* __restrict__ lam_vac) {
    const long long m = (long long)blockIdx.x * blockDim.x + threadIdx.x;
    if (m >= M) return;
    if (f[M + m] > 0.0) return;
    const int u = (int)(m % U), v = (int)((m / U) % V), w = (int)(m / ((long long)U * V));
    double o[3] = {0.0, 0.0, 0.0};
    for (int ez = -1; ez <= 1; ++ez)
        for (int ey = -1; ey <= 1; ++ey)
            for (int ex = -1; ex <= 1; ++ex) {
                const int u2 = u + ex, v2 = v + ey, w2 = w + ez;
                if (u2 < 0 || u2 >= U || v2 < 0 || v2 >= V || w2 < 0 || w2 >= W) continue;
                const long long m2 = ((long long)w2 * V + v2) * U + u2;
                const double* S = c_stencil + ((ez + 1) * 9 + (ey + 1) * 3 + (ex + 1)) * 6;
                const double X = mu[m2], Y = mu[M + m2], Z = mu[2 * M + m2];
                o[0] += S[0] * X + S[3] * Y + S[4] * Z;
                o[1] += S[3] * X + S[1] * Y + S[5] * Z;
                o[2] += S[4] * X + S[5] * Y + S[2] * Z;
            }
    for (int beta = 0; beta < 3; ++beta)
        lam_vac[beta * M + m] = (rhs[beta * M + m] + o[beta]) * f[2 * M + m];
}

__global__ void k_adj_post(long long M, const double* __restrict__ f, double* __restrict__ Ln,
                           const double* __restrict__ lam_vac, const double* __restrict__ J,
                           int j_first, int n, Taps tp, double* __restrict__ grad_chi,
                           double* __restrict__ lam_out) {
    const long long m = (long long)blockIdx.x * blockDim.x + threadIdx.x;
    if (m >= M) return;
    const double ichi = f[M + m];
    double gsum = 0.0;
    for (int beta = 0; beta < 3; ++beta) {
        double lam;
        if (ichi > 0.0) {
            lam = Ln[beta * M + m] * ichi;
            double q = 0.0;
            const int L = tp.n > 2 ? tp.n : 2;
            for (int l = 0; l < L && n - l >= 1; ++l) {   // J[0] holds step j_first
                const double w = (l < 2 ? 0.5 : 0.0) + (l < tp.n ? tp.d[l] : 0.0);
                q += w * J[((long long)(n - l - j_first) * M + m) * 3 + beta];
            }
            gsum += lam * q * ichi;
        } else {
            lam = lam_vac[beta * M + m];
        }
        Ln[beta * M + m] = lam;
        if (lam_out) lam_out[m * 3 + beta] = lam;
    }
    grad_chi[m] += gsum;
}

// P_{n-1} = T(1)/eps J_{n-1} + sum_{l=1}^{L-1} delta_l J_{n-l} - chi (G * J)_hist, AoS out
template <typename R>
__global__ void k_history_out(long long M, const double* __restrict__ eps,
                              const double* __restrict__ chi, const R* __restrict__ hist,
                              const double* __restrict__ Jring, int s0, int jring, Taps tp,
                              double* __restrict__ out) {
    const long long i = (long long)blockIdx.x * blockDim.x + threadIdx.x;
    if (i >= 3 * M) return;
    const long long m = i % M;
    const int beta = (int)(i / M);
    const long long st = 3 * M;
    double P = 0.5 / eps[m] * Jring[jslot(s0, 1, jring, st) + i] - chi[m] * (double)hist[i];
    for (int l = 1; l < tp.n; ++l) P += tp.d[l] * Jring[jslot(s0, l, jring, st) + i];
    out[m * 3 + beta] = P;
}

// y = A x (FP64) on active voxels, for the setup-time eigenvalue estimate
__global__ void k_apply64(const __grid_constant__ CGArgs a, const double* __restrict__ x,
                          double* __restrict__ y) {
    const long long i = (long long)blockIdx.x * blockDim.x + threadIdx.x;
    if (i >= a.nact) return;
    const int m = a.act[i];
    double o[3];
    applyA64(a, x, m, a.nmask[i], o);
    y[m] = o[0];
    y[a.M + m] = o[1];
    y[2 * a.M + m] = o[2];
}

// The setup's Lanczos recurrence with its scalars on the device (sc[2 j] = alpha_j,
// sc[2 j + 1] = ||w||^2 after step j): partial sums per block, added up by every block of
// the next kernel in the same order.
constexpr int kLzBlocks = NT;
__device__ __forceinline__ double lz_sum(const double* part) {
    double s = part[threadIdx.x], d = 0.0;      // one partial per thread
    block_sum2<NT>(s, d);
    return s;
}
__global__ void __launch_bounds__(NT) k_lz_dot(const double* __restrict__ x, const double* __restrict__ y,
                                               long long n, double* __restrict__ part) {
    double s = 0.0, d = 0.0;
    for (long long i = (long long)blockIdx.x * NT + threadIdx.x; i < n; i += (long long)gridDim.x * NT)
        s += x[i] * y[i];
    block_sum2<NT>(s, d);
    if (threadIdx.x == 0) part[blockIdx.x] = s;
}
// w -= alpha v + beta u with alpha = sum(part_in), beta^2 = *b2 (0: none); partial |w|^2
__global__ void __launch_bounds__(NT) k_lz_step(double* __restrict__ w, const double* __restrict__ v,
                                                const double* __restrict__ u,
                                                const double* __restrict__ part_in,
                                                const double* __restrict__ b2, long long n,
                                                double* __restrict__ alpha_out,
                                                double* __restrict__ part) {
    const double alpha = lz_sum(part_in), beta = b2 ? sqrt(*b2) : 0.0;
    double s = 0.0, d = 0.0;
    for (long long i = (long long)blockIdx.x * NT + threadIdx.x; i < n; i += (long long)gridDim.x * NT) {
        const double r = w[i] - (alpha * v[i] + (b2 ? beta * u[i] : 0.0));
        w[i] = r;
        s += r * r;
    }
    block_sum2<NT>(s, d);
    if (threadIdx.x == 0) part[blockIdx.x] = s;
    if (blockIdx.x == 0 && threadIdx.x == 0) *alpha_out = alpha;
}
// w /= ||w|| (left alone when it vanished: the host stops there); ||w||^2 out
__global__ void __launch_bounds__(NT) k_lz_scale(double* __restrict__ w, const double* __restrict__ part_in,
                                                 long long n, double* __restrict__ b2_out) {
    const double b2 = lz_sum(part_in);
    const double f = b2 > 0.0 ? 1.0 / sqrt(b2) : 0.0;
    for (long long i = (long long)blockIdx.x * NT + threadIdx.x; i < n; i += (long long)gridDim.x * NT)
        w[i] *= f;
    if (blockIdx.x == 0 && threadIdx.x == 0) *b2_out = b2;
}

}  // namespace

namespace mot {

void stencil_setup(mot_ctx* c) {
    // lag-0 elements of the 8 octant offsets in {0,1}^3 (window index 0 is lag 0 there)
    std::vector<double> oct(8 * 6);
    std::vector<double> row(6 * WIN);
    const long long U = c->U, V = c->V;
    for (int ez = 0; ez <= 1; ++ez)
        for (int ey = 0; ey <= 1; ++ey)
            for (int ex = 0; ex <= 1; ++ex) {
                for (int cc = 0; cc < 6; ++cc) oct[((ez * 2 + ey) * 2 + ex) * 6 + cc] = 0.0;
                if (ex >= c->U || ey >= c->V || ez >= c->W) continue;
                const long long o = ((long long)ez * V + ey) * U + ex;
                MOT_CUDA_TRY(cudaMemcpy(row.data(), c->tab + o * 6 * WIN, sizeof(double) * 6 * WIN,
                                        cudaMemcpyDeviceToHost));
                for (int cc = 0; cc < 6; ++cc) oct[((ez * 2 + ey) * 2 + ex) * 6 + cc] = row[cc * WIN];
            }
    for (int ez = -1; ez <= 1; ++ez)
        for (int ey = -1; ey <= 1; ++ey)
            for (int ex = -1; ex <= 1; ++ex) {
                const int k = ((ez + 1) * 9 + (ey + 1) * 3 + (ex + 1)) * 6;
                const double* src = &oct[((std::abs(ez) * 2 + std::abs(ey)) * 2 + std::abs(ex)) * 6];
                const int sx = ex < 0 ? -1 : 1, sy = ey < 0 ? -1 : 1, sz = ez < 0 ? -1 : 1;
                c->stencil[k + 0] = src[0];
                c->stencil[k + 1] = src[1];
                c->stencil[k + 2] = src[2];
                // component (a, b), a != b, is odd in d_a and in d_b: exactly zero when
                // either offset coordinate is 0 (the stencil kernels skip those products)
                c->stencil[k + 3] = (ex && ey) ? src[3] * sx * sy : 0.0;
                c->stencil[k + 4] = (ex && ez) ? src[4] * sx * sz : 0.0;
                c->stencil[k + 5] = (ey && ez) ? src[5] * sy * sz : 0.0;
            }
    // The stencil constants are shared by every context on the device: G_0 at offsets
    // |d_i| <= 1 depends on the unit voxel only, so all contexts compute the same
    // values.  A grid of extent 1 along some axis lacks those neighbours (its entries
    // are zero, and masked out of its own stencil), so it writes the constants only
    // while no complete stencil is there.
    const bool complete = c->U > 1 && c->V > 1 && c->W > 1;
    int dev = 0;
    MOT_CUDA_TRY(cudaGetDevice(&dev));
    static bool have_complete[64] = {};
    if (complete || dev >= 64 || !have_complete[dev]) {
        upload_symbol(c_stencil, c->stencil, sizeof(double) * 27 * 6, c->stream);
        float st32[27 * 6];
        float stl[27 * 6];
        for (int k = 0; k < 27 * 6; ++k) {
            st32[k] = (float)c->stencil[k];
            stl[k] = (float)(c->stencil[k] - (double)st32[k]);
        }
        upload_symbol(c_st32, st32, sizeof st32, c->stream);
        upload_symbol(c_stl, stl, sizeof stl, c->stream);
        if (complete && dev < 64) have_complete[dev] = true;
    }
    int noff[27];
    for (int ez = -1; ez <= 1; ++ez)
        for (int ey = -1; ey <= 1; ++ey)
            for (int ex = -1; ex <= 1; ++ex)
                noff[(ez + 1) * 9 + (ey + 1) * 3 + (ex + 1)] = ex + c->U * (ey + c->V * ez);
    for (int e = 0; e < 27; ++e) c->noff[e] = noff[e];
    if (c->n_taps > MAXTAPS) throw MotError{MOT_ERR_ARG, "at most 64 FIR taps are supported"};
    int khz = 0;
    MOT_CUDA_TRY(cudaDeviceGetAttribute(&khz, cudaDevAttrClockRate, c->device));
    c->bar_budget = (long long)(kBarrierBudgetS * 1e3 * std::max(khz, 1000000));
}

namespace {

// number of eigenvalues of the symmetric tridiagonal (al, be) below x (Sturm count)
int sturm_count(const std::vector<double>& al, const std::vector<double>& be, double x) {
    int cnt = 0;
    double q = 1.0;
    for (size_t i = 0; i < al.size(); ++i) {
        const double b2 = i ? be[i] * be[i] : 0.0;
        q = al[i] - x - (i ? b2 / q : 0.0);
        if (q == 0.0) q = -1e-300;
        if (q < 0.0) ++cnt;
    }
    return cnt;
}

double tridiag_eig(const std::vector<double>& al, const std::vector<double>& be, int k,
                   double lo, double hi) {
    for (int it = 0; it < 200; ++it) {
        const double mid = 0.5 * (lo + hi);
        if (sturm_count(al, be, mid) > k) hi = mid; else lo = mid;
    }
    return 0.5 * (lo + hi);
}

}  // namespace

// Spectral bounds of A = diag(1/chi) Z_0 on the active voxels by 40 Lanczos steps from a
// seeded start vector, and the Chebyshev coefficients for the inner solve:
// [a, b] = [theta_min, 1.02 theta_max] of the Ritz values (modes below a still
// converge; the bound above keeps every mode in (0, a + b)).
void chebyshev_setup(mot_ctx* c) {
    const long long n3 = 3 * c->M;
    constexpr int kSteps = 40;
    double *v0 = nullptr, *v1 = nullptr, *w = nullptr, *part = nullptr;
    MOT_CUDA_TRY(cudaMalloc(&v0, sizeof(double) * n3));
    MOT_CUDA_TRY(cudaMalloc(&v1, sizeof(double) * n3));
    MOT_CUDA_TRY(cudaMalloc(&w, sizeof(double) * n3));
    // two sets of partial sums, then the scalars of every step (read once at the end)
    MOT_CUDA_TRY(cudaMalloc(&part, sizeof(double) * (2 * kLzBlocks + 2 * kSteps)));
    double *pa = part, *pb = part + kLzBlocks, *sc = part + 2 * kLzBlocks;
    std::vector<double> al, be;
    try {
        std::vector<double> h(n3, 0.0), act(c->nact);
        std::vector<int> ai(c->nact);
        MOT_CUDA_TRY(cudaMemcpyAsync(ai.data(), c->active, sizeof(int) * c->nact,
                                     cudaMemcpyDeviceToHost, c->stream));
        MOT_CUDA_TRY(cudaStreamSynchronize(c->stream));
        unsigned long long st = 240703323ULL;
        double nrm = 0.0;
        for (long long i = 0; i < c->nact; ++i)
            for (int k = 0; k < 3; ++k) {
                st = st * 6364136223846793005ULL + 1442695040888963407ULL;
                const double r = (double)(st >> 11) / 9007199254740992.0 - 0.5;
                h[k * c->M + ai[i]] = r;
                nrm += r * r;
            }
        nrm = std::sqrt(nrm);
        for (double& x : h) x /= nrm;
        upload(v1, h.data(), n3, c->stream);
        clear(v0, n3, c->stream);
        CGArgs a{};
        a.M = c->M; a.act = c->active; a.nmask = c->nmask; a.nact = c->nact; a.diag = c->cg_diag;
        for (int e = 0; e < 27; ++e) a.noff[e] = c->noff[e];
        for (int j = 0; j < kSteps; ++j) {
            MOT_CUDA_TRY(cudaMemsetAsync(w, 0, sizeof(double) * n3, c->stream));
            k_apply64<<<(int)((c->nact + NT - 1) / NT), NT, 0, c->stream>>>(a, v1, w);
            MOT_LAUNCH_CHECK();
            k_lz_dot<<<kLzBlocks, NT, 0, c->stream>>>(w, v1, n3, pa);
            MOT_LAUNCH_CHECK();
            k_lz_step<<<kLzBlocks, NT, 0, c->stream>>>(w, v1, v0, pa, j ? sc + 2 * j - 1 : nullptr,
                                                       n3, sc + 2 * j, pb);
            MOT_LAUNCH_CHECK();
            k_lz_scale<<<kLzBlocks, NT, 0, c->stream>>>(w, pb, n3, sc + 2 * j + 1);
            MOT_LAUNCH_CHECK();
            std::swap(v0, v1);
            std::swap(v1, w);
        }
        std::vector<double> hs(2 * kSteps);
        MOT_CUDA_TRY(cudaMemcpyAsync(hs.data(), sc, sizeof(double) * 2 * kSteps,
                                     cudaMemcpyDeviceToHost, c->stream));
        MOT_CUDA_TRY(cudaStreamSynchronize(c->stream));
        double beta = 0.0;
        for (int j = 0; j < kSteps; ++j) {
            al.push_back(hs[2 * j]);
            be.push_back(beta);
            beta = std::sqrt(std::max(hs[2 * j + 1], 0.0));
            if (!(beta > 1e-14)) break;      // invariant: the steps after it are dropped
        }
    } catch (...) {
        cudaFree(v0); cudaFree(v1); cudaFree(w); cudaFree(part);
        throw;
    }
    cudaFree(v0); cudaFree(v1); cudaFree(w); cudaFree(part);
    double lo = 1e300, hi = -1e300;
    for (size_t i = 0; i < al.size(); ++i) {
        const double r = std::fabs(al[i]) + (i ? std::fabs(be[i]) : 0.0) +
                         (i + 1 < al.size() ? std::fabs(be[i + 1]) : 0.0);
        lo = std::min(lo, al[i] - r);
        hi = std::max(hi, al[i] + r);
    }
    const int k = (int)al.size();
    const double tmin = tridiag_eig(al, be, 0, lo, hi);
    const double tmax = tridiag_eig(al, be, k - 1, lo, hi);
    // tmax == tmin when A is a multiple of the identity (a single voxel: G_0(0) is
    // isotropic); the interval [tmin, 1.02 tmax] below is still non-empty
    if (!(tmin > 0.0) || !(tmax >= tmin))
        throw MotError{MOT_ERR_ARG, "diag(1/chi) Z_0 is not positive definite on this grid"};
    const double A = tmin, B = 1.02 * tmax;
    c->cheb_lmin = A;
    c->cheb_lmax = B;
    const double theta = 0.5 * (B + A), delta = 0.5 * (B - A), sigma = theta / delta;
    const double kap = B / A;
    const double rate = (std::sqrt(kap) - 1.0) / (std::sqrt(kap) + 1.0);
    int nk = (int)std::ceil(std::log(0.5 * kFloor) / std::log(rate));
    nk = std::max(4, std::min(nk, MAXCHEB));
    c->cheb_n = nk;
    c->cheb_log_rate = std::log(rate);
    c->cheb_inv_theta = (float)(1.0 / theta);
    double rho = 1.0 / sigma;
    for (int i = 0; i < nk; ++i) {
        const double rn = 1.0 / (2.0 * sigma - rho);
        c->cheb_c1[i] = (float)(rn * rho);
        c->cheb_c2[i] = (float)(2.0 * rn / delta);
        rho = rn;
    }
}

namespace {

int fit_slot(int n) { return n % kSlots; }

// pairs (x, b) of the steps before the one being launched
int fit_pairs(const mot_ctx* c) { return std::min(c->fit_steps, kFit); }

double* norm_shares(const mot_ctx* c, int parity) { return c->norm_part + (long long)parity * c->norm_blocks; }

EpiArgs make_epi_args(mot_ctx* c, int n, const double* En, double* out, bool adj) {
    EpiArgs a;
    a.out = out;
    a.M = c->M;
    a.f = c->vfac;
    a.En = En;
    a.hist = c->precision == MOT_FP64 ? (const void*)c->h64.hist_spatial : (const void*)c->h32.hist_spatial;
    a.Jring = c->J;
    a.s0 = (int)slot_index(n, c->jring);
    a.jring = c->jring;
    a.tp = taps_of(c);
    a.n = n;
    a.bs = fit_slot(n);
    a.nv = fit_pairs(c);
    a.b64 = c->b_ring;
    a.xb = reinterpret_cast<float2*>(c->xb_ring);
    a.bl = c->b_lo;
    a.x0 = reinterpret_cast<float4*>(c->cg_xl);
    a.rhs = c->rhs;
    a.fit = reinterpret_cast<const FitState*>(c->fit);
    a.part = c->fit_part;
    a.nrm = norm_shares(c, (c->solve_seq + 1) & 1) + c->cg_blocks;
    a.adj = adj;
    return a;
}

template <typename R, bool ADJ>
void epilogue(mot_ctx* c, const EpiArgs& a, cudaStream_t s) {
    launch_dependent(mot::dependent_launches(c), k_epilogue<R, ADJ>, c->epi_blocks, NT, 0, s, a);
    MOT_LAUNCH_CHECK();
}

}  // namespace

namespace {

CGArgs make_cg_args(mot_ctx* c, int n, double* norm2_out, double* out) {
    CGArgs a;
    a.out = out;
    a.M = c->M;
    for (int e = 0; e < 27; ++e) a.noff[e] = c->noff[e];
    a.act = c->active;
    a.nmask = c->nmask;
    a.nact = c->nact;
    a.U = c->U; a.V = c->V; a.W = c->W;
    a.tiles = c->tiles;
    a.ntiles = c->ntiles;
    a.halo = c->halo;
    a.nw = c->cg_blocks;
    a.x = c->J + slot_index(n, c->jring) * 3 * c->M;
    a.bs = fit_slot(n);
    a.nv = fit_pairs(c);
    a.b = c->b_ring ? c->b_ring + (long long)a.bs * 3 * c->M : nullptr;
    a.xb = c->xb_ring ? reinterpret_cast<float2*>(c->xb_ring) + (long long)a.bs * 3 * c->M : nullptr;
    a.bl = c->b_lo;
    a.diag32 = c->diag32;
    a.diag = c->cg_diag;
    a.diag_lo = c->diag_lo;
    a.r = reinterpret_cast<float4*>(c->cg32);
    a.p = a.r + c->M;
    a.q = a.r + 2 * c->M;
    a.e = a.r + 3 * c->M;
    a.xl = c->cg_xl ? reinterpret_cast<float4*>(c->cg_xl) : nullptr;
    a.red = c->red;
    a.red4 = reinterpret_cast<float4*>(c->red + 2LL * c->cg_blocks);
    a.tol = (float)c->tol;
    a.inv_theta = c->cheb_inv_theta;
    a.n_cheb = c->cheb_n;
    a.inv_log2_rate = (float)(std::log(2.0) / c->cheb_log_rate);
    for (int k = 0; k < MAXCHEB; ++k) {
        a.c1[k] = k < c->cheb_n ? c->cheb_c1[k] : 0.f;
        a.c2[k] = k < c->cheb_n ? c->cheb_c2[k] : 0.f;
    }
    a.max_iter = c->max_iter;
    a.max_outer = 12;
    a.step = n;
    a.status = c->dstatus;
    a.bar = reinterpret_cast<unsigned*>(c->dstatus + 4);
    a.bar_budget = c->bar_budget;
    a.fit = reinterpret_cast<FitState*>(c->fit);
    a.part = c->fit_part;
    a.nepi = c->epi_blocks;
    a.part4 = reinterpret_cast<float4*>(c->fit_part);
    // every active voxel's words in p and q are rewritten by each launch, so numbers that
    // only have to differ from those of the launch before may wrap
    a.seq = ++c->solve_seq * 1024u;
    a.parity = (int)(c->solve_seq & 1u);
    a.nrm = norm_shares(c, a.parity);
    a.nrm_prev = norm_shares(c, a.parity ^ 1);
    a.norm_prev = c->norm_pending;
    a.prev_step = c->norm_step;
    a.nred = c->norm_blocks;
    a.vac = c->vac;
    a.nvac = (int)c->nvac;
    a.nvb = c->cg_resident ? c->norm_blocks - c->cg_blocks : 0;
    c->norm_pending = norm2_out;
    c->norm_step = n;
    return a;
}

// kernel variant of a context's solve and its block size
struct SolveKernel { void* fn; int threads; };
template <class T> SolveKernel kernel_of(bool df, bool split) {
    if (df) return {(void*)k_cg<true, T, true, false>, T::NTH};
    if (split) return {(void*)k_cg<false, T, true, true>, T::NTH};
    return {(void*)k_cg<false, T, true, false>, T::NTH};
}
// tile 1, 2 or 4 (voxels per thread); vectors in memory only with tile 4
SolveKernel solve_kernel(int precision, int tile, bool resident, bool split) {
    const bool df = precision != MOT_FP64;
    if (!resident)
        return {df ? (void*)k_cg<true, TileMem, false, false>
                   : (void*)k_cg<false, TileMem, false, false>, TileMem::NTH};
    return tile == 1 ? kernel_of<Tile1>(df, split)
           : tile == 2 ? kernel_of<Tile2>(df, split) : kernel_of<Tile4>(df, split);
}

// Right-hand side, start and solve of step n: one kernel where the tiles are resident, the
// epilogue before it where not (a grid of that size hides a launch: 1.6 ms a step at 104^3).
void launch_solve(mot_ctx* c, int n, const double* En, double* norm2_out, double* out, bool adj,
                  cudaStream_t s) {
    EpiArgs ep = make_epi_args(c, n, En, out, adj);
    if (!c->cg_resident) {
        if (c->precision == MOT_FP64) adj ? epilogue<double, true>(c, ep, s) : epilogue<double, false>(c, ep, s);
        else adj ? epilogue<float, true>(c, ep, s) : epilogue<float, false>(c, ep, s);
        c->stats.launches += 1;
    }
    CGArgs a = make_cg_args(c, n, norm2_out, out);
    void* args[] = {&a, &ep};
    const SolveKernel k = solve_kernel(c->precision, c->cg_tile, c->cg_resident, c->cg_split);
    MOT_CUDA_TRY(cudaLaunchCooperativeKernel(k.fn, c->cg_blocks + 1 + a.nvb, k.threads, args, 0, s));
    ++c->fit_steps;
    c->stats.launches += 1;
}

}  // namespace

// adds up the norm of the last step launched
void solve_finish(mot_ctx* c, cudaStream_t s) {
    if (!c->norm_pending) return;
    k_norm_total<<<1, 32, 0, s>>>(norm_shares(c, (int)(c->solve_seq & 1u)), c->norm_blocks,
                                  c->norm_pending, c->dstatus, c->norm_step);
    MOT_LAUNCH_CHECK();
    c->norm_pending = nullptr;
}

// Shape of the solve on this geometry.  tiles[i]: active tiles of 8 x 4 x 4, 8 x 4 x 8 and
// 8 x 8 x 8 voxels; sets the tile, the worker blocks and the epilogue's launch, and returns
// the chosen list.
const std::vector<int>& solve_shape(mot_ctx* c, const std::vector<int> (&tiles)[3]) {
    // FP64 residual by components while the voxels' warps are fewer than the GPU's
    // sub-partitions (an FP64 chain of one voxel is 170 instructions of 64 cycles each)
    c->cg_split = c->precision == MOT_FP64 && c->nact <= 128LL * c->nsm;
    int pick = 2, per_sm = 0;
    c->cg_resident = false;
    for (int i = 0; i < 3 && !c->cg_resident; ++i) {
        const SolveKernel k = solve_kernel(c->precision, 1 << i, true, c->cg_split);
        MOT_CUDA_TRY(cudaOccupancyMaxActiveBlocksPerMultiprocessor(&per_sm, k.fn, k.threads, 0));
        if ((long long)tiles[i].size() + 2 <= (long long)per_sm * c->nsm) {
            c->cg_resident = true;
            pick = i;
        }
    }
    if (!c->cg_resident) {
        c->cg_split = false;
        const SolveKernel k = solve_kernel(c->precision, 4, false, false);
        MOT_CUDA_TRY(cudaOccupancyMaxActiveBlocksPerMultiprocessor(&per_sm, k.fn, k.threads, 0));
    }
    if (per_sm < 1) throw MotError{MOT_ERR_CUDA, "CG kernel cannot be made resident"};
    c->cg_tile = 1 << pick;
    c->ntiles = (int)tiles[pick].size();
    // one block per tile at most: the tiled passes give a block one tile at a time, so
    // further blocks would only wait (and keep SMs from concurrent solves of other
    // contexts).  The component-split FP64 residual has work for more: a block for every
    // four warps of it, up to two per SM.
    int want = std::max(c->ntiles, 1);
    if (c->cg_split)
        want = std::max(want, std::min(2 * c->nsm, (int)(3 * ((c->nact + 31) / 32) + 3) / 4));
    c->cg_blocks = std::max(1, std::min(per_sm * c->nsm - 2, want));
    c->epi_blocks = (int)std::min<long long>((c->M + NT - 1) / NT, 8LL * c->nsm);
    // blocks with a share of the norm: the solve's, then the epilogue's or (resident) those
    // that take the voxels outside the tiles
    static const int dims[3][3] = {{8, 4, 4}, {8, 4, 8}, {8, 8, 8}};
    c->nvac = c->M;
    for (int o : tiles[pick])
        c->nvac -= (long long)std::min(dims[pick][0], c->U - (o & 1023)) *
                   std::min(dims[pick][1], c->V - ((o >> 10) & 1023)) *
                   std::min(dims[pick][2], c->W - (o >> 20));
    const int room = per_sm * c->nsm - 1 - c->cg_blocks;
    c->norm_blocks = c->cg_blocks +
                     (c->cg_resident ? (int)std::min<long long>(room, (c->nvac + 127) / 128)
                                     : c->epi_blocks);
    return tiles[pick];
}

namespace {
template <class T> void halo_lists(mot_ctx* c) {
    typedef Resident<T> RT;
    MOT_CUDA_TRY(cudaMalloc(&c->halo, sizeof(int) * RT::HPT * T::NTH * (size_t)c->ntiles));
    k_halo_list<T><<<c->ntiles, T::NTH, 0, c->stream>>>(c->tiles, c->diag32, c->U, c->V, c->W,
                                                        c->halo);
    MOT_LAUNCH_CHECK();
}
}  // namespace

// halo lists of the resident tiles (tiles and diag32 on the device)
void solve_halo_lists(mot_ctx* c) {
    if (!c->cg_resident || !c->ntiles) return;
    if (c->cg_tile == 1) halo_lists<Tile1>(c);
    else if (c->cg_tile == 2) halo_lists<Tile2>(c);
    else halo_lists<Tile4>(c);
}

// right-hand side and solve of step n; ||J_n||^2 into norm2_out (device; by the next step or
// solve_finish), J_n in ring slot n and (AoS) in out
void solve_step(mot_ctx* c, int n, const double* En, double* norm2_out, double* out,
                cudaStream_t s) {
    launch_solve(c, n, En, norm2_out, out, false, s);
}

void read_aos(mot_ctx* c, const double* in_dev, double* slot, cudaStream_t s) {
    const long long tot = 3 * c->M;
    k_from_aos<<<(int)((tot + NT - 1) / NT), NT, 0, s>>>(in_dev, c->M, slot);
    MOT_LAUNCH_CHECK();
}

void history_out(mot_ctx* c, int n, double* out_dev, cudaStream_t s) {
    const long long tot = 3 * c->M;
    if (c->precision == MOT_FP64)
        k_history_out<double><<<(int)((tot + NT - 1) / NT), NT, 0, s>>>(
            c->M, c->eps, c->chi, c->h64.hist_spatial, c->J, (int)slot_index(n, c->jring), c->jring,
            taps_of(c), out_dev);
    else
        k_history_out<float><<<(int)((tot + NT - 1) / NT), NT, 0, s>>>(
            c->M, c->eps, c->chi, c->h32.hist_spatial, c->J, (int)slot_index(n, c->jring), c->jring,
            taps_of(c), out_dev);
    MOT_LAUNCH_CHECK();
}

// one adjoint step: tau = adjoint time (ring index), n = N + 1 - tau (forward time)
void adjoint_step(mot_ctx* c, int tau, int n, const double* g_aos, const double* J_aos,
                  int j_first, double* grad_chi, double* lam_out, double* norm2_out,
                  cudaStream_t s) {
    const int s0 = (int)slot_index(tau, c->jring);
    launch_solve(c, tau, g_aos, norm2_out, nullptr, true, s);
    double* mu = c->J + (long long)s0 * 3 * c->M;
    k_adj_vacuum<<<(int)((c->M + NT - 1) / NT), NT, 0, s>>>(c->M, c->U, c->V, c->W, c->vfac, mu,
                                                           c->rhs, c->cg_q);
    MOT_LAUNCH_CHECK();
    k_adj_post<<<(int)((c->M + NT - 1) / NT), NT, 0, s>>>(c->M, c->vfac, mu, c->cg_q, J_aos,
                                                         j_first, n, taps_of(c), grad_chi,
                                                         lam_out);
    MOT_LAUNCH_CHECK();
    c->stats.launches += 2;
}

}  // namespace mot

extern "C" mot_status mot_barrier_check(int n_blocks, int rounds, int absent, double budget_s,
                                        int* passed, int* timeout_round) {
    if (!passed || !timeout_round || rounds < 1 || rounds > (1 << 20) || absent < -1 ||
        absent >= n_blocks || !(budget_s > 0.0 && budget_s <= 10.0))
        return MOT_ERR_ARG;
    int dev = 0, nsm = 0, per_sm = 0, khz = 0;
    if (cudaGetDevice(&dev) != cudaSuccess ||
        cudaDeviceGetAttribute(&nsm, cudaDevAttrMultiProcessorCount, dev) != cudaSuccess ||
        cudaDeviceGetAttribute(&khz, cudaDevAttrClockRate, dev) != cudaSuccess ||
        cudaOccupancyMaxActiveBlocksPerMultiprocessor(&per_sm, k_barrier_check, NT, 0) !=
            cudaSuccess) {
        cudaGetLastError();
        return MOT_ERR_CUDA;
    }
    if (n_blocks < 1 || n_blocks > per_sm * nsm) return MOT_ERR_ARG;   // must be co-resident
    int* w = nullptr;
    if (cudaMalloc(&w, sizeof(int) * 9) != cudaSuccess) {
        cudaGetLastError();
        return MOT_ERR_OOM;
    }
    long long budget = (long long)(budget_s * 1e3 * std::max(khz, 1000000));
    void* args[] = {&w, &budget, &rounds, &absent};
    int h[9] = {0};
    cudaError_t e = cudaMemset(w, 0, sizeof(int) * 9);
    if (e == cudaSuccess)
        e = cudaLaunchCooperativeKernel((void*)k_barrier_check, n_blocks, NT, args, 0, nullptr);
    if (e == cudaSuccess) e = cudaMemcpy(h, w, sizeof h, cudaMemcpyDeviceToHost);
    cudaFree(w);
    if (e != cudaSuccess) {
        cudaGetLastError();
        return MOT_ERR_CUDA;
    }
    *passed = h[8];
    *timeout_round = h[2];
    return (h[1] & 4) ? MOT_ERR_TIMEOUT : MOT_OK;
}
