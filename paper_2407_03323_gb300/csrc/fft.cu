// Zero-padded 3D FFTs of the current densities and of the history spectrum
// (Sec. 3, Eq. PnFFTMOT; App. A: a Toeplitz product becomes a circulant one after
// zero-padding to P >= n_row + n_col - 1 per axis).
//
// Layouts (per component, 3 components stacked):
//   spatial   [W][V][U]        u fastest (m = u + U (v + V w), Sec. 2.2)
//   after x   [W][V][Hu]       Hu = Pu/2 + 1 (real-to-complex along u)
//   after y   [W][Pv][Hu]
//   spectrum  [Pw][Pv][Hu]
// Forward: three passes x (r2c of paired real rows), y, z; every pass reads only the
// nonzero (unpadded) inputs.  Inverse: z, y, x (c2r), storing only the N outputs the
// grid needs.  Each pass runs batched length-P transforms in shared memory: a CTA
// holds a tile of TB lines as buf[j * (TB+1) + t] and runs mixed-radix Stockham
// stages (radices 2, 3, 4, 5, 7) over it.  Twiddles come from a table of
// exp(-2 pi i k / P) built once per axis with sincospi.  No normalisation is applied.
#include "mot_internal.cuh"

#include <algorithm>

#include "fft_core.cuh"

using namespace mot_fft;

namespace {

constexpr int NT = 256;
constexpr int kLoadBatch = 8;   // global loads a thread keeps in flight while staging a tile

// lines per CTA: 8 (FP64) / 16 (FP32) keeps the shared tile near 60 KB at P = 210,
// so that several CTAs are resident per SM
template <typename R> struct Tile { static constexpr int TB = 8; };
template <> struct Tile<float> { static constexpr int TB = 16; };

// ------------------------------------------------------------------ pass x, forward
// rows (comp, w, v) of a real [3][W][V][U] array, paired (v, v+1) -> [3][W][V][Hu]
template <typename R>
__global__ void __launch_bounds__(NT) k_fwd_x(const double* __restrict__ in, int U, int V, int W,
                                              typename CT<R>::c* __restrict__ out,
                                              const typename CT<R>::c* __restrict__ tw,
                                              RadixList rl, const double* __restrict__ scale) {
    typedef typename CT<R>::c C;
    constexpr int TB = Tile<R>::TB;
    constexpr int ld = TB + 1;
    extern __shared__ __align__(16) unsigned char smem_raw[];
    C* stw = reinterpret_cast<C*>(smem_raw);
    C* b0 = stw + tw_entries<C>(rl.P);
    C* b1 = b0 + rl.P * ld;
    const int P = rl.P, Hu = P / 2 + 1;
    const int VP = (V + 1) / 2;
    const long long npairs = 3LL * W * VP;
    const long long pair0 = (long long)blockIdx.x * TB;
    load_tw(stw, tw, P);
    pdl_trigger();
    pdl_wait();
    // load: z = a + i b, zero-padded; batches of kLoadBatch loads in flight per thread
    for (int it0 = threadIdx.x; it0 < TB * P; it0 += kLoadBatch * blockDim.x) {
        double va[kLoadBatch], vb[kLoadBatch];
#pragma unroll
        for (int q = 0; q < kLoadBatch; ++q) {
            const int it = it0 + q * blockDim.x;
            const int t = it / P, j = it % P;
            const long long pr = pair0 + t;
            va[q] = 0.0;
            vb[q] = 0.0;
            if (it < TB * P && pr < npairs && j < U) {
                const long long cw = pr / VP;
                const int v = (int)(pr % VP) * 2;
                const double* row = in + (cw * V + v) * (long long)U;
                va[q] = row[j];
                if (v + 1 < V) vb[q] = row[U + j];
                if (scale) {   // per-voxel factor (the adjoint transforms chi * lambda)
                    const long long m0 = ((cw % W) * V + v) * (long long)U + j;
                    va[q] *= scale[m0];
                    if (v + 1 < V) vb[q] *= scale[m0 + U];
                }
            }
        }
#pragma unroll
        for (int q = 0; q < kLoadBatch; ++q) {
            const int it = it0 + q * blockDim.x;
            if (it >= TB * P) break;
            const int t = it / P, j = it % P;
            C z;
            z.x = (R)va[q];
            z.y = (R)vb[q];
            b0[j * ld + t] = z;
        }
    }
    __syncthreads();
    C* res = fft_tile<C, TB>(b0, b1, P, rl.r, rl.n, ld, stw, -1);
    // split: A = (Z[k] + conj Z[P-k]) / 2, B = -i (Z[k] - conj Z[P-k]) / 2
    for (int it = threadIdx.x; it < TB * Hu; it += blockDim.x) {
        const int t = it / Hu, k = it % Hu;
        const long long pr = pair0 + t;
        if (pr >= npairs) continue;
        const long long cw = pr / VP;
        const int v = (int)(pr % VP) * 2;
        const C zk = res[k * ld + t];
        const C zm = res[((P - k) % P) * ld + t];
        C A, B;
        A.x = (R)0.5 * (zk.x + zm.x);
        A.y = (R)0.5 * (zk.y - zm.y);
        B.x = (R)0.5 * (zk.y + zm.y);
        B.y = (R)0.5 * (zm.x - zk.x);
        out[(cw * V + v) * (long long)Hu + k] = A;
        if (v + 1 < V) out[(cw * V + v + 1) * (long long)Hu + k] = B;
    }
}

// ------------------------------------------------------------------ pass x, inverse
// [3][W][V][Hu] Hermitian halves -> real rows [3][W][V][U] (first U outputs)
template <typename R>
__global__ void __launch_bounds__(NT) k_inv_x(const typename CT<R>::c* __restrict__ in, int U,
                                              int V, int W, R* __restrict__ out,
                                              const typename CT<R>::c* __restrict__ tw,
                                              RadixList rl) {
    typedef typename CT<R>::c C;
    constexpr int TB = Tile<R>::TB;
    constexpr int ld = TB + 1;
    extern __shared__ __align__(16) unsigned char smem_raw[];
    C* stw = reinterpret_cast<C*>(smem_raw);
    C* b0 = stw + tw_entries<C>(rl.P);
    C* b1 = b0 + rl.P * ld;
    const int P = rl.P, Hu = P / 2 + 1;
    const int VP = (V + 1) / 2;
    const long long npairs = 3LL * W * VP;
    const long long pair0 = (long long)blockIdx.x * TB;
    load_tw(stw, tw, P);
    pdl_trigger();
    pdl_wait();
    for (int it0 = threadIdx.x; it0 < TB * Hu; it0 += kLoadBatch * blockDim.x) {
        C Aq[kLoadBatch], Bq[kLoadBatch];
#pragma unroll
        for (int q = 0; q < kLoadBatch; ++q) {
            const int it = it0 + q * blockDim.x;
            const int t = it / Hu, k = it % Hu;
            const long long pr = pair0 + t;
            Aq[q].x = 0; Aq[q].y = 0; Bq[q].x = 0; Bq[q].y = 0;
            if (it < TB * Hu && pr < npairs) {
                const long long cw = pr / VP;
                const int v = (int)(pr % VP) * 2;
                Aq[q] = in[(cw * V + v) * (long long)Hu + k];
                if (v + 1 < V) Bq[q] = in[(cw * V + v + 1) * (long long)Hu + k];
            }
        }
#pragma unroll
        for (int q = 0; q < kLoadBatch; ++q) {
            const int it = it0 + q * blockDim.x;
            if (it >= TB * Hu) break;
            const int t = it / Hu, k = it % Hu;
            const C A = Aq[q], B = Bq[q];
            C z;
            z.x = A.x - B.y;
            z.y = A.y + B.x;
            b0[k * ld + t] = z;
            if (k >= 1 && k < P - k) {
                C zm;
                zm.x = A.x + B.y;
                zm.y = B.x - A.y;
                b0[(P - k) * ld + t] = zm;
            }
        }
    }
    __syncthreads();
    C* res = fft_tile<C, TB>(b0, b1, P, rl.r, rl.n, ld, stw, +1);
    for (int it = threadIdx.x; it < TB * U; it += blockDim.x) {
        const int t = it / U, j = it % U;
        const long long pr = pair0 + t;
        if (pr >= npairs) continue;
        const long long cw = pr / VP;
        const int v = (int)(pr % VP) * 2;
        const C z = res[j * ld + t];
        out[(cw * V + v) * (long long)U + j] = z.x;
        if (v + 1 < V) out[(cw * V + v + 1) * (long long)U + j] = z.y;
    }
}

// ------------------------------------------------------------------ pass x, four-step codelets
// For P = P1 P2 (64 = 8 x 8, 96 = 8 x 12, 210 = 14 x 15): 32 row pairs per CTA, each
// pair a complex line of P points in shared memory ([P][33], line fastest).  Phase A
// (warp n1 < P1, lane = line): x[n1 + P1 n2] -> DFT of length P2 over n2 in registers
// (compile-time radices and twiddles, dft_ct) -> times W_P^{n1 k2}; phase B (warp
// k2 < P2): DFT of length P1 over n1 -> X[k2 + P2 k1].  Every phase first reads its
// values into registers, then (after a barrier) writes them back into the same buffer.
constexpr int kXL = 32;          // row pairs per CTA
constexpr int kXLD = kXL + 1;    // padded line stride of the shared buffer

template <typename C, int P1, int P2, int DIR>
__device__ __forceinline__ void x_four_step(C* X, const C* stw, int nvalid) {
    constexpr int P = P1 * P2;
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    C x[P2];
    if (warp < P1) {
        const int n1 = warp;
        Unroll1<0, P2>::run([&](auto q) {
            constexpr int n2 = decltype(q)::value;
            const int idx = n1 + P1 * n2;
            C v;
            v.x = 0; v.y = 0;
            if (idx < nvalid) v = X[idx * kXLD + lane];
            x[n2] = v;
        });
        dft_ct<P2, DIR>(x);
        Unroll1<0, P2>::run([&](auto q) {
            constexpr int k2 = decltype(q)::value;
            x[k2] = twmul_tab(stw, (n1 * k2) % P, P, DIR, x[k2]);
        });
    }
    __syncthreads();
    if (warp < P1)
        Unroll1<0, P2>::run([&](auto q) {
            constexpr int k2 = decltype(q)::value;
            X[(warp * P2 + k2) * kXLD + lane] = x[k2];
        });
    __syncthreads();
    C y[P1];
    if (warp < P2) {
        Unroll1<0, P1>::run([&](auto q) {
            constexpr int n1 = decltype(q)::value;
            y[n1] = X[(n1 * P2 + warp) * kXLD + lane];
        });
        dft_ct<P1, DIR>(y);
    }
    __syncthreads();
    if (warp < P2)
        Unroll1<0, P1>::run([&](auto q) {
            constexpr int k1 = decltype(q)::value;
            X[(warp + P2 * k1) * kXLD + lane] = y[k1];
        });
    __syncthreads();
}

template <typename R, int P1, int P2>
__global__ void k_fwd_x4s(const double* __restrict__ in, int U, int V, int W,
                          typename CT<R>::c* __restrict__ out,
                          const typename CT<R>::c* __restrict__ tw,
                          const double* __restrict__ scale) {
    typedef typename CT<R>::c C;
    constexpr int P = P1 * P2, Hu = P / 2 + 1;
    extern __shared__ __align__(16) unsigned char smem_raw[];
    C* X = reinterpret_cast<C*>(smem_raw);          // [P][kXLD]
    C* stw = X + P * kXLD;                          // [tw_entries(P)]
    const int VP = (V + 1) / 2;
    const long long npairs = 3LL * W * VP;
    const long long pair0 = (long long)blockIdx.x * kXL;
    for (int i = threadIdx.x; i < tw_entries<C>(P); i += blockDim.x) stw[i] = tw[i];
    pdl_trigger();
    pdl_wait();
    // z = a + i b of the two rows of a pair; positions >= U are the zero padding
    for (int it = threadIdx.x; it < kXL * U; it += blockDim.x) {
        const int t = it / U, j = it % U;
        const long long pr = pair0 + t;
        double va = 0.0, vb = 0.0;
        if (pr < npairs) {
            const long long cw = pr / VP;
            const int v = (int)(pr % VP) * 2;
            const double* row = in + (cw * V + v) * (long long)U;
            va = row[j];
            if (v + 1 < V) vb = row[U + j];
            if (scale) {   // per-voxel factor (the adjoint transforms chi * lambda)
                const long long m0 = ((cw % W) * V + v) * (long long)U + j;
                va *= scale[m0];
                if (v + 1 < V) vb *= scale[m0 + U];
            }
        }
        C z;
        z.x = (R)va;
        z.y = (R)vb;
        X[j * kXLD + t] = z;
    }
    __syncthreads();
    x_four_step<C, P1, P2, -1>(X, stw, U);
    // split: A = (Z[k] + conj Z[P-k]) / 2, B = -i (Z[k] - conj Z[P-k]) / 2
    for (int it = threadIdx.x; it < kXL * Hu; it += blockDim.x) {
        const int t = it / Hu, k = it % Hu;
        const long long pr = pair0 + t;
        if (pr >= npairs) continue;
        const long long cw = pr / VP;
        const int v = (int)(pr % VP) * 2;
        const C zk = X[k * kXLD + t];
        const C zm = X[((P - k) % P) * kXLD + t];
        C A, B;
        A.x = (R)0.5 * (zk.x + zm.x);
        A.y = (R)0.5 * (zk.y - zm.y);
        B.x = (R)0.5 * (zk.y + zm.y);
        B.y = (R)0.5 * (zm.x - zk.x);
        out[(cw * V + v) * (long long)Hu + k] = A;
        if (v + 1 < V) out[(cw * V + v + 1) * (long long)Hu + k] = B;
    }
}

template <typename R, int P1, int P2>
__global__ void k_inv_x4s(const typename CT<R>::c* __restrict__ in, int U, int V, int W,
                          R* __restrict__ out, const typename CT<R>::c* __restrict__ tw) {
    typedef typename CT<R>::c C;
    constexpr int P = P1 * P2, Hu = P / 2 + 1;
    extern __shared__ __align__(16) unsigned char smem_raw[];
    C* X = reinterpret_cast<C*>(smem_raw);
    C* stw = X + P * kXLD;
    const int VP = (V + 1) / 2;
    const long long npairs = 3LL * W * VP;
    const long long pair0 = (long long)blockIdx.x * kXL;
    for (int i = threadIdx.x; i < tw_entries<C>(P); i += blockDim.x) stw[i] = tw[i];
    pdl_trigger();
    pdl_wait();
    // Z[k] = A[k] + i B[k] and Z[P-k] = conj A[k] + i conj B[k] from the two halves
    for (int it = threadIdx.x; it < kXL * Hu; it += blockDim.x) {
        const int t = it / Hu, k = it % Hu;
        const long long pr = pair0 + t;
        C A, B;
        A.x = 0; A.y = 0; B.x = 0; B.y = 0;
        if (pr < npairs) {
            const long long cw = pr / VP;
            const int v = (int)(pr % VP) * 2;
            A = in[(cw * V + v) * (long long)Hu + k];
            if (v + 1 < V) B = in[(cw * V + v + 1) * (long long)Hu + k];
        }
        C z;
        z.x = A.x - B.y;
        z.y = A.y + B.x;
        X[k * kXLD + t] = z;
        if (k >= 1 && k < P - k) {
            C zm;
            zm.x = A.x + B.y;
            zm.y = B.x - A.y;
            X[(P - k) * kXLD + t] = zm;
        }
    }
    __syncthreads();
    x_four_step<C, P1, P2, +1>(X, stw, P);
    for (int it = threadIdx.x; it < kXL * U; it += blockDim.x) {
        const int t = it / U, j = it % U;
        const long long pr = pair0 + t;
        if (pr >= npairs) continue;
        const long long cw = pr / VP;
        const int v = (int)(pr % VP) * 2;
        const C z = X[j * kXLD + t];
        out[(cw * V + v) * (long long)U + j] = z.x;
        if (v + 1 < V) out[(cw * V + v + 1) * (long long)U + j] = z.y;
    }
}

// ------------------------------------------------------------------ strided passes
struct MidArgs {
    int n_in, n_out;          // inputs read / outputs stored along the axis
    int n_o2;                 // outer index o = comp * n_o2 + o2
    long long in_c, in_o, in_a;    // strides: component, outer, axis (in elements)
    long long out_c, out_o, out_a;
    int Hu;                   // contiguous extent
    int dir;
};

// Line L of a strided pass: its element offsets in the input and output; false past the
// last line.  Lines are numbered through (component, outer, ku), and a CTA takes
// consecutive ones: runs cut at each row of Hu = P/2 + 1 would leave much of the last run
// of every row idle (Hu = 33: 1 of 32 lines).
__device__ __forceinline__ bool mid_line(const MidArgs& a, long long L, long long& src,
                                         long long& dst) {
    const long long o = L / a.Hu;
    const int ku = (int)(L - o * a.Hu);
    const int comp = (int)(o / a.n_o2), o2 = (int)(o - (long long)comp * a.n_o2);
    const bool live = comp < 3;
    src = live ? comp * a.in_c + o2 * a.in_o + ku : 0;
    dst = live ? comp * a.out_c + o2 * a.out_o + ku : 0;
    return live;
}

template <typename R>
__global__ void __launch_bounds__(NT) k_mid(const typename CT<R>::c* __restrict__ in,
                                            typename CT<R>::c* __restrict__ out,
                                            const typename CT<R>::c* __restrict__ tw,
                                            RadixList rl, MidArgs a) {
    typedef typename CT<R>::c C;
    constexpr int TB = Tile<R>::TB;
    constexpr int ld = TB + 1;
    extern __shared__ __align__(16) unsigned char smem_raw[];
    C* stw = reinterpret_cast<C*>(smem_raw);
    C* b0 = stw + tw_entries<C>(rl.P);
    C* b1 = b0 + rl.P * ld;
    const int P = rl.P;
    // a thread's line t is the same in every round (blockDim is a multiple of TB)
    const int t = threadIdx.x % TB;
    long long src_off, dst_off;
    const bool live = mid_line(a, (long long)blockIdx.x * TB + t, src_off, dst_off);
    const C* src = in + src_off;
    C* dst = out + dst_off;
    load_tw(stw, tw, P);
    pdl_trigger();
    pdl_wait();
    for (int it = threadIdx.x; it < P * TB; it += blockDim.x) {
        const int j = it / TB;
        const bool ok = live && j < a.n_in;
        cp_async_c(&b0[j * ld + t], ok ? src + j * a.in_a : in, ok);
    }
    cp_async_commit_wait();
    __syncthreads();
    C* res = fft_tile<C, TB>(b0, b1, P, rl.r, rl.n, ld, stw, a.dir);
    if (!live) return;
    for (int j = threadIdx.x / TB; j < a.n_out; j += blockDim.x / TB)
        dst[j * a.out_a] = res[j * ld + t];
}

// ------------------------------------------------------------------ strided passes, four-step
// Length P = P1 P2 with both factors small: n = n1 + P1 n2, k = k2 + P2 k1,
//   X[k2 + P2 k1] = sum_{n1} W_P1^{n1 k1} (W_P^{n1 k2} sum_{n2} x[n1 + P1 n2] W_P2^{n2 k2}).
// A CTA holds 32 consecutive lines (lane = line, so every load and store is one
// coalesced run); phase A: warp n1 loads its P2 strided inputs (only the unpadded
// ones), runs the P2-point DFT in registers (compile-time structure and roots) and
// applies W_P^{n1 k2}; phase B: warp k2 gathers the P1 values over n1 from shared
// memory, runs the P1-point DFT and stores the outputs the pass needs.
template <typename R, int P1, int P2, int DIR>
__global__ void __launch_bounds__(32 * (P1 > P2 ? P1 : P2))
k_mid4s(const typename CT<R>::c* __restrict__ in, typename CT<R>::c* __restrict__ out,
        const typename CT<R>::c* __restrict__ tw, MidArgs a) {
    typedef typename CT<R>::c C;
    constexpr int P = P1 * P2, NL = 32;
    extern __shared__ __align__(16) unsigned char smem_raw[];
    C* Y = reinterpret_cast<C*>(smem_raw);          // [P1][P2][NL]
    C* stw = Y + P * NL;                            // roots exp(-2 pi i k / P) (tw_entries)
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    long long src_off, dst_off;
    const bool live = mid_line(a, (long long)blockIdx.x * NL + lane, src_off, dst_off);
    const C* src = in + src_off;
    C* dst = out + dst_off;
    for (int i = threadIdx.x; i < tw_entries<C>(P); i += blockDim.x) stw[i] = tw[i];
    pdl_trigger();
    pdl_wait();
    __syncthreads();
    if (warp < P1) {
        const int n1 = warp;
        C x[P2];
        Unroll1<0, P2>::run([&](auto q) {
            constexpr int n2 = decltype(q)::value;
            const int idx = n1 + P1 * n2;
            C v;
            v.x = 0; v.y = 0;
            if (idx < a.n_in && live) v = src[(long long)idx * a.in_a];
            x[n2] = v;
        });
        dft_ct<P2, DIR>(x);
        Unroll1<0, P2>::run([&](auto q) {
            constexpr int k2 = decltype(q)::value;
            Y[(n1 * P2 + k2) * NL + lane] = twmul_tab(stw, (n1 * k2) % P, P, DIR, x[k2]);
        });
    }
    __syncthreads();
    if (warp < P2) {
        const int k2 = warp;
        C y[P1];
        Unroll1<0, P1>::run([&](auto q) {
            constexpr int n1 = decltype(q)::value;
            y[n1] = Y[(n1 * P2 + k2) * NL + lane];
        });
        dft_ct<P1, DIR>(y);
        if (!live) return;
        Unroll1<0, P1>::run([&](auto q) {
            constexpr int k1 = decltype(q)::value;
            const int k = k2 + P2 * k1;
            if (k < a.n_out) dst[(long long)k * a.out_a] = y[k1];
        });
    }
}

// ------------------------------------------------------------------ x and y passes in one kernel
// A CTA takes one plane (component, w): the row pairs along u, then the Hu lines along v,
// both in shared memory, the Stockham stages of fft_core.cuh with the number of lines at run
// time.  On small grids the two passes of an axis each are all latency (launch, table, load,
// store, 6 to 7 us a pass whatever its length); larger planes have enough lines to fill the
// GPU with a launch of their own (see plane_pass).
template <typename C, int R, int DIR>
__device__ __forceinline__ void stage_lines(const C* __restrict__ x, C* __restrict__ y, int P,
                                            int Ns, int nl, int ld, const C* tw) {
    const int nb = P / R, items = nb * nl, tstep = P / (Ns * R);
    const float inv_nl = 1.0f / (float)nl, inv_ns = 1.0f / (float)Ns;
    for (int it = threadIdx.x; it < items; it += blockDim.x) {
        // exact for it, j < 2^20, as in stage()
        const int j = __float2int_rz(((float)it + 0.5f) * inv_nl), t = it - j * nl;
        const int jq = __float2int_rz(((float)j + 0.5f) * inv_ns), k = j - jq * Ns;
        C v[R];
#pragma unroll
        for (int r = 0; r < R; ++r) v[r] = x[(j + r * nb) * ld + t];
        if (Ns > 1) {
            const int kt = k * tstep;
#pragma unroll
            for (int r = 1; r < R; ++r) v[r] = twmul_tab(tw, r * kt, P, DIR, v[r]);
        }
        dft_small<C, R>(v, tw, P, DIR);
        const int base = jq * Ns * R + k;
#pragma unroll
        for (int r = 0; r < R; ++r) y[(base + r * Ns) * ld + t] = v[r];
    }
}
// transforms of nl lines x[j * ld + t]; returns the buffer that holds the result
template <typename C, int DIR>
__device__ __forceinline__ C* fft_lines(C* x, C* y, const RadixList& rl, int nl, int ld,
                                        const C* tw) {
    int Ns = 1;
    for (int s = 0; s < rl.n; ++s) {
        const int R = rl.r[s];
        switch (R) {
            case 2: stage_lines<C, 2, DIR>(x, y, rl.P, Ns, nl, ld, tw); break;
            case 3: stage_lines<C, 3, DIR>(x, y, rl.P, Ns, nl, ld, tw); break;
            case 4: stage_lines<C, 4, DIR>(x, y, rl.P, Ns, nl, ld, tw); break;
            case 5: stage_lines<C, 5, DIR>(x, y, rl.P, Ns, nl, ld, tw); break;
            case 7: stage_lines<C, 7, DIR>(x, y, rl.P, Ns, nl, ld, tw); break;
        }
        __syncthreads();
        Ns *= R;
        C* tmp = x; x = y; y = tmp;
    }
    return x;
}

constexpr int kPlaneThreads = 512;
constexpr size_t kPlaneSmem = 96 << 10;
// odd line strides: neither the transposed stores nor the line-fastest ones conflict
__host__ __device__ constexpr int plane_ldx(int V) { return ((V + 1) / 2) | 1; }
__host__ __device__ constexpr int plane_ldy(int Hu) { return Hu | 1; }
__host__ __device__ inline int plane_elems(int Pu, int Pv, int V) {
    const int x = Pu * plane_ldx(V), y = Pv * plane_ldy(Pu / 2 + 1);
    return x > y ? x : y;
}

// [3][W][V][U] -> [3][W][Pv][Hu]
template <typename R>
__global__ void __launch_bounds__(kPlaneThreads)
k_plane_fwd(const double* __restrict__ in, int U, int V, int W, typename CT<R>::c* __restrict__ out,
            const typename CT<R>::c* __restrict__ twx, const typename CT<R>::c* __restrict__ twy,
            RadixList rx, RadixList ry, const double* __restrict__ scale) {
    typedef typename CT<R>::c C;
    extern __shared__ __align__(16) unsigned char smem_raw[];
    const int Pu = rx.P, Pv = ry.P, Hu = Pu / 2 + 1, VP = (V + 1) / 2;
    const int ldx = plane_ldx(V), ldy = plane_ldy(Hu), ne = plane_elems(Pu, Pv, V);
    C* sx = reinterpret_cast<C*>(smem_raw);
    C* sy = sx + tw_entries<C>(Pu);
    C* b0 = sy + tw_entries<C>(Pv);
    C* b1 = b0 + ne;
    const long long cw = blockIdx.x;
    load_tw(sx, twx, Pu);
    load_tw(sy, twy, Pv);
    for (int i = threadIdx.x; i < (Pu - U) * ldx; i += blockDim.x) {   // the padding of the rows
        b0[U * ldx + i].x = 0;
        b0[U * ldx + i].y = 0;
    }
    pdl_trigger();
    pdl_wait();
    const float inv_u = 1.0f / (float)U;
    for (int it = threadIdx.x; it < VP * U; it += blockDim.x) {
        const int t = __float2int_rz(((float)it + 0.5f) * inv_u), j = it - t * U, v = 2 * t;
        const double* row = in + (cw * V + v) * (long long)U;
        double va = row[j], vb = 0.0;
        if (v + 1 < V) vb = row[U + j];
        if (scale) {   // per-voxel factor (the adjoint transforms chi * lambda)
            const long long m0 = ((cw % W) * V + v) * (long long)U + j;
            va *= scale[m0];
            if (v + 1 < V) vb *= scale[m0 + U];
        }
        b0[j * ldx + t].x = (R)va;
        b0[j * ldx + t].y = (R)vb;
    }
    __syncthreads();
    C* X = fft_lines<C, -1>(b0, b1, rx, VP, ldx, sx);
    C* Y = X == b0 ? b1 : b0;
    // split: A = (Z[k] + conj Z[P-k]) / 2, B = -i (Z[k] - conj Z[P-k]) / 2
    const float inv_vp = 1.0f / (float)VP;
    for (int it = threadIdx.x; it < VP * Hu; it += blockDim.x) {
        const int k = __float2int_rz(((float)it + 0.5f) * inv_vp), t = it - k * VP;
        const C zk = X[k * ldx + t], zm = X[(k ? Pu - k : 0) * ldx + t];
        C A, B;
        A.x = (R)0.5 * (zk.x + zm.x);
        A.y = (R)0.5 * (zk.y - zm.y);
        B.x = (R)0.5 * (zk.y + zm.y);
        B.y = (R)0.5 * (zm.x - zk.x);
        Y[2 * t * ldy + k] = A;
        if (2 * t + 1 < V) Y[(2 * t + 1) * ldy + k] = B;
    }
    for (int i = threadIdx.x; i < (Pv - V) * ldy; i += blockDim.x) {
        Y[V * ldy + i].x = 0;
        Y[V * ldy + i].y = 0;
    }
    __syncthreads();
    const C* Z = fft_lines<C, -1>(Y, X, ry, Hu, ldy, sy);
    const float inv_hu = 1.0f / (float)Hu;
    C* dst = out + cw * Pv * Hu;
    for (int it = threadIdx.x; it < Pv * Hu; it += blockDim.x) {
        const int j = __float2int_rz(((float)it + 0.5f) * inv_hu);
        dst[it] = Z[j * ldy + it - j * Hu];
    }
}

// [3][W][Pv][Hu] -> real [3][W][V][U]
template <typename R>
__global__ void __launch_bounds__(kPlaneThreads)
k_plane_inv(const typename CT<R>::c* __restrict__ in, int U, int V, R* __restrict__ out,
            const typename CT<R>::c* __restrict__ twx, const typename CT<R>::c* __restrict__ twy,
            RadixList rx, RadixList ry) {
    typedef typename CT<R>::c C;
    extern __shared__ __align__(16) unsigned char smem_raw[];
    const int Pu = rx.P, Pv = ry.P, Hu = Pu / 2 + 1, VP = (V + 1) / 2;
    const int ldx = plane_ldx(V), ldy = plane_ldy(Hu), ne = plane_elems(Pu, Pv, V);
    C* sx = reinterpret_cast<C*>(smem_raw);
    C* sy = sx + tw_entries<C>(Pu);
    C* b0 = sy + tw_entries<C>(Pv);
    C* b1 = b0 + ne;
    const long long cw = blockIdx.x;
    load_tw(sx, twx, Pu);
    load_tw(sy, twy, Pv);
    pdl_trigger();
    pdl_wait();
    const float inv_hu = 1.0f / (float)Hu;
    const C* src = in + cw * Pv * Hu;
    for (int it = threadIdx.x; it < Pv * Hu; it += blockDim.x) {
        const int j = __float2int_rz(((float)it + 0.5f) * inv_hu);
        cp_async_c(&b0[j * ldy + it - j * Hu], src + it);
    }
    cp_async_commit_wait();
    __syncthreads();
    C* Y = fft_lines<C, +1>(b0, b1, ry, Hu, ldy, sy);
    C* X = Y == b0 ? b1 : b0;
    // Z[k] = A[k] + i B[k] and Z[P-k] = conj A[k] + i conj B[k] from the two halves
    const float inv_vp = 1.0f / (float)VP;
    for (int it = threadIdx.x; it < VP * Hu; it += blockDim.x) {
        const int k = __float2int_rz(((float)it + 0.5f) * inv_vp), t = it - k * VP;
        const C A = Y[2 * t * ldy + k];
        C B;
        B.x = 0; B.y = 0;
        if (2 * t + 1 < V) B = Y[(2 * t + 1) * ldy + k];
        C z;
        z.x = A.x - B.y;
        z.y = A.y + B.x;
        X[k * ldx + t] = z;
        if (k >= 1 && k < Pu - k) {
            z.x = A.x + B.y;
            z.y = B.x - A.y;
            X[(Pu - k) * ldx + t] = z;
        }
    }
    __syncthreads();
    const C* Z = fft_lines<C, +1>(X, Y, rx, VP, ldx, sx);
    const float inv_u = 1.0f / (float)U;
    for (int it = threadIdx.x; it < VP * U; it += blockDim.x) {
        const int t = __float2int_rz(((float)it + 0.5f) * inv_u), j = it - t * U;
        const C z = Z[j * ldx + t];
        R* row = out + (cw * V + 2 * t) * (long long)U + j;
        row[0] = z.x;
        if (2 * t + 1 < V) row[U] = z.y;
    }
}

RadixList radix_list(const AxisFFT& ax) {
    RadixList rl;
    rl.P = ax.P;
    rl.n = ax.nrad;
    for (int i = 0; i < 16; ++i) rl.r[i] = ax.rad[i];
    return rl;
}

template <typename R> const typename CT<R>::c* table(const AxisFFT& a);
template <> const double2* table<double>(const AxisFFT& a) { return a.tw64; }
template <> const float2* table<float>(const AxisFFT& a) { return a.tw32; }

template <typename R> size_t smem_bytes(int P) {
    typedef typename CT<R>::c C;
    return sizeof(C) * ((size_t)tw_entries<C>(P) + 2 * (size_t)P * (Tile<R>::TB + 1));
}

template <typename R, int P1, int P2>
void launch_mid4s(const typename CT<R>::c* in, typename CT<R>::c* out,
                  const typename CT<R>::c* tw, const MidArgs& a, int nblocks, bool dep,
                  cudaStream_t s) {
    typedef typename CT<R>::c C;
    const size_t sm = sizeof(C) * ((size_t)P1 * P2 * 32 + (size_t)tw_entries<C>(P1 * P2));
    constexpr int threads = 32 * (P1 > P2 ? P1 : P2);
    if (a.dir < 0) {
        allow_smem<k_mid4s<R, P1, P2, -1>>(sm);
        launch_dependent(dep, k_mid4s<R, P1, P2, -1>, nblocks, threads, sm, s, in, out, tw, a);
    } else {
        allow_smem<k_mid4s<R, P1, P2, +1>>(sm);
        launch_dependent(dep, k_mid4s<R, P1, P2, +1>, nblocks, threads, sm, s, in, out, tw, a);
    }
    MOT_LAUNCH_CHECK();
}

// lengths with a four-step codelet (mid_pass, x_pass_codelet)
bool has_codelet(int P) { return P == 64 || P == 96 || P == 210; }

// a strided pass of length ax.P over [3][n_o2] x Hu lines: the four-step kernel for the
// lengths that have a factor pair below, the generic Stockham tile otherwise
template <typename R>
void mid_pass(const typename CT<R>::c* in, typename CT<R>::c* out, const AxisFFT& ax,
              const MidArgs& a, bool dep, cudaStream_t s) {
    const int P = ax.P;
    const long long lines = 3LL * a.n_o2 * a.Hu;
    const int nb32 = (int)((lines + 31) / 32);
    switch (P) {
        case 64: launch_mid4s<R, 8, 8>(in, out, table<R>(ax), a, nb32, dep, s); return;
        case 96: launch_mid4s<R, 8, 12>(in, out, table<R>(ax), a, nb32, dep, s); return;
        case 210: launch_mid4s<R, 14, 15>(in, out, table<R>(ax), a, nb32, dep, s); return;
        default: break;
    }
    constexpr int TB = Tile<R>::TB;
    const size_t sm = smem_bytes<R>(P);
    allow_smem<k_mid<R>>(sm);
    launch_dependent(dep, k_mid<R>, (int)((lines + TB - 1) / TB), NT, sm, s, in, out, table<R>(ax),
                     radix_list(ax), a);
    MOT_LAUNCH_CHECK();
}

__global__ void twiddle_kernel(int P, double2* t64, float2* t32) {
    const int k = blockIdx.x * blockDim.x + threadIdx.x;
    if (k >= P) return;
    double s, c;
    sincospi(2.0 * (double)k / (double)P, &s, &c);
    t64[k] = make_double2(c, -s);
    const float2 h = make_float2((float)c, (float)-s);
    t32[k] = h;                                                   // hi
    t32[P + k] = make_float2((float)(c - (double)h.x), (float)(-s - (double)h.y));   // lo
}

}  // namespace

namespace mot {

void fft_plan_axis(AxisFFT& a, int P) {
    a.P = P;
    a.nrad = 0;
    int n = P;
    while (n % 4 == 0) { a.rad[a.nrad++] = 4; n /= 4; }
    while (n % 2 == 0) { a.rad[a.nrad++] = 2; n /= 2; }
    for (int r : {3, 5, 7})
        while (n % r == 0) { a.rad[a.nrad++] = r; n /= r; }
    if (n != 1) throw MotError{MOT_ERR_ARG, "FFT length has a prime factor above 7"};
    MOT_CUDA_TRY(cudaMalloc(&a.tw64, sizeof(double2) * P));
    MOT_CUDA_TRY(cudaMalloc(&a.tw32, sizeof(float2) * 2 * P));
    twiddle_kernel<<<(P + 255) / 256, 256>>>(P, a.tw64, a.tw32);
    MOT_LAUNCH_CHECK();
    MOT_CUDA_TRY(cudaDeviceSynchronize());
}

void fft_free_axis(AxisFFT& a) {
    cudaFree(a.tw64);
    cudaFree(a.tw32);
    a.tw64 = nullptr;
    a.tw32 = nullptr;
}

// x passes through the four-step codelets where P has one (false: use the generic kernel)
template <typename R, int P1, int P2>
void launch_x4s(bool fwd, mot_ctx* c, const double* Jsoa, typename CT<R>::c* spec, R* real,
                const double* scale, cudaStream_t s) {
    typedef typename CT<R>::c C;
    constexpr int P = P1 * P2;
    const size_t sm = sizeof(C) * ((size_t)P * kXLD + tw_entries<C>(P));
    const int threads = 32 * (P1 > P2 ? P1 : P2);
    const long long npairs = 3LL * c->W * ((c->V + 1) / 2);
    const int blocks = (int)((npairs + kXL - 1) / kXL);
    if (fwd) {
        allow_smem<k_fwd_x4s<R, P1, P2>>(sm);
        launch_dependent(mot::dependent_launches(c), k_fwd_x4s<R, P1, P2>, blocks, threads, sm, s,
                         Jsoa, c->U, c->V, c->W, spec, table<R>(c->ax[0]), scale);
    } else {
        allow_smem<k_inv_x4s<R, P1, P2>>(sm);
        launch_dependent(mot::dependent_launches(c), k_inv_x4s<R, P1, P2>, blocks, threads, sm, s,
                         spec, c->U, c->V, c->W, real, table<R>(c->ax[0]));
    }
    MOT_LAUNCH_CHECK();
}

template <typename R>
bool x_pass_codelet(bool fwd, mot_ctx* c, const double* Jsoa, typename CT<R>::c* spec, R* real,
                    const double* scale, cudaStream_t s) {
    switch (c->ax[0].P) {
        case 64: launch_x4s<R, 8, 8>(fwd, c, Jsoa, spec, real, scale, s); return true;
        case 96: launch_x4s<R, 8, 12>(fwd, c, Jsoa, spec, real, scale, s); return true;
        case 210: launch_x4s<R, 14, 15>(fwd, c, Jsoa, spec, real, scale, s); return true;
        default: return false;
    }
}

// Shared memory of the plane kernels where they are the faster ones, else 0.  Forward +
// inverse x and y passes of a step, microseconds, two kernels each -> the plane kernels:
//   FP32  8^3 20.8 -> 16.3, 24^3 27.9 -> 21.0, 40^3 49.4 -> 40.7, 44^3 63.0 -> 53.9,
//         21 x 27 x 133 46.7 -> 33.3, 64 x 16 x 16 41.7 -> 33.4; but with a codelet for both
//         lengths 32^3 29.3 -> 29.1 and 48^3 41.4 -> 46.1 (its transforms stay in registers)
//   FP64  8^3 29.8 -> 24.0, 16^3 32.6 -> 28.6, 20^3 37.3 -> 36.5, 24^3 40.8 -> 41.4, 28^3
//         52.5 -> 54.2, 16 x 64 x 16 48.1 -> 66.7: a plane is bound by the FP64 units of its
//         one SM unless it is small
// A whole step: FP32 8^3 56.9 -> 50.8, 24^3 85.1 -> 78.8, 44^3 244 -> 239; FP64 8^3 85.6 ->
// 79.4, 16^3 132 -> 123; but 20^3 0.5 us slower, and 16 x 16 x 64 (192 planes, two on some
// SMs) 326 -> 340; with planes enough to even that out 4 x 100 x 100 (300) 1003 -> 956, 21 x
// 27 x 133 (399) 1483 -> 1452.  Between 152 and 300 planes the line is cautious, forward +
// inverse of FP64 grids U x V x W, two kernels -> plane kernels: 27 x 21 153 planes 69.6 -> 80.9,
// 210 81.0 -> 83.3, 228 104 -> 83.2, 294 115 -> 84.9; 20 x 20 153 51.3 -> 53.0, 240 65.3 -> 58.0, 294
// 84.5 -> 60.3; 16 x 16 153 42.7 -> 37.2, 294 57.1 -> 44.6.
template <typename R> size_t plane_pass(const mot_ctx* c) {
    typedef typename CT<R>::c C;
    const int Pu = c->ax[0].P, Pv = c->ax[1].P;
    const size_t sm = sizeof(C) * ((size_t)tw_entries<C>(Pu) + tw_entries<C>(Pv) +
                                   2 * (size_t)plane_elems(Pu, Pv, c->V));
    if (sm > kPlaneSmem) return 0;
    if (std::is_same<R, float>::value) return has_codelet(Pu) && has_codelet(Pv) ? 0 : sm;
    return (Pu * Pv <= 32 * 32 && 3 * c->W <= c->nsm) || 3 * c->W >= 2 * (c->nsm - 2) ? sm : 0;
}
int plane_threads(const mot_ctx* c) {
    const int want = c->ax[1].P * c->Hu / 4;
    return std::min(kPlaneThreads, std::max(64, (want + 31) / 32 * 32));
}

// Every length needs a codelet or a tile of the general kernel (P <= 764 in FP64, 807 in FP32),
// also where another kernel takes the axis: which one does depends on the grid and the step, so a
// longer axis would fail in the middle of a march, and with it the z pass of only some steps.
template <typename R> void fft_require(const mot_ctx* c) {
    for (const AxisFFT& ax : c->ax)
        if (!has_codelet(ax.P)) allow_smem<k_mid<R>>(smem_bytes<R>(ax.P));
}

// kernels of the x and y passes of a transform
template <typename R> int fft_xy_launches(const mot_ctx* c) { return plane_pass<R>(c) ? 1 : 2; }

// x and y passes of the forward transform, [3][W][V][U] -> hb.tmp2 [3][W][Pv][Hu]
template <typename R>
void fft_forward_xy(mot_ctx* c, const double* Jsoa, cudaStream_t s, const double* scale) {
    fft_require<R>(c);
    HistoryBuffers<R>& hb = hbuf<R>(c);
    constexpr int TB = Tile<R>::TB;
    const int U = c->U, V = c->V, W = c->W;
    const int Pu = c->ax[0].P, Pv = c->ax[1].P, Hu = c->Hu;
    if (const size_t sm = plane_pass<R>(c)) {
        allow_smem<k_plane_fwd<R>>(sm);
        launch_dependent(dependent_launches(c), k_plane_fwd<R>, 3 * W, plane_threads(c), sm, s, Jsoa,
                         U, V, W, hb.tmp2, table<R>(c->ax[0]), table<R>(c->ax[1]),
                         radix_list(c->ax[0]), radix_list(c->ax[1]), scale);
        MOT_LAUNCH_CHECK();
        return;
    }
    // x
    if (!x_pass_codelet<R>(true, c, Jsoa, hb.tmp1, nullptr, scale, s)) {
        const long long npairs = 3LL * W * ((V + 1) / 2);
        const size_t sm = smem_bytes<R>(Pu);
        allow_smem<k_fwd_x<R>>(sm);
        launch_dependent(dependent_launches(c), k_fwd_x<R>, (int)((npairs + TB - 1) / TB), NT, sm, s,
                         Jsoa, U, V, W, hb.tmp1, table<R>(c->ax[0]), radix_list(c->ax[0]), scale);
        MOT_LAUNCH_CHECK();
    }
    // y: [3][W][V][Hu] -> [3][W][Pv][Hu]
    {
        MidArgs a;
        a.n_in = V; a.n_out = Pv; a.n_o2 = W;
        a.in_c = (long long)W * V * Hu; a.in_o = (long long)V * Hu; a.in_a = Hu;
        a.out_c = (long long)W * Pv * Hu; a.out_o = (long long)Pv * Hu; a.out_a = Hu;
        a.Hu = Hu; a.dir = -1;
        mid_pass<R>(hb.tmp1, hb.tmp2, c->ax[1], a, dependent_launches(c), s);
    }
}

// z pass of the forward transform, hb.tmp2 -> [3][Pw][Pv][Hu]
template <typename R>
void fft_forward_z(mot_ctx* c, typename CT<R>::c* out, cudaStream_t s) {
    const int W = c->W, Pv = c->ax[1].P, Pw = c->ax[2].P, Hu = c->Hu;
    MidArgs a;
    a.n_in = W; a.n_out = Pw; a.n_o2 = Pv;
    a.in_c = (long long)W * Pv * Hu; a.in_o = Hu; a.in_a = (long long)Pv * Hu;
    a.out_c = (long long)Pw * Pv * Hu; a.out_o = Hu; a.out_a = (long long)Pv * Hu;
    a.Hu = Hu; a.dir = -1;
    mid_pass<R>(hbuf<R>(c).tmp2, out, c->ax[2], a, dependent_launches(c), s);
}

// y and x passes of the inverse transform, hb.tmp2 [3][W][Pv][Hu] -> [3][W][V][U]
template <typename R>
void fft_inverse_yx(mot_ctx* c, R* out, cudaStream_t s) {
    HistoryBuffers<R>& hb = hbuf<R>(c);
    constexpr int TB = Tile<R>::TB;
    const int U = c->U, V = c->V, W = c->W;
    const int Pu = c->ax[0].P, Pv = c->ax[1].P, Hu = c->Hu;
    if (const size_t sm = plane_pass<R>(c)) {
        allow_smem<k_plane_inv<R>>(sm);
        launch_dependent(dependent_launches(c), k_plane_inv<R>, 3 * W, plane_threads(c), sm, s, hb.tmp2,
                         U, V, out, table<R>(c->ax[0]), table<R>(c->ax[1]), radix_list(c->ax[0]),
                         radix_list(c->ax[1]));
        MOT_LAUNCH_CHECK();
        return;
    }
    // y: [3][W][Pv][Hu] -> [3][W][V][Hu]
    {
        MidArgs a;
        a.n_in = Pv; a.n_out = V; a.n_o2 = W;
        a.in_c = (long long)W * Pv * Hu; a.in_o = (long long)Pv * Hu; a.in_a = Hu;
        a.out_c = (long long)W * V * Hu; a.out_o = (long long)V * Hu; a.out_a = Hu;
        a.Hu = Hu; a.dir = +1;
        mid_pass<R>(hb.tmp2, hb.tmp1, c->ax[1], a, dependent_launches(c), s);
    }
    // x: c2r
    if (!x_pass_codelet<R>(false, c, nullptr, hb.tmp1, out, nullptr, s)) {
        const long long npairs = 3LL * W * ((V + 1) / 2);
        const size_t sm = smem_bytes<R>(Pu);
        allow_smem<k_inv_x<R>>(sm);
        launch_dependent(dependent_launches(c), k_inv_x<R>, (int)((npairs + TB - 1) / TB), NT, sm, s,
                         hb.tmp1, U, V, W, out, table<R>(c->ax[0]), radix_list(c->ax[0]));
        MOT_LAUNCH_CHECK();
    }
}

template <typename R>
void fft_inverse(mot_ctx* c, const typename CT<R>::c* in, R* out, cudaStream_t s) {
    const int W = c->W, Pv = c->ax[1].P, Pw = c->ax[2].P, Hu = c->Hu;
    // z: [3][Pw][Pv][Hu] -> [3][W][Pv][Hu]
    MidArgs a;
    a.n_in = Pw; a.n_out = W; a.n_o2 = Pv;
    a.in_c = (long long)Pw * Pv * Hu; a.in_o = Hu; a.in_a = (long long)Pv * Hu;
    a.out_c = (long long)W * Pv * Hu; a.out_o = Hu; a.out_a = (long long)Pv * Hu;
    a.Hu = Hu; a.dir = +1;
    mid_pass<R>(in, hbuf<R>(c).tmp2, c->ax[2], a, dependent_launches(c), s);
    fft_inverse_yx<R>(c, out, s);
}

template void fft_require<double>(const mot_ctx*);
template void fft_require<float>(const mot_ctx*);
template int fft_xy_launches<double>(const mot_ctx*);
template int fft_xy_launches<float>(const mot_ctx*);
template void fft_forward_xy<double>(mot_ctx*, const double*, cudaStream_t, const double*);
template void fft_forward_xy<float>(mot_ctx*, const double*, cudaStream_t, const double*);
template void fft_forward_z<double>(mot_ctx*, double2*, cudaStream_t);
template void fft_forward_z<float>(mot_ctx*, float2*, cudaStream_t);
template void fft_inverse_yx<double>(mot_ctx*, double*, cudaStream_t);
template void fft_inverse_yx<float>(mot_ctx*, float*, cudaStream_t);
template void fft_inverse<double>(mot_ctx*, const double2*, double*, cudaStream_t);
template void fft_inverse<float>(mot_ctx*, const float2*, float*, cudaStream_t);

}  // namespace mot
