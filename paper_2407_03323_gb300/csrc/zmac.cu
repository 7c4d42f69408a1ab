// The z passes of the spatial transforms and the lag products in one kernel (Sec. 3, Eq.
// PnFFTMOT).  Per step, for every line along kw of the (kv, ku) plane:
//   1. forward z transform of the y-transformed J_{n-1} (zero-padded W -> Pw), stored to the
//      spectral ring;
//   2. Phat(k) = scale * (sum of the far levels' entries + sum_{l=1}^{L} Ghat_l(k) Jhat_{n-l}(k)),
//      lag 1 from the transform just made;
//   3. inverse z transform of Phat, of which the W rows the grid needs go back in place.
// As three kernels the step wrote Jhat and read it back for lag 1, wrote and read Phat, and
// had two more launches.  Used for FP64 and for small FP32 grids (fused_z in history.cu says
// where the line lies); FP32 on large grids keeps the separate HBM-bound product kernel.
//
// A block takes TB consecutive positions of the (kv, ku) plane (contiguous in every array,
// also across rows) and all three components: 3 TB lines in two shared-memory buffers.  TB
// is 8 (64-byte runs of FP32 bins), less where the plane would give fewer blocks than SMs
// or where the lines would not fit.  The line transforms are the four-step codelets for the
// lengths that have one, Stockham stages otherwise (fft_core.cuh).  The product step takes
// kw and its mirror Pw - kw together: the kernel spectrum covers the octant k_i <= P_i / 2,
// its (a, b) component is odd in k_a and k_b, so one load serves both with the signs of the
// components with z flipped; kv beyond Pv / 2 flips those with y.
// FP32-history: each lag's contribution is formed with FP32 FMAs and added into the running sum
// with an error-free two-sum (accumulate.cuh).
#include "mot_internal.cuh"
#include "accumulate.cuh"
#include "fft_core.cuh"

#include <algorithm>

using namespace mot_fft;

namespace {

template <typename R> struct ZArgs {
    typedef typename CT<R>::c C;
    C* tmp;               // [3][W][plane]: y-transformed J_{n-1} in, z-inverted Phat out
    C* ring;              // [hring][3][nbins]
    const R* ghat;        // [lag][noct][6], lag 1 first
    const C* far[8];      // this step's entries of the far levels ([3][nbins] each)
    const C* tw;
    int nfar, fwd;        // fwd: make Jhat_{n-1} here (else it is in the ring already)
    int hring, slot1;     // ring slot of J_{n-1}
    int L;                // lags 1 .. L
    int split;            // lanes that share the lags of a bin (a power of two, <= 8 and hring)
    int W, Pv, Pw, Hu, Hv, Hw;
    int plane;            // Pv * Hu
    long long nbins, noct;
    R scale;
    RadixList rl;
};

// acc += G x for the real symmetric G = (xx, yy, zz, xy, xz, yz).  FP64 chains the 18
// multiply-adds into the sums (no separate additions: every FP64 instruction holds a
// sub-partition for 64 cycles); FP32 forms a lag's contribution first, for the two-sum
__device__ __forceinline__ void add_product(Acc<double>* acc, const double* G, const double2& x,
                                            const double2& y, const double2& z) {
    double2 &o0 = acc[0].s, &o1 = acc[1].s, &o2 = acc[2].s;
    o0.x = fma(G[0], x.x, fma(G[3], y.x, fma(G[4], z.x, o0.x)));
    o0.y = fma(G[0], x.y, fma(G[3], y.y, fma(G[4], z.y, o0.y)));
    o1.x = fma(G[3], x.x, fma(G[1], y.x, fma(G[5], z.x, o1.x)));
    o1.y = fma(G[3], x.y, fma(G[1], y.y, fma(G[5], z.y, o1.y)));
    o2.x = fma(G[4], x.x, fma(G[5], y.x, fma(G[2], z.x, o2.x)));
    o2.y = fma(G[4], x.y, fma(G[5], y.y, fma(G[2], z.y, o2.y)));
}
__device__ __forceinline__ void add_product(Acc<float>* acc, const float* G, const float2& x,
                                            const float2& y, const float2& z) {
    typedef float2 C;
    C ox, oy, oz;
    ox.x = G[0] * x.x + G[3] * y.x + G[4] * z.x;
    ox.y = G[0] * x.y + G[3] * y.y + G[4] * z.y;
    oy.x = G[3] * x.x + G[1] * y.x + G[5] * z.x;
    oy.y = G[3] * x.y + G[1] * y.y + G[5] * z.y;
    oz.x = G[4] * x.x + G[5] * y.x + G[2] * z.x;
    oz.y = G[4] * x.y + G[5] * y.y + G[2] * z.y;
    acc[0].add(ox);
    acc[1].add(oy);
    acc[2].add(oz);
}

// Phat on the block's lines: lag 1 from X (if made here), result to Y, both [kw][ld]
template <typename R, int TB>
__device__ __forceinline__ void products(const ZArgs<R>& a, const typename CT<R>::c* X,
                                         typename CT<R>::c* Y, int ld, int f0) {
    typedef typename CT<R>::c C;
    typedef typename std::conditional<std::is_same<R, double>::value, double2, float2>::type R2;
    constexpr int U = sizeof(R) == 4 ? 3 : 2;    // lags whose loads are issued together
    const int g = threadIdx.x & (a.split - 1);     // this lane's share of the lags
    const int items = a.Hw * TB, per = blockDim.x / a.split;
    // all lanes of a warp make a round, the surplus on the last item (their results are
    // dropped): the shares are added with full-warp shuffles
    for (int it0 = 0; it0 < items; it0 += per) {
        if (it0 + (int)(threadIdx.x & ~31u) / a.split >= items) break;     // a warp without items
        const int it = min(it0 + (int)threadIdx.x / a.split, items - 1);
        const int t = it % TB, kw = it / TB;
        const int f = min(f0 + t, a.plane - 1);
        const bool keep = it0 + (int)threadIdx.x / a.split < items && f0 + t < a.plane;
        const int kv = f / a.Hu, ku = f - kv * a.Hu;
        const bool fv = 2 * kv > a.Pv;
        const int kvo = fv ? a.Pv - kv : kv;
        const bool pair = kw > 0 && 2 * kw < a.Pw;
        const int kw2 = pair ? a.Pw - kw : kw;
        const long long o = ((long long)kw * a.Hv + kvo) * a.Hu + ku;
        const long long bin1 = (long long)kw * a.plane + f, bin2 = (long long)kw2 * a.plane + f;
        const R sv = fv ? (R)-1 : (R)1;
        // (without a mirror the second set repeats the first and is dropped: no branch
        // stands between the loads of one lag and the next, so several lags are in flight)
        Acc<R> acc1[3], acc2[3];
#pragma unroll
        for (int c = 0; c < 3; ++c) { acc1[c].zero(); acc2[c].zero(); }
#pragma unroll 2
        for (int k = g; k < a.nfar; k += a.split) {   // far-lag contributions of this step
            const C* p = a.far[k];
            C u[3], v[3];
#pragma unroll
            for (int c = 0; c < 3; ++c) { u[c] = p[c * a.nbins + bin1]; v[c] = p[c * a.nbins + bin2]; }
#pragma unroll
            for (int c = 0; c < 3; ++c) { acc1[c].add(u[c]); acc2[c].add(v[c]); }
        }
        const R2* gp = reinterpret_cast<const R2*>(a.ghat + o * 6) + g * (a.noct * 3);
        const long long gstep = a.noct * 3 * a.split;   // in R2 units per lag of this lane
        const long long stride = 3 * a.nbins;
        auto lag = [&](const R2& g01, const R2& g23, const R2& g45, const C* x, const C* y) {
            const R G[6] = {g01.x, g01.y, g23.x, sv * g23.y, g45.x, sv * g45.y};
            const R H[6] = {G[0], G[1], G[2], G[3], -G[4], -G[5]};
            add_product(acc1, G, x[0], x[1], x[2]);
            add_product(acc2, H, y[0], y[1], y[2]);
        };
        int l = 1 + g, slot = a.slot1 - g;
        if (slot < 0) slot += a.hring;
        if (a.fwd && l == 1 && a.L >= 1) {
            const C* x = X + kw * ld + (f - f0);
            const C* y = X + kw2 * ld + (f - f0);
            const C xs[3] = {x[0], x[TB], x[2 * TB]}, ys[3] = {y[0], y[TB], y[2 * TB]};
            lag(gp[0], gp[1], gp[2], xs, ys);
            gp += gstep;
            slot -= a.split;
            if (slot < 0) slot += a.hring;
            l += a.split;
        }
        for (; l <= a.L; l += U * a.split) {
            R2 gv[U][3];
            C x[U][3], y[U][3];
#pragma unroll
            for (int u = 0; u < U; ++u) {
                if (l + u * a.split > a.L) break;
                const C* base = a.ring + (long long)slot * stride;
                slot -= a.split;
                if (slot < 0) slot += a.hring;
#pragma unroll
                for (int c = 0; c < 3; ++c) {
                    gv[u][c] = gp[c];
                    x[u][c] = base[c * a.nbins + bin1];
                    y[u][c] = base[c * a.nbins + bin2];
                }
                gp += gstep;
            }
#pragma unroll
            for (int u = 0; u < U; ++u) {
                if (l + u * a.split > a.L) break;
                lag(gv[u][0], gv[u][1], gv[u][2], x[u], y[u]);
            }
        }
        for (int o2 = 1; o2 < a.split; o2 <<= 1)
#pragma unroll
            for (int c = 0; c < 3; ++c) { acc1[c].merge(o2); acc2[c].merge(o2); }
        if (!keep || g != 0) continue;
#pragma unroll
        for (int c = 0; c < 3; ++c) {
            C v = acc1[c].get();
            v.x *= a.scale;
            v.y *= a.scale;
            Y[kw * ld + c * TB + t] = v;
            if (pair) {
                v = acc2[c].get();
                v.x *= a.scale;
                v.y *= a.scale;
                Y[kw2 * ld + c * TB + t] = v;
            }
        }
    }
}

// Four-step transform of the NL lines of `in` ([P1 P2][ld], the first nvalid rows valid, the
// others zero) through `mid`: n = n1 + P1 n2, k = k2 + P2 k1; out(k, line, value).
template <typename C, int P1, int P2, int DIR, int NL, typename Out>
__device__ __forceinline__ void four_step_lines(const C* in, C* mid, const C* stw, int ld,
                                                int nvalid, Out&& out) {
    constexpr int P = P1 * P2;
    for (int it = threadIdx.x; it < P1 * NL; it += blockDim.x) {
        const int line = it % NL, n1 = it / NL;
        C x[P2];
        Unroll1<0, P2>::run([&](auto q) {
            constexpr int n2 = decltype(q)::value;
            const int idx = n1 + P1 * n2;
            C v;
            v.x = 0; v.y = 0;
            if (idx < nvalid) v = in[idx * ld + line];
            x[n2] = v;
        });
        dft_ct<P2, DIR>(x);
        Unroll1<0, P2>::run([&](auto q) {
            constexpr int k2 = decltype(q)::value;
            mid[(n1 * P2 + k2) * ld + line] = twmul_tab(stw, (n1 * k2) % P, P, DIR, x[k2]);
        });
    }
    __syncthreads();
    for (int it = threadIdx.x; it < P2 * NL; it += blockDim.x) {
        const int line = it % NL, k2 = it / NL;
        C y[P1];
        Unroll1<0, P1>::run([&](auto q) {
            constexpr int n1 = decltype(q)::value;
            y[n1] = mid[(n1 * P2 + k2) * ld + line];
        });
        dft_ct<P1, DIR>(y);
        Unroll1<0, P1>::run([&](auto q) {
            constexpr int k1 = decltype(q)::value;
            out(k2 + P2 * k1, line, y[k1]);
        });
    }
}

template <typename R, int TB, int P1, int P2>
__global__ void __launch_bounds__(256, 2) k_zmac(const __grid_constant__ ZArgs<R> a) {
    typedef typename CT<R>::c C;
    constexpr int NL = 3 * TB, ld = NL + 1;
    constexpr bool kFourStep = P1 * P2 > 1;
    extern __shared__ __align__(16) unsigned char smem_raw[];
    const int P = kFourStep ? P1 * P2 : a.Pw;
    C* stw = reinterpret_cast<C*>(smem_raw);
    C* b0 = stw + tw_entries<C>(P);
    C* b1 = b0 + P * ld;
    const int f0 = blockIdx.x * TB;
    load_tw(stw, a.tw, P);
    pdl_trigger();
    pdl_wait();
    if (a.fwd) {
        // lines c * TB + t: component c, plane position f0 + t
        const int rows = kFourStep ? a.W : P;      // Stockham reads the zero padding too
        for (int it = threadIdx.x; it < rows * NL; it += blockDim.x) {
            const int line = it % NL, w = it / NL;
            const int c = line / TB, f = f0 + line % TB;
            const bool ok = w < a.W && f < a.plane;
            cp_async_c(&b0[w * ld + line],
                       ok ? a.tmp + ((long long)c * a.W + w) * a.plane + f : a.tmp, ok);
        }
        cp_async_commit_wait();
    }
    __syncthreads();
    C* slot = a.ring + (long long)a.slot1 * 3 * a.nbins + f0;
    C* X = b0;
    if (a.fwd) {
        if constexpr (kFourStep) {
            four_step_lines<C, P1, P2, -1, NL>(b0, b1, stw, ld, a.W, [&](int k, int line, C v) {
                b0[k * ld + line] = v;
                const int c = line / TB, t = line % TB;
                if (f0 + t < a.plane) slot[c * a.nbins + (long long)k * a.plane + t] = v;
            });
            __syncthreads();
        } else {
            X = fft_tile<C, NL>(b0, b1, P, a.rl.r, a.rl.n, ld, stw, -1);
            for (int it = threadIdx.x; it < P * NL; it += blockDim.x) {
                const int line = it % NL, k = it / NL;
                const int c = line / TB, t = line % TB;
                if (f0 + t < a.plane) slot[c * a.nbins + (long long)k * a.plane + t] = X[k * ld + line];
            }
        }
    }
    C* Y = X == b0 ? b1 : b0;
    products<R, TB>(a, X, Y, ld, f0);
    __syncthreads();
    auto store = [&](int w, int line, C v) {
        const int c = line / TB, t = line % TB;
        if (w < a.W && f0 + t < a.plane)
            a.tmp[((long long)c * a.W + w) * a.plane + f0 + t] = v;
    };
    if constexpr (kFourStep) {
        four_step_lines<C, P1, P2, +1, NL>(Y, X, stw, ld, P, store);
    } else {
        const C* Z = fft_tile<C, NL>(Y, X, P, a.rl.r, a.rl.n, ld, stw, +1);
        for (int it = threadIdx.x; it < a.W * NL; it += blockDim.x) {
            const int line = it % NL, w = it / NL;
            store(w, line, Z[w * ld + line]);
        }
    }
}

template <typename R> const typename CT<R>::c* table(const AxisFFT& a);
template <> const double2* table<double>(const AxisFFT& a) { return a.tw64; }
template <> const float2* table<float>(const AxisFFT& a) { return a.tw32; }

template <typename R> size_t zmac_smem(int P, int TB) {
    typedef typename CT<R>::c C;
    return sizeof(C) * ((size_t)tw_entries<C>(P) + 2 * (size_t)P * (3 * TB + 1));
}

template <typename R, int TB, int P1, int P2>
void launch(mot_ctx* c, const ZArgs<R>& a, cudaStream_t s) {
    const size_t sm = zmac_smem<R>(a.Pw, TB);
    allow_smem<k_zmac<R, TB, P1, P2>>(sm);
    // Threads: whole rounds of the product step (Hw = P / 2 + 1 is odd, and 33 x 4 pairs on
    // 128 threads would take a second round for 4 of them); where the transforms are the
    // larger part (FP32, or up to three lags on a small plane), a stage of them in one round
    // too.  More threads than that leave room for fewer blocks: FP64, 28^3, 7 lags 64 us with
    // 128, 72 with 256.  FP64 with the lags of block 2 (one) and 4 (three), without -> with the
    // stage's threads: 12^3 18.9 -> 15.7 and 19.1 -> 18.3, 20^3 24.3 -> 23.4 and 30.9 -> 31.7,
    // 24^3 28.6 -> 26.5 and 34.4 -> 32.8; but past eight positions an SM 28^3 40.9 -> 46.9 and
    // 49.6 -> 57.1, 64 x 16 x 16 31.0 -> 37.7 and 39.5 -> 46.3.
    const int lanes = a.Hw * TB * a.split, rounds = (lanes + 255) / 256;
    int threads = (lanes + rounds - 1) / rounds;
    if (sizeof(R) == 4 || (a.L < 4 && a.plane <= 8 * c->nsm))
        threads = std::max(threads,
                           std::min(256, 3 * TB * (P1 * P2 > 1 ? std::max(P1, P2) : a.Pw / 2)));
    launch_dependent(mot::dependent_launches(c), k_zmac<R, TB, P1, P2>, (a.plane + TB - 1) / TB,
                     (threads + 31) / 32 * 32, sm, s, a);
    MOT_LAUNCH_CHECK();
}

template <typename R, int TB>
void launch_len(mot_ctx* c, const ZArgs<R>& a, cudaStream_t s) {
    switch (a.Pw) {
        case 64: launch<R, TB, 8, 8>(c, a, s); break;
        case 96: launch<R, TB, 8, 12>(c, a, s); break;
        case 210: launch<R, TB, 14, 15>(c, a, s); break;
        default: launch<R, TB, 1, 1>(c, a, s);
    }
}

template <typename R>
ZArgs<R> z_args(mot_ctx* c) {
    ZArgs<R> a;
    a.tmp = hbuf<R>(c).tmp2;
    for (int k = 0; k < 8; ++k) a.far[k] = nullptr;
    a.tw = table<R>(c->ax[2]);
    a.W = c->W;
    a.Pv = c->ax[1].P; a.Pw = c->ax[2].P;
    a.Hu = c->Hu; a.Hv = c->Hv; a.Hw = c->Hw;
    a.plane = a.Pv * a.Hu;
    a.nbins = c->nbins; a.noct = c->noct;
    a.scale = (R)(1.0 / ((double)c->ax[0].P * c->ax[1].P * c->ax[2].P));
    a.rl.P = c->ax[2].P;
    a.rl.n = c->ax[2].nrad;
    for (int i = 0; i < 16; ++i) a.rl.r[i] = c->ax[2].rad[i];
    return a;
}

template <typename R>
void run(mot_ctx* c, ZArgs<R>& a, cudaStream_t s) {
    // Lanes that share the lags of a bin: an FP64 instruction holds its sub-partition for 64
    // cycles whatever its lanes do, so a small grid spreads its products over the GPU
    // (8^3, 15 lags, 1,296 bin pairs: 35 us without the split)
    a.split = 1;
    const long long items = (long long)a.plane * a.Hw;
    while (sizeof(R) == 8 && a.split < 8 && a.L >= 2 * a.split &&
           2 * a.split * items <= 32LL * 8 * c->nsm)
        a.split *= 2;
    // TB = 8 where that gives two blocks per SM at least and two blocks fit an SM's shared
    // memory (FP64 only: FP32 comes here with small planes); fewer for small planes
    // (16 x 9: 18 blocks of 8) and long lines
    const bool wide = a.plane >= 16LL * c->nsm && zmac_smem<R>(a.Pw, 8) <= 110 * 1024;
    const bool mid = a.plane >= 4LL * c->nsm && zmac_smem<R>(a.Pw, 4) <= 200 * 1024;
    if constexpr (sizeof(R) == 8) {
        if (wide) return launch_len<R, 8>(c, a, s);
    }
    if (mid) launch_len<R, 4>(c, a, s);
    else if (a.plane >= 2LL * c->nsm) launch_len<R, 2>(c, a, s);
    else launch<R, 1, 1, 1>(c, a, s);
}

}  // namespace

namespace mot {

template <typename R>
void zmac(mot_ctx* c, int n, bool fwd, int L, const typename CT<R>::c* const* far, int nfar,
          cudaStream_t s) {
    HistoryBuffers<R>& hb = hbuf<R>(c);
    ZArgs<R> a = z_args<R>(c);
    a.ring = hb.jhat_ring;
    a.ghat = hb.ghat;
    for (int k = 0; k < nfar; ++k) a.far[k] = far[k];
    a.nfar = nfar;
    a.fwd = fwd;
    a.hring = c->hring;
    a.slot1 = (int)slot_index(n - 1, c->hring);
    a.L = L;
    run(c, a, s);
}

template void zmac<double>(mot_ctx*, int, bool, int, const double2* const*, int, cudaStream_t);
template void zmac<float>(mot_ctx*, int, bool, int, const float2* const*, int, cudaStream_t);

}  // namespace mot
