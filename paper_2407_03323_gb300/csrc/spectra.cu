// Spatial spectra of the interaction elements (App. A, Sec. 3).
//
// The product G_l * J over the N-voxel grid is a 3-level block-Toeplitz product.
// Embedded in a circulant of size P >= 2N - 1 per axis (App. A), it becomes a
// pointwise product of DFTs, with the kernel's DFT
//     Ghat_l(k) = sum_{d = -(N-1)}^{N-1} G_l(d) exp(-2 pi i k . d / P).
// G is even in every d_i for the diagonal components and odd in d_a, d_b (even in the
// third) for the (a, b) component, so Ghat is real, has the same parity in k, and is
// a product of one-sided cosine / sine sums along each axis:
//     even axis: sum_{d>=0} c_d G(d) cos(2 pi k d / P),  c_0 = 1, c_{d>0} = 2
//     odd axis:  sum_{d>0} 2 G(d) sin(2 pi k d / P) times -i; two odd axes give -1.
// Only the octant k_i in [0, P_i/2] is stored; the other bins follow by parity.
#include "mot_internal.cuh"

#include <algorithm>

namespace {

// trig tables laid out [d][k] (k fastest), k < H = P/2 + 1, d < N
__global__ void trig_table_kernel(int P, int N, int H, double* cosw, double* sinw) {
    const int i = blockIdx.x * blockDim.x + threadIdx.x;
    if (i >= N * H) return;
    const int d = i / H, k = i % H;
    const long long kd = ((long long)k * d) % P;
    double s, c;
    sincospi(2.0 * (double)kd / (double)P, &s, &c);
    cosw[i] = (d == 0 ? 1.0 : 2.0) * c;
    sinw[i] = (d == 0 ? 0.0 : 2.0) * s;
}

// Batches of transforms: slab b = (lag - l_first) * 6 + component, one after the other in
// every array.  (One launch per lag, component and pass is 900 launches for a 20^3 grid's 36
// lags, 6.5 of 21 ms of its creation.)

// slab b of g: the octant elements of its lag and component
__global__ void extract_lags_kernel(const int* __restrict__ tab_l0, const double* __restrict__ tab,
                                    long long noff, int l_first, int nslab, double* __restrict__ g) {
    const long long i = (long long)blockIdx.x * blockDim.x + threadIdx.x;
    if (i >= noff * nslab) return;
    const int b = (int)(i / noff), cc = b % 6;
    const long long o = i % noff;
    const int idx = l_first + b / 6 - tab_l0[o];
    g[i] = (idx >= 0 && idx < mot::WIN) ? tab[(o * 6 + cc) * mot::WIN + idx] : 0.0;
}

// g[d] = sum_{l <= n} w[l] G_l(d) for component cc (the lags of the window at d)
__global__ void extract_weighted_kernel(const int* __restrict__ tab_l0,
                                        const double* __restrict__ tab, long long noff,
                                        const double* __restrict__ w, int n, int cc,
                                        double* __restrict__ g) {
    const long long i = (long long)blockIdx.x * blockDim.x + threadIdx.x;
    if (i >= noff) return;
    const int l0 = tab_l0[i];
    double acc = 0.0;
    for (int k = 0; k < mot::WIN && l0 + k <= n; ++k)
        if (l0 + k >= 0) acc = fma(w[l0 + k], tab[(i * 6 + cc) * mot::WIN + k], acc);
    g[i] = acc;
}

// dst[o][cc] += w * src[cc][o], src optionally rounded to FP32 first
__global__ void accum_kernel(const double* __restrict__ src, long long noct, double w,
                             int round32, double* __restrict__ dst) {
    const long long i = (long long)blockIdx.x * blockDim.x + threadIdx.x;
    if (i >= 6 * noct) return;
    const long long o = i / 6;
    const int cc = (int)(i % 6);
    double v = src[cc * noct + o];
    if (round32) v = (double)(float)v;
    dst[i] = fma(w, v, dst[i]);
}

// cosine or sine table of one axis for each component (cc0: component of slab 0)
struct AxisTables {
    const double* w[6];
    int cc0;
    double sign;       // of the odd components' result (two odd axes: (-i)(-i) = -1)
};
// odd axes of component cc (order xx, yy, zz, xy, xz, yz): bit a set if odd along a
__host__ __device__ constexpr int odd_mask(int cc) { return cc < 3 ? 0 : cc == 3 ? 3 : cc == 4 ? 5 : 6; }

// out[row][k] = sum_{d < n} in[row][d] * w[d][k]       (along the fastest axis; rows per slab)
__global__ void pass_fast(const double* __restrict__ in, int n, long long rows, int nslab,
                          AxisTables t, int K, double* __restrict__ out) {
    const long long i = (long long)blockIdx.x * blockDim.x + threadIdx.x;
    if (i >= rows * nslab * K) return;
    const long long row = i / K;
    const int k = (int)(i % K);
    const double* w = t.w[(t.cc0 + (int)(row / rows)) % 6];
    const double* src = in + row * n;
    double acc = 0.0;
    for (int d = 0; d < n; ++d) acc = fma(src[d], w[(long long)d * K + k], acc);
    out[i] = acc;
}

// out[o][k][f] = sum_{d < n} in[o][d][f] * w[d][k]     (along a middle axis; outer per slab)
__global__ void pass_mid(const double* __restrict__ in, int n, int F, long long outer, int nslab,
                         AxisTables t, int K, double* __restrict__ out) {
    const long long i = (long long)blockIdx.x * blockDim.x + threadIdx.x;
    if (i >= outer * nslab * K * F) return;
    const int f = (int)(i % F);
    const int k = (int)((i / F) % K);
    const long long o = i / ((long long)F * K);
    const int cc = (t.cc0 + (int)(o / outer)) % 6;
    const double* w = t.w[cc];
    const double* src = in + o * (long long)n * F + f;
    double acc = 0.0;
    for (int d = 0; d < n; ++d) acc = fma(src[(long long)d * F], w[(long long)d * K + k], acc);
    out[i] = odd_mask(cc) ? t.sign * acc : acc;
}

// [lags][6][noct] (component-major) -> [lags][noct][6] in the history precision
template <typename R>
__global__ void interleave_kernel(const double* __restrict__ src, long long noct, int lags,
                                  R* __restrict__ dst) {
    const long long i = (long long)blockIdx.x * blockDim.x + threadIdx.x;
    if (i >= 6 * noct * lags) return;
    const long long l = i / (6 * noct), r = i % (6 * noct);
    const long long o = r / 6;
    const int cc = (int)(r % 6);
    dst[i] = (R)src[(l * 6 + cc) * noct + o];
}

inline int nblk(long long n, int b) { return (int)((n + b - 1) / b); }

struct TrigTables {
    double* cosw[3] = {nullptr, nullptr, nullptr};
    double* sinw[3] = {nullptr, nullptr, nullptr};
    ~TrigTables() {
        for (int a = 0; a < 3; ++a) { cudaFree(cosw[a]); cudaFree(sinw[a]); }
    }
};

struct Scratch {
    double* g = nullptr;
    double* t1 = nullptr;
    double* t2 = nullptr;
    ~Scratch() { cudaFree(g); cudaFree(t1); cudaFree(t2); }
};

AxisTables axis_tables(const TrigTables& tt, int axis, int cc0, bool last) {
    AxisTables t;
    for (int cc = 0; cc < 6; ++cc)
        t.w[cc] = (odd_mask(cc) >> axis) & 1 ? tt.sinw[axis] : tt.cosw[axis];
    t.cc0 = cc0;
    t.sign = last ? -1.0 : 1.0;
    return t;
}

// spectra of the nslab octant kernels in sc.g (components cc0, cc0 + 1, .. modulo 6) into
// dst [nslab][noct]
void transform(mot_ctx* c, const TrigTables& tt, Scratch& sc, int cc0, int nslab, double* dst) {
    const int U = c->U, V = c->V, W = c->W;
    const int Hu = c->Hu, Hv = c->Hv, Hw = c->Hw;
    cudaStream_t s = c->stream;
    // x: [W][V][U] -> [W][V][Hu]
    pass_fast<<<nblk((long long)W * V * Hu * nslab, 256), 256, 0, s>>>(
        sc.g, U, (long long)W * V, nslab, axis_tables(tt, 0, cc0, false), Hu, sc.t1);
    MOT_LAUNCH_CHECK();
    // y: [W][V][Hu] -> [W][Hv][Hu]
    pass_mid<<<nblk((long long)W * Hv * Hu * nslab, 256), 256, 0, s>>>(
        sc.t1, V, Hu, W, nslab, axis_tables(tt, 1, cc0, false), Hv, sc.t2);
    MOT_LAUNCH_CHECK();
    // z: [W][Hv*Hu] -> [Hw][Hv*Hu]
    pass_mid<<<nblk((long long)Hw * Hv * Hu * nslab, 256), 256, 0, s>>>(
        sc.t2, W, Hv * Hu, 1, nslab, axis_tables(tt, 2, cc0, true), Hw, dst);
    MOT_LAUNCH_CHECK();
}

// spectra of lags l .. l + lags - 1, all components, into dst [lags][6][noct]
void spectra_of_lags(mot_ctx* c, const TrigTables& tt, Scratch& sc, int l, int lags, double* dst) {
    const long long noff = (long long)c->U * c->V * c->W;
    extract_lags_kernel<<<nblk(noff * 6 * lags, 256), 256, 0, c->stream>>>(
        c->tab_l0, c->tab, noff, l, 6 * lags, sc.g);
    MOT_LAUNCH_CHECK();
    transform(c, tt, sc, 0, 6 * lags, dst);
}

void make_tables(mot_ctx* c, TrigTables& tt) {
    const int N[3] = {c->U, c->V, c->W};
    const int H[3] = {c->Hu, c->Hv, c->Hw};
    for (int a = 0; a < 3; ++a) {
        MOT_CUDA_TRY(cudaMalloc(&tt.cosw[a], sizeof(double) * N[a] * H[a]));
        MOT_CUDA_TRY(cudaMalloc(&tt.sinw[a], sizeof(double) * N[a] * H[a]));
        trig_table_kernel<<<nblk((long long)N[a] * H[a], 256), 256, 0, c->stream>>>(
            c->ax[a].P, N[a], H[a], tt.cosw[a], tt.sinw[a]);
        MOT_LAUNCH_CHECK();
    }
}

// scratch of `slabs` transforms at a time
void make_scratch(mot_ctx* c, Scratch& sc, int slabs) {
    const long long noff = (long long)c->U * c->V * c->W;
    MOT_CUDA_TRY(cudaMalloc(&sc.g, sizeof(double) * noff * slabs));
    MOT_CUDA_TRY(cudaMalloc(&sc.t1, sizeof(double) * (long long)c->W * c->V * c->Hu * slabs));
    MOT_CUDA_TRY(cudaMalloc(&sc.t2, sizeof(double) * (long long)c->W * c->Hv * c->Hu * slabs));
}

// lags per batch: about a million octant bins, a few tens of MB of scratch (one lag at a
// time from about 50^3 on, where its passes fill the GPU by themselves)
int batch_lags(const mot_ctx* c, int lags) {
    return (int)std::max(1LL, std::min((long long)lags, (1LL << 20) / (6 * c->noct)));
}

}  // namespace

namespace mot {

// ghat[lag-1][octant bin][6] for lags 1..ell, in the history precision, unnormalised
void compute_spectra(mot_ctx* c) {
    TrigTables tt;
    Scratch sc;
    const int nb = batch_lags(c, c->ell);
    make_tables(c, tt);
    make_scratch(c, sc, 6 * nb);
    double* tmp = nullptr;
    MOT_CUDA_TRY(cudaMalloc(&tmp, sizeof(double) * c->noct * 6 * nb));
    try {
        for (int l = 1; l <= c->ell; l += nb) {
            const int m = std::min(nb, c->ell - l + 1);
            spectra_of_lags(c, tt, sc, l, m, tmp);
            const long long off = (long long)(l - 1) * 6 * c->noct;
            if (c->precision == MOT_FP64)
                interleave_kernel<double><<<nblk(6 * c->noct * m, 256), 256, 0, c->stream>>>(
                    tmp, c->noct, m, c->h64.ghat + off);
            else
                interleave_kernel<float><<<nblk(6 * c->noct * m, 256), 256, 0, c->stream>>>(
                    tmp, c->noct, m, c->h32.ghat + off);
            MOT_LAUNCH_CHECK();
        }
        MOT_CUDA_TRY(cudaStreamSynchronize(c->stream));
    } catch (...) {
        cudaFree(tmp);
        throw;
    }
    cudaFree(tmp);
}

void spectrum_of_lag(mot_ctx* c, int l, double* host_out) {
    TrigTables tt;
    Scratch sc;
    make_tables(c, tt);
    make_scratch(c, sc, 6);
    double* tmp = nullptr;
    MOT_CUDA_TRY(cudaMalloc(&tmp, sizeof(double) * c->noct * 6));
    try {
        spectra_of_lags(c, tt, sc, l, 1, tmp);
        MOT_CUDA_TRY(cudaMemcpyAsync(host_out, tmp, sizeof(double) * c->noct * 6,
                                     cudaMemcpyDeviceToHost, c->stream));
        MOT_CUDA_TRY(cudaStreamSynchronize(c->stream));
    } catch (...) {
        cudaFree(tmp);
        throw;
    }
    cudaFree(tmp);
}


// dst [noct][6] (FP64, unnormalised) = spectrum of sum_{l=0}^{n} w_l G_l.  Without
// round32 the weighted kernel is combined in space and transformed once; with round32
// every lag l >= 1 is transformed alone and rounded to FP32 before it is weighted (the
// per-lag spectra the FP32-history direct scheme multiplies; lag 0 stays FP64, as in
// the Z_0 solve).
void spectrum_of_combination(mot_ctx* c, const double* w_host, int n, bool round32,
                             double* dst) {
    TrigTables tt;
    Scratch sc;
    make_tables(c, tt);
    make_scratch(c, sc, 6);
    double* tmp = nullptr;
    double* w = nullptr;
    const long long noff = (long long)c->U * c->V * c->W;
    cudaStream_t s = c->stream;
    try {
        MOT_CUDA_TRY(cudaMalloc(&tmp, sizeof(double) * c->noct * 6));
        MOT_CUDA_TRY(cudaMalloc(&w, sizeof(double) * (n + 1)));
        MOT_CUDA_TRY(cudaMemcpyAsync(w, w_host, sizeof(double) * (n + 1),
                                     cudaMemcpyHostToDevice, s));
        if (!round32) {
            for (int cc = 0; cc < 6; ++cc) {
                extract_weighted_kernel<<<nblk(noff, 256), 256, 0, s>>>(c->tab_l0, c->tab, noff,
                                                                       w, n, cc, sc.g + cc * noff);
                MOT_LAUNCH_CHECK();
            }
            transform(c, tt, sc, 0, 6, tmp);
            interleave_kernel<double><<<nblk(6 * c->noct, 256), 256, 0, s>>>(tmp, c->noct, 1, dst);
            MOT_LAUNCH_CHECK();
        } else {
            MOT_CUDA_TRY(cudaMemsetAsync(dst, 0, sizeof(double) * 6 * c->noct, s));
            for (int l = 0; l <= n; ++l) {
                if (w_host[l] == 0.0) continue;
                spectra_of_lags(c, tt, sc, l, 1, tmp);
                accum_kernel<<<nblk(6 * c->noct, 256), 256, 0, s>>>(tmp, c->noct, w_host[l],
                                                                    l >= 1, dst);
                MOT_LAUNCH_CHECK();
            }
        }
        MOT_CUDA_TRY(cudaStreamSynchronize(s));
    } catch (...) {
        cudaFree(tmp);
        cudaFree(w);
        throw;
    }
    cudaFree(tmp);
    cudaFree(w);
}

}  // namespace mot
