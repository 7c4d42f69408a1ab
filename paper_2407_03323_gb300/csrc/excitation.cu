// Tested incident field (Eq. E) on the GPU:
//   E^b_{m,n} = chi_m p_b (1/V) int_{V_m} g(n dt - t0 - r . k_hat) dV,
//   g(tau) = sin(2 pi f_c tau) exp(-tau^2 / (2 sigma_t^2)),
// voxel m occupying [u, u+1] x [v, v+1] x [w, w+1] (h = c dt = 1).  The voxel average
// is a 6-point-per-axis tensor Gauss-Legendre rule; the pulse varies on a scale of
// many voxels so the rule is exact to rounding.
//
// The average A(tau) = int_{[-1/2,1/2]^3} g(tau - q . k_hat) dq is one function of
// tau = n dt - t0 - r_c . k_hat (r_c the voxel centre) for every voxel, so it is
// tabulated once per call on the nodes j / K (j integer) covering every needed tau
// (the tensor rule at each node) and each voxel and step interpolates it through the 10
// nearest nodes (degree 9, Lagrange form).  K is an integer, so the steps of a voxel lie K
// nodes apart at the same fraction of a node spacing: its 10 weights are formed once and a
// step costs 10 multiply-adds.  With f_eff = f_c + 6 / (2 pi sigma_t) bounding the pulse's
// spectrum, the interpolation error is at most (2 pi f_eff / K)^10 * 870 / 10! of max|g|;
// K >= max(2, 2 pi f_eff / 0.057) keeps it below 1e-16, under the rule's rounding.
#include "mot_internal.cuh"

#include <algorithm>
#include <cmath>
#include <mutex>

namespace {

constexpr int NQ = 6;
constexpr int kMaxSetupDevices = 64;
__constant__ double c_qx[NQ], c_qw[NQ];

__global__ void k_plane_wave(long long M, int U, int V, const double* __restrict__ chi, double kx,
                             double ky, double kz, double px, double py, double pz, double fc,
                             double st, double t0, int n_first, int n_steps,
                             double* __restrict__ E) {
    const long long i = (long long)blockIdx.x * blockDim.x + threadIdx.x;
    if (i >= M * n_steps) return;
    const long long m = i % M;
    const int step = (int)(i / M);
    const double ch = chi[m];
    double* o = E + i * 3;
    if (ch == 0.0) { o[0] = o[1] = o[2] = 0.0; return; }
    const int u = (int)(m % U), v = (int)((m / U) % V), w = (int)(m / ((long long)U * V));
    const double tc = (double)(n_first + step) - t0 -
                      ((u + 0.5) * kx + (v + 0.5) * ky + (w + 0.5) * kz);
    const double inv2s2 = 1.0 / (2.0 * st * st);
    double acc = 0.0;
    for (int a = 0; a < NQ; ++a)
        for (int b = 0; b < NQ; ++b)
            for (int c = 0; c < NQ; ++c) {
                const double tau = tc - (c_qx[a] * kx + c_qx[b] * ky + c_qx[c] * kz);
                acc += c_qw[a] * c_qw[b] * c_qw[c] * sinpi(2.0 * fc * tau) * exp(-tau * tau * inv2s2);
            }
    const double g = ch * acc;
    o[0] = g * px;
    o[1] = g * py;
    o[2] = g * pz;
}

// A((j0 + j) / K), j < J, by the tensor rule (nodes on a fixed lattice, so a value does not
// depend on which call tabulates it).  One warp per node, the 216 points dealt to its lanes:
// a table has a few hundred to a few thousand nodes, and with a thread per node they would
// fill only J / 128 SMs (1700 nodes: 14), each bound by its FP64 units.
__global__ void k_pw_table(int J, long long j0, double K, double kx, double ky, double kz,
                           double fc, double st, double* __restrict__ A) {
    const int j = blockIdx.x * (blockDim.x >> 5) + (threadIdx.x >> 5), lane = threadIdx.x & 31;
    if (j >= J) return;
    const double tc = (double)(j0 + j) / K;
    const double inv2s2 = 1.0 / (2.0 * st * st);
    double acc = 0.0;
    for (int i = lane; i < NQ * NQ * NQ; i += 32) {
        const int a = i / (NQ * NQ), b = (i / NQ) % NQ, c = i % NQ;
        const double tau = tc - (c_qx[a] * kx + c_qx[b] * ky + c_qx[c] * kz);
        acc += c_qw[a] * c_qw[b] * c_qw[c] * sinpi(2.0 * fc * tau) * exp(-tau * tau * inv2s2);
    }
    for (int o = 16; o > 0; o >>= 1) acc += __shfl_down_sync(0xffffffffu, acc, o);
    if (lane == 0) A[j] = acc;
}

constexpr int kInterp = 10;   // interpolation points (degree 9)
constexpr int kStepsPerThread = 16;

// One thread per voxel and kStepsPerThread steps: the Lagrange weights of its fraction t of
// a node spacing once (prefix and suffix products of the distances t + 4 - j), then a
// 10-term sum per step.  The warp's 32 x 3 output values are one contiguous run; the lanes
// write it in order (value e of the run is voxel e / 3, component e % 3) instead of three
// stores with a stride of 24 bytes.  Bound by the FP64 units (2 multiply-adds a clock and
// SM): about 13 operations for each active voxel and step.
__global__ void __launch_bounds__(256) k_plane_wave_tab(
    long long M, int U, int V, const double* __restrict__ chi, double kx, double ky, double kz,
    double px, double py, double pz, double phase, int n_steps, long long jr, int K,
    const double* __restrict__ A, double* __restrict__ E) {
    const long long m0 = (long long)blockIdx.x * blockDim.x + (threadIdx.x & ~31);
    const int lane = threadIdx.x & 31;
    const long long m = m0 + lane;
    const int s_lo = blockIdx.y * kStepsPerThread, s_hi = min(n_steps, s_lo + kStepsPerThread);
    const double ch = m < M ? chi[m] : 0.0;
    double wt[kInterp];
    const double* Ai = A;
    if (ch != 0.0) {
        const int u = (int)(m % U), v = (int)((m / U) % V), w = (int)(m / ((long long)U * V));
        // position on the node lattice, counted from the whole part of the call's first
        // n - t0, with phase = floor(t0) - t0: the same for every call, and no digits are lost
        // to a late pulse; step s lies s K nodes further
        const double y = (phase - ((u + 0.5) * kx + (v + 0.5) * ky + (w + 0.5) * kz)) * (double)K;
        const double fl = floor(y), t = y - fl;
        Ai = A + ((long long)fl - (kInterp / 2 - 1) + s_lo * K - jr);
        // 1 / prod_{i != j} (j - i) = (-1)^(9 - j) C(9, j) / 9!
        constexpr double f9 = 362880.0;
        constexpr double cj[kInterp] = {-1 / f9, 9 / f9, -36 / f9, 84 / f9, -126 / f9,
                                        126 / f9, -84 / f9, 36 / f9, -9 / f9, 1 / f9};
        double pre = ch;
#pragma unroll
        for (int j = 0; j < kInterp; ++j) {
            wt[j] = pre * cj[j];
            pre *= t + (double)(kInterp / 2 - 1 - j);
        }
        double suf = 1.0;
#pragma unroll
        for (int j = kInterp - 1; j >= 0; --j) {
            wt[j] *= suf;
            suf *= t + (double)(kInterp / 2 - 1 - j);
        }
    }
    const int run = (int)min(96LL, 3 * (M - m0));      // values of this warp's run
    // component of this lane's values e = lane, lane + 32, lane + 64
    const int c0 = lane % 3, c1 = (lane + 32) % 3, c2 = (lane + 64) % 3;
    const double p0 = c0 == 0 ? px : c0 == 1 ? py : pz, p1 = c1 == 0 ? px : c1 == 1 ? py : pz,
                 p2 = c2 == 0 ? px : c2 == 1 ? py : pz;
    for (int s = s_lo; s < s_hi; ++s, Ai += K) {
        double g = 0.0;
        if (ch != 0.0) {
            double ga = wt[0] * Ai[0], gb = wt[1] * Ai[1];
#pragma unroll
            for (int j = 2; j < kInterp; j += 2) {
                ga += wt[j] * Ai[j];
                gb += wt[j + 1] * Ai[j + 1];
            }
            g = ga + gb;
        }
        const double v0 = __shfl_sync(0xffffffffu, g, lane / 3) * p0;
        const double v1 = __shfl_sync(0xffffffffu, g, (lane + 32) / 3) * p1;
        const double v2 = __shfl_sync(0xffffffffu, g, (lane + 64) / 3) * p2;
        if (run <= 0) continue;
        double* o = E + ((long long)s * M + m0) * 3;
        if (lane < run) o[lane] = v0;
        if (lane + 32 < run) o[lane + 32] = v1;
        if (lane + 64 < run) o[lane + 64] = v2;
    }
}

}  // namespace

namespace mot {

void excitation_setup(int dev) {
    // the __constant__ nodes live once per device and module: upload them the first
    // time a context is created on `dev` (a blocking copy, kept out of the per-call path)
    static std::mutex mu;
    static bool done[kMaxSetupDevices] = {};
    if (dev < 0 || dev >= kMaxSetupDevices)
        throw MotError{MOT_ERR_ARG, "device index beyond the supported range"};
    std::lock_guard<std::mutex> lock(mu);
    if (done[dev]) return;
    // Gauss-Legendre nodes on [-1/2, 1/2] (weights sum to 1)
    double x[NQ], w[NQ];
    {
        const double pi = 3.14159265358979323846;
        for (int i = 0; i < NQ; ++i) {
            double z = std::cos(pi * (i + 0.75) / (NQ + 0.5)), dp = 0.0;
            for (int it = 0; it < 100; ++it) {
                double p0 = 1.0, p1 = z;
                for (int kk = 2; kk <= NQ; ++kk) {
                    const double p2 = ((2.0 * kk - 1.0) * z * p1 - (kk - 1.0) * p0) / kk;
                    p0 = p1;
                    p1 = p2;
                }
                dp = NQ * (z * p1 - p0) / (z * z - 1.0);
                const double dz = p1 / dp;
                z -= dz;
                if (std::fabs(dz) < 1e-17) break;
            }
            x[i] = 0.5 * z;
            w[i] = 1.0 / ((1.0 - z * z) * dp * dp);
        }
    }
    MOT_CUDA_TRY(cudaMemcpyToSymbol(c_qx, x, sizeof x));
    MOT_CUDA_TRY(cudaMemcpyToSymbol(c_qw, w, sizeof w));
    done[dev] = true;
}

void plane_wave(mot_ctx* c, const double k[3], const double p[3], double fc, double st, double t0,
                int n_first, int n_steps, double* Edev, cudaStream_t s) {
    if (!c->pw_tab) {   // no table buffer: the tensor rule at every voxel and step
        const long long tot = c->M * n_steps;
        k_plane_wave<<<(int)((tot + 255) / 256), 256, 0, s>>>(c->M, c->U, c->V, c->chi, k[0], k[1],
                                                              k[2], p[0], p[1], p[2], fc, st, t0,
                                                              n_first, n_steps, Edev);
        MOT_LAUNCH_CHECK();
        return;
    }
    // node spacing from the pulse's spectral extent; range of r_c . k_hat over the grid
    const double pi = 3.14159265358979323846;
    const double feff = std::fabs(fc) + 6.0 / (2.0 * pi * st);
    const double kmin = std::max(2.0, 2.0 * pi * feff / 0.057);
    const int K = (int)std::min(std::ceil(kmin), (double)kPwTable);   // nodes per dt
    const double hstep = 1.0 / K;
    const int N[3] = {c->U, c->V, c->W};
    double rk_lo = 0.0, rk_hi = 0.0;
    for (int a = 0; a < 3; ++a) {
        const double e0 = 0.5 * k[a], e1 = (N[a] - 0.5) * k[a];
        rk_lo += std::min(e0, e1);
        rk_hi += std::max(e0, e1);
    }
    // steps per sub-call so that its tau range fits the table with 6 spare nodes a side
    const double cap = std::floor((kPwTable - 40) * hstep - (rk_hi - rk_lo));
    // Node numbers are whole numbers near (n - t0 - r . k_hat) K.  Below 2^44 FP64 leaves them
    // 2^-7 of a node: the kernel's and the host's differ by less than the spare nodes.  Past that
    // (|t0| of 1e11 steps and more, or a number that is not finite) there is no table.
    const double t0i = std::floor(t0), phase = t0i - t0;
    const bool exact = (std::fabs(t0i) + std::fabs((double)n_first) + n_steps +
                        std::fabs(rk_lo) + std::fabs(rk_hi)) * K < 0x1p44;
    if (!(cap >= 1.0) || !exact) {   // nor for a grid too large for one table at one step
        const long long tot = c->M * n_steps;
        k_plane_wave<<<(int)((tot + 255) / 256), 256, 0, s>>>(c->M, c->U, c->V, c->chi, k[0], k[1],
                                                              k[2], p[0], p[1], p[2], fc, st, t0,
                                                              n_first, n_steps, Edev);
        MOT_LAUNCH_CHECK();
        return;
    }
    const int per = (int)std::min((double)n_steps, cap);
    for (int s0 = 0; s0 < n_steps; s0 += per) {
        const int cnt = std::min(per, n_steps - s0);
        const int nf = n_first + s0;
        // the table's nodes relative to (nf - floor(t0)) K, from the same sums as the kernel's
        const long long jr = (long long)std::floor((phase - rk_hi) * K) - 6;
        const int J = (int)std::min((long long)kPwTable,
                                    (long long)std::ceil((phase - rk_lo + (cnt - 1)) * K) + 7 - jr);
        const long long j0 = (long long)((double)nf - t0i) * K + jr;
        k_pw_table<<<(J + 7) / 8, 256, 0, s>>>(J, j0, (double)K, k[0], k[1], k[2], fc, st,
                                               c->pw_tab);
        MOT_LAUNCH_CHECK();
        const dim3 grid((unsigned)((c->M + 255) / 256),
                        (unsigned)((cnt + kStepsPerThread - 1) / kStepsPerThread));
        k_plane_wave_tab<<<grid, 256, 0, s>>>(
            c->M, c->U, c->V, c->chi, k[0], k[1], k[2], p[0], p[1], p[2], phase, cnt, jr, K,
            c->pw_tab, Edev + (long long)s0 * 3 * c->M);
        MOT_LAUNCH_CHECK();
    }
}

}  // namespace mot
