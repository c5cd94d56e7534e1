// gf_observables.cu -- observables of the flow / MH chain on the device
// (paper arXiv:2208.08903 Sec. 1: expectation values as chain averages, the
// autocorrelation time tau_ac with N_indep = N_conf / (2 tau_ac); Sec. 3: the
// condensate, the zero-momentum two-point function and the effective sample
// size of the analysis tools).
//
//  - per configuration: M = mean of phi and C(t) = (1/V) sum_tau Phi(tau)
//    Phi(tau + t), Phi(tau) = sum of phi over the slice at outermost
//    coordinate tau (V/L contiguous sites).  Threads accumulate in FP32 pairs
//    (error-free transformations), so the kernel reads each field once with
//    little FP64 work.  FP32 fields of 2D L = 16, 32, 64 and 3D L = 8, 16 are
//    streamed through shared memory by bulk copies; other shapes read global
//    memory directly (a warp per configuration or a block per configuration).
//  - chain gather: the chain's series O[chain_idx[k]] of a per-proposal
//    observable.
//  - Gamma(t) of a series (a CTA takes up to eight lags, fixed-order FP64
//    reduction), then the Madras-Sokal automatic window for tau_int in one warp.
//  - ESS fraction (sum w)^2 / (n sum w^2) of w = exp(log w), the largest
//    log w factored out (one cluster of CTAs).
#include <algorithm>
#include <cmath>

#include <cooperative_groups.h>

#include "gf_async.cuh"
#include "gf_common.cuh"

namespace gf {
namespace {

namespace cg = cooperative_groups;

constexpr int kObsThreads = 256;
constexpr int kRedThreads = 1024;

// One CTA per configuration (grid-stride).  Dynamic shared memory: L pairs.
// Each warp sums whole slices: every lane first issues up to four 16-byte loads,
// then adds them into its FP32 pair; the warp reduces the pairs the same way.
// M and C(t) are formed from the slice pairs in pair arithmetic too and widened
// to FP64 once per output, so FP64 instructions are a few per configuration.
__global__ void __launch_bounds__(kObsThreads) obs_kernel(int L, int64_t V, int64_t B, double inv_v,
                                                         const float* __restrict__ phi, double* __restrict__ M,
                                                         double* __restrict__ C) {
    extern __shared__ FF Phi[];
    const int lane = threadIdx.x & 31, wid = threadIdx.x >> 5, nw = blockDim.x >> 5;
    const int64_t S = V / L;
    for (int64_t b = blockIdx.x; b < B; b += gridDim.x) {
        const float* p = phi + b * V;
        const bool vec = (S % 4 == 0) && ((reinterpret_cast<uintptr_t>(p) & 15) == 0);
        for (int tau = wid; tau < L; tau += nw) {
            const float* q = p + (int64_t)tau * S;
            FF acc{0.f, 0.f};
            if (vec) {
                const float4* q4 = reinterpret_cast<const float4*>(q);
                const int64_t S4 = S / 4;
                for (int64_t i0 = lane; i0 < S4; i0 += 4 * 32) {
                    float4 v[4];
#pragma unroll
                    for (int k = 0; k < 4; ++k)
                        if (i0 + 32 * k < S4) v[k] = __ldg(q4 + i0 + 32 * k);
#pragma unroll
                    for (int k = 0; k < 4; ++k)
                        if (i0 + 32 * k < S4) {
                            ff_add(acc, v[k].x);
                            ff_add(acc, v[k].y);
                            ff_add(acc, v[k].z);
                            ff_add(acc, v[k].w);
                        }
                }
            } else {
                for (int64_t i = lane; i < S; i += 32) ff_add(acc, __ldg(q + i));
            }
            acc = warp_sum_ff(acc);
            if (lane == 0) Phi[tau] = acc;
        }
        __syncthreads();
        if (M && threadIdx.x == 0) {
            FF m{0.f, 0.f};
            for (int tau = 0; tau < L; ++tau) ff_add(m, Phi[tau]);
            M[b] = ff_to_double(m) * inv_v;
        }
        if (C) {
            for (int t = threadIdx.x; t < L; t += blockDim.x) {
                FF acc{0.f, 0.f};
                for (int tau = 0, u = t; tau < L; ++tau, u = (u + 1 == L) ? 0 : u + 1) ff_fma(acc, Phi[tau], Phi[u]);
                C[b * L + t] = ff_to_double(acc) * inv_v;
            }
        }
        __syncthreads();
    }
}

// One warp per configuration (grid-stride over configurations), for slices of
// a multiple of 128 sites and L <= kObsWarpMaxL: lane l reads 16-byte pieces
// l, l + 32, ... of the field in batches of eight loads, so every lane sees the
// same slice at the same step.  Each lane sums its part of a slice with a
// compensated sum (Knuth's TwoSum into hi, the exact rounding errors added
// into lo: seven FP32 operations per site) and, at the slice's end, leaves the
// pair in the warp's table (dynamic shared memory, [L][32] pairs, lane index
// xor-swizzled by the slice so stores and the column reads below are free of
// bank conflicts).  Lane tau then adds up the 32 pairs of slice tau in pair
// arithmetic; M and C(t) follow from the L slice sums, as pairs, widened to
// FP64 once per output.  No CTA barrier is needed.  1/V comes from the host.
constexpr int kObsWarpMaxL = 64;
__global__ void __launch_bounds__(kObsThreads) obs_warp_kernel(int L, int64_t V, int64_t B, double inv_v,
                                                              const float* __restrict__ phi,
                                                              double* __restrict__ M, double* __restrict__ C) {
    extern __shared__ FF tab_all[];
    const int lane = threadIdx.x & 31, wid = threadIdx.x >> 5, wpb = blockDim.x >> 5;
    FF* tab = tab_all + (size_t)wid * L * 32;
    const int64_t S4 = V / L / 4;                 // 16-byte pieces per slice, a multiple of 32
    const int per = (int)(S4 / 32);               // batches of 32 pieces per slice
    const int nk = L * per;                       // pieces per lane
    for (int64_t b = (int64_t)blockIdx.x * wpb + wid; b < B; b += (int64_t)gridDim.x * wpb) {
        const float4* q4 = reinterpret_cast<const float4*>(phi + b * V) + lane;
        float hi = 0.f, lo = 0.f;
        for (int k0 = 0; k0 < nk; k0 += 8) {
            float4 v[8];
#pragma unroll
            for (int j = 0; j < 8; ++j)
                if (k0 + j < nk) v[j] = __ldg(q4 + (int64_t)32 * (k0 + j));
#pragma unroll
            for (int j = 0; j < 8; ++j) {
                if (k0 + j < nk) {
                    const float c[4] = {v[j].x, v[j].y, v[j].z, v[j].w};
#pragma unroll
                    for (int q = 0; q < 4; ++q) {
                        const float s = hi + c[q];
                        const float bp = s - hi;
                        lo += (hi - (s - bp)) + (c[q] - bp);
                        hi = s;
                    }
                    if ((k0 + j + 1) % per == 0) {             // end of slice (k0 + j) / per
                        const int tau = (k0 + j) / per;
                        tab[tau * 32 + ((lane ^ tau) & 31)] = FF{hi, lo};
                        hi = 0.f;
                        lo = 0.f;
                    }
                }
            }
        }
        __syncwarp();
        for (int tau = lane; tau < L; tau += 32) {
            FF acc{0.f, 0.f};
            for (int i = 0; i < 32; ++i) ff_add(acc, tab[tau * 32 + ((i ^ tau) & 31)]);
            tab[tau * 32 + ((0 ^ tau) & 31)] = acc;     // the slice sum, in lane 0's entry
        }
        __syncwarp();
        const auto slice = [&](int tau) -> FF { return tab[tau * 32 + (tau & 31)]; };
        if (M && lane == 0) {
            FF m{0.f, 0.f};
            for (int tau = 0; tau < L; ++tau) ff_add(m, slice(tau));
            M[b] = ff_to_double(m) * inv_v;
        }
        if (C) {
            for (int t = lane; t < L; t += 32) {
                FF a{0.f, 0.f};
                for (int tau = 0, u = t; tau < L; ++tau, u = (u + 1 == L) ? 0 : u + 1) ff_fma(a, slice(tau), slice(u));
                C[b * L + t] = ff_to_double(a) * inv_v;
            }
        }
        __syncwarp();
    }
}

// Streaming form: a block of 128 threads owns a ring of shared-memory buffers
// that bulk copies fill with whole configurations (BulkRing), so the next
// configurations arrive while the current one is summed.  The TPS = 128 / L
// consecutive threads of slice tau each sum every TPS-th 4-site chunk of it
// with a compensated sum (TwoSum into hi, the exact rounding errors into lo:
// seven FP32 operations per site), combine their pairs by shuffles and leave
// Phi(tau) in shared memory; after one block barrier threads t < L form C(t)
// and thread L forms M, in pair arithmetic widened to FP64 once per output.
// Phi is double-buffered, so one barrier per configuration suffices.
constexpr int kOsThreads = 128;
constexpr long long kOsWaitLimit = 1ll << 24;     // bounded wait for a configuration's bulk copy

template <int ND, int L>
__global__ void __launch_bounds__(kOsThreads) obs_stream_kernel(int64_t B, double inv_v,
                                                                const float* __restrict__ phi,
                                                                double* __restrict__ M_out,
                                                                double* __restrict__ C_out,
                                                                int32_t* __restrict__ status) {
    constexpr int V = ND == 3 ? L * L * L : L * L;
    constexpr int NBUF = ring_depth<V * 4>();
    constexpr int CPS = V / L / 4;                          // chunks per slice
    constexpr int TPS = kOsThreads / L;                     // threads per slice
    constexpr int PER = CPS >= TPS ? CPS / TPS : 1;         // chunks per thread
    static_assert((L & (L - 1)) == 0 && L >= 8 && L <= 64 && TPS <= 32, "streaming lattice");
    static_assert(CPS % TPS == 0 || TPS % CPS == 0, "slice split");
    extern __shared__ __align__(16) unsigned char smem_raw[];
    uint64_t* full = reinterpret_cast<uint64_t*>(smem_raw + NBUF * V * 4);  // [NBUF]
    FF* Phi = reinterpret_cast<FF*>(full + NBUF);                          // [2][L]
    int* abort_s = reinterpret_cast<int*>(Phi + 2 * L);
    const int tid = threadIdx.x, tau = tid / TPS, sub = tid % TPS;
    const BulkRing<NBUF> ring(smem_raw, full, phi, V * 4, B);
    if (tid == 0) {
        *abort_s = 0;
        ring.start();
    }
    __syncthreads();
    int64_t k = 0;
    for (; k < ring.count; ++k) {
        const int64_t b = blockIdx.x + k * gridDim.x;
        const float4* p4 = static_cast<const float4*>(ring.data(k));
        float hi = 0.f, lo = 0.f;
        if (!ring.wait(k, kOsWaitLimit)) {
            set_status(status, GF_ETIMEOUT);
            *abort_s = 1;
        } else if (CPS >= TPS || sub < CPS) {
#pragma unroll
            for (int j = 0; j < PER; ++j) {
                const float4 v = p4[tau * CPS + sub + TPS * j];
                const float c[4] = {v.x, v.y, v.z, v.w};
#pragma unroll
                for (int q = 0; q < 4; ++q) {
                    const float s = hi + c[q], bp = s - hi;
                    lo += (hi - (s - bp)) + (c[q] - bp);
                    hi = s;
                }
            }
        }
        FF a{hi, lo};
#pragma unroll
        for (int o = TPS / 2; o > 0; o >>= 1)
            ff_add(a, FF{__shfl_xor_sync(0xffffffffu, a.hi, o), __shfl_xor_sync(0xffffffffu, a.lo, o)});
        FF* ph = Phi + (k & 1) * L;
        if (sub == 0) ph[tau] = a;
        __syncthreads();
        if (*abort_s) break;                    // block-uniform
        if (tid == 0) ring.refill(k);           // every thread has read this buffer
        if (tid < L) {
            if (C_out) {
                FF c{0.f, 0.f};
#pragma unroll 4
                for (int u = 0; u < L; ++u) ff_fma(c, ph[u], ph[(u + tid) & (L - 1)]);
                C_out[b * L + tid] = ff_to_double(c) * inv_v;
            }
        } else if (tid == L && M_out) {
            FF m{0.f, 0.f};
#pragma unroll 4
            for (int u = 0; u < L; ++u) ff_add(m, ph[u]);
            M_out[b] = ff_to_double(m) * inv_v;
        }
    }
    if (tid == 0) ring.drain(k, kOsWaitLimit);
}

template <int ND, int L>
void launch_obs_stream(int64_t B, double inv_v, const float* phi, double* M, double* C, cudaStream_t stream,
                       bool* ok) {
    constexpr int V = ND == 3 ? L * L * L : L * L;
    constexpr int NBUF = ring_depth<V * 4>();
    const size_t smem = (size_t)NBUF * V * 4 + NBUF * 8 + 2 * L * sizeof(FF) + 16;
    auto kern = obs_stream_kernel<ND, L>;
    if (cudaFuncSetAttribute(kern, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem) != cudaSuccess) return;
    int per_sm = 0;
    if (cudaOccupancyMaxActiveBlocksPerMultiprocessor(&per_sm, kern, kOsThreads, smem) != cudaSuccess ||
        per_sm < 1)
        per_sm = 1;
    const int64_t grid = std::min<int64_t>(B, (int64_t)num_sms() * per_sm);
    kern<<<(unsigned)grid, kOsThreads, smem, stream>>>(B, inv_v, phi, M, C, status_word(stream));
    *ok = true;
}

// The streaming kernel for FP32 fields of 2D L = 16, 32, 64 and 3D L = 8, 16
// that start on a 16-byte boundary; false when the shape or the alignment does
// not qualify.
bool launch_obs_stream_if(int nd, int L, int64_t B, double inv_v, const float* phi, double* M, double* C,
                          cudaStream_t stream) {
    if ((reinterpret_cast<uintptr_t>(phi) & 15) != 0) return false;
    bool ok = false;
    if (nd == 2 && L == 16) launch_obs_stream<2, 16>(B, inv_v, phi, M, C, stream, &ok);
    else if (nd == 2 && L == 32) launch_obs_stream<2, 32>(B, inv_v, phi, M, C, stream, &ok);
    else if (nd == 2 && L == 64) launch_obs_stream<2, 64>(B, inv_v, phi, M, C, stream, &ok);
    else if (nd == 3 && L == 8) launch_obs_stream<3, 8>(B, inv_v, phi, M, C, stream, &ok);
    else if (nd == 3 && L == 16) launch_obs_stream<3, 16>(B, inv_v, phi, M, C, stream, &ok);
    return ok;
}

// out[k][j] = values[(chain_idx[k] - idx0) * width + j]; an index outside
// [0, n_values) writes NaN and records GF_EINVAL in the status word.
__global__ void gather_kernel(int64_t n, const int64_t* __restrict__ chain_idx, int64_t idx0, int64_t n_values,
                              const double* __restrict__ values, int width, double* __restrict__ out,
                              int32_t* status) {
    const int64_t total = n * width;
    for (int64_t i = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; i < total;
         i += (int64_t)gridDim.x * blockDim.x) {
        const int64_t k = i / width;
        const int j = (int)(i - k * width);
        const int64_t r = chain_idx[k] - idx0;
        if (r < 0 || r >= n_values) {
            out[i] = __longlong_as_double(0x7ff8000000000000ll);
            set_status(status, GF_EINVAL);
        } else {
            out[i] = values[r * width + j];
        }
    }
}

// The reductions over a series run as one cluster of kRedCluster CTAs (one for
// short series): FP64 instructions take about 19 cycles of an SM per warp, so a
// single CTA is bound by its SM's FP64 pipe, and a cluster combines its CTAs'
// sums through distributed shared memory without scratch memory or a second
// launch.  Fixed order: rank by rank.  Measured on 16,384 values against one CTA:
// ESS 112 -> 32 us, mean 24 -> 10 us.
constexpr int kRedCluster = 8;
constexpr int64_t kRedClusterMinN = 2048;

struct ClusterPos {
    cg::cluster_group cl = cg::this_cluster();
    int rank = (int)cl.block_rank(), size = (int)cl.num_blocks();
    __device__ int64_t first() const { return (int64_t)rank * blockDim.x + threadIdx.x; }
    __device__ int64_t stride() const { return (int64_t)size * blockDim.x; }
    // v of every rank, combined by op in rank order (slot: a shared variable of this CTA)
    template <typename Op>
    __device__ double combine(double v, double* slot, Op op) {
        if (threadIdx.x == 0) *slot = v;
        cl.sync();
        double r = *cl.map_shared_rank(slot, 0);
        for (int i = 1; i < size; ++i) r = op(r, *cl.map_shared_rank(slot, i));
        cl.sync();                                   // every rank has read it
        return r;
    }
};
__device__ __forceinline__ double dadd(double a, double b) { return a + b; }
__device__ __forceinline__ double dmax(double a, double b) { return fmax(a, b); }

__device__ __forceinline__ double warp_max(double v) {
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) v = fmax(v, __shfl_xor_sync(0xffffffffu, v, o));
    return v;
}
// The block's N values combined per warp, then over the warps by thread 0..N-1
// (valid in red_out[0 .. N) after the trailing barrier).
template <int N, typename WarpOp, typename Op>
__device__ void block_combine(const double (&v)[N], double (*red)[32], double* red_out, WarpOp wop, Op op) {
    const int lane = threadIdx.x & 31, wid = threadIdx.x >> 5, nw = blockDim.x >> 5;
#pragma unroll
    for (int i = 0; i < N; ++i) {
        const double w = wop(v[i]);
        if (lane == 0) red[i][wid] = w;
    }
    __syncthreads();
    if (threadIdx.x < N) {
        double r = red[threadIdx.x][0];
        for (int w = 1; w < nw; ++w) r = op(r, red[threadIdx.x][w]);
        red_out[threadIdx.x] = r;
    }
    __syncthreads();
}

// dbar = mean of (y_k - y_0), one cluster, fixed order.  Stored in out[3].
__global__ void __launch_bounds__(kRedThreads) mean_dev_kernel(int64_t n, const double* __restrict__ y,
                                                              double* __restrict__ out) {
    __shared__ double red[1][32], tot[1], slot;
    ClusterPos c;
    const double y0 = y[0];
    double acc[1] = {0.0};
    for (int64_t k = c.first(); k < n; k += c.stride()) acc[0] += y[k] - y0;
    block_combine<1>(acc, red, tot, [](double v) { return warp_sum(v); }, dadd);
    const double sum = c.combine(tot[0], &slot, dadd);
    if (c.rank == 0 && threadIdx.x == 0) out[3] = sum / (double)n;
}

// Gamma(t) for LT consecutive lags per block (grid-stride): a tile of the
// centred series is formed once in shared memory and read by every lag, so an
// element costs 2 / LT subtractions and one multiply-add per lag instead of
// four and one (16,384 values, 1,001 lags: 167 -> 70 us).  The FP64 pipe bounds it; LT = the lags divided by the SMs (at
// most 8) keeps one block per SM.
constexpr int kGammaTile = 1024, kGammaMaxLags = 8;
template <int LT>
__global__ void __launch_bounds__(kObsThreads) gamma_kernel(int64_t n, const double* __restrict__ y, int t_max,
                                                           const double* __restrict__ stats,
                                                           double* __restrict__ gamma) {
    __shared__ double d[kGammaTile], e[kGammaTile + LT], red[LT][32], tot[LT];
    const double y0 = y[0], dbar = stats[3];
    const auto centred = [&](int64_t k) { return k < n ? (y[k] - y0) - dbar : 0.0; };
    for (int t0 = blockIdx.x * LT; t0 <= t_max; t0 += gridDim.x * LT) {
        double acc[LT];
#pragma unroll
        for (int l = 0; l < LT; ++l) acc[l] = 0.0;
        for (int64_t k0 = 0; k0 + t0 < n; k0 += kGammaTile) {
            __syncthreads();
            for (int i = threadIdx.x; i < kGammaTile; i += blockDim.x) d[i] = centred(k0 + i);
            for (int i = threadIdx.x; i < kGammaTile + LT; i += blockDim.x) e[i] = centred(k0 + t0 + i);
            __syncthreads();
            // (the centred series is zero past its end: no bound per lag)
            for (int i = threadIdx.x; i < kGammaTile; i += blockDim.x) {
                const double v = d[i];
#pragma unroll
                for (int l = 0; l < LT; ++l) acc[l] = fma(v, e[i + l], acc[l]);
            }
        }
        block_combine<LT>(acc, red, tot, [](double v) { return warp_sum(v); }, dadd);
        if (threadIdx.x < LT && t0 + (int)threadIdx.x <= t_max)
            gamma[t0 + threadIdx.x] = tot[threadIdx.x] / (double)(n - t0 - (int)threadIdx.x);
    }
}

// Madras-Sokal window and the summary {tau, W, error, mean}; one warp: the
// ratios of 32 lags at a time, added in order.
__global__ void window_kernel(int64_t n, const double* __restrict__ y, const double* __restrict__ gamma, int t_max,
                              double c, double* __restrict__ out) {
    const int lane = threadIdx.x;
    const double mean = y[0] + out[3], g0 = gamma[0];
    double tau = 0.5;
    int W = t_max;
    if (g0 > 0.0) {
        bool found = false;
        for (int w0 = 1; w0 <= t_max && !found; w0 += 32) {
            const double r = w0 + lane <= t_max ? gamma[w0 + lane] / g0 : 0.0;
            for (int i = 0; i < 32 && w0 + i <= t_max; ++i) {
                tau += __shfl_sync(0xffffffffu, r, i);
                if ((double)(w0 + i) >= c * tau) { W = w0 + i; found = true; break; }
            }
        }
    } else {
        W = 0;
    }
    __syncwarp();
    if (lane != 0) return;
    out[0] = tau;
    out[1] = (double)W;
    out[2] = g0 > 0.0 ? tau * sqrt((4.0 * W + 2.0) / (double)n) : 0.0;
    out[3] = mean;
}

// ESS fraction in one cluster: max, then sum w and sum w^2 in a fixed order.
__global__ void __launch_bounds__(kRedThreads) ess_kernel(int64_t n, const double* __restrict__ logw,
                                                         double* __restrict__ out) {
    __shared__ double red[2][32], tot[2], slot;
    ClusterPos c;
    double mx[1] = {-INFINITY};
    for (int64_t k = c.first(); k < n; k += c.stride()) mx[0] = fmax(mx[0], logw[k]);
    block_combine<1>(mx, red, tot, [](double v) { return warp_max(v); }, dmax);
    const double top = c.combine(tot[0], &slot, dmax);
    if (!(top > -INFINITY)) {                      // n == 0 or all weights zero (the same in every rank)
        if (c.rank == 0 && threadIdx.x == 0) *out = 0.0;
        return;
    }
    double s[2] = {0.0, 0.0};
    for (int64_t k = c.first(); k < n; k += c.stride()) {
        const double w = exp(logw[k] - top);
        s[0] += w;
        s[1] += w * w;
    }
    block_combine<2>(s, red, tot, [](double v) { return warp_sum(v); }, dadd);
    const double s1 = c.combine(tot[0], &slot, dadd), s2 = c.combine(tot[1], &slot, dadd);
    if (c.rank == 0 && threadIdx.x == 0) *out = s1 * s1 / ((double)n * s2);
}

// Launches a reduction over n elements as one cluster.
template <typename... P, typename... A>
bool launch_reduction(void (*kern)(P...), int64_t n, cudaStream_t stream, A... args) {
    const unsigned size = n >= kRedClusterMinN ? kRedCluster : 1;
    cudaLaunchConfig_t cfg = {};
    cfg.gridDim = dim3(size);
    cfg.blockDim = dim3(kRedThreads);
    cfg.stream = stream;
    cudaLaunchAttribute attr;
    attr.id = cudaLaunchAttributeClusterDimension;
    attr.val.clusterDim.x = size;
    attr.val.clusterDim.y = attr.val.clusterDim.z = 1;
    cfg.attrs = &attr;
    cfg.numAttrs = 1;
    return cudaLaunchKernelEx(&cfg, kern, args...) == cudaSuccess;
}

template <int LT = kGammaMaxLags>
void launch_gamma(int lags_per_block, int64_t n, const double* y, int t_max, const double* stats, double* gamma,
                  cudaStream_t stream) {
    if constexpr (LT > 1) {
        if (lags_per_block < LT) {
            launch_gamma<LT - 1>(lags_per_block, n, y, t_max, stats, gamma, stream);
            return;
        }
    }
    const int64_t blocks = ((int64_t)t_max + LT) / LT;
    gamma_kernel<LT><<<(unsigned)std::min<int64_t>(blocks, (int64_t)num_sms() * 8), kObsThreads, 0, stream>>>(
        n, y, t_max, stats, gamma);
}

int64_t ipow(int64_t a, int e) {
    int64_t r = 1;
    while (e-- > 0) r *= a;
    return r;
}

}  // namespace
}  // namespace gf

using namespace gf;

extern "C" {

gf_status gf_observables(int32_t nd, int32_t L, int64_t B, const float* d_phi, double* d_M_out, double* d_C_out,
                         cudaStream_t stream) {
    if ((nd != 2 && nd != 3) || L < 1 || L > GF_OBS_MAX_L || B < 0) return GF_EINVAL;
    if (B > 0 && (!d_phi || (!d_M_out && !d_C_out))) return GF_EINVAL;
    if (B == 0) return GF_OK;
    const int64_t V = ipow(L, nd);
    const int64_t S = V / L;
    if (launch_obs_stream_if(nd, L, B, 1.0 / (double)V, d_phi, d_M_out, d_C_out, stream)) {
        // streaming kernel launched
    } else if (S % 128 == 0 && L <= kObsWarpMaxL && (reinterpret_cast<uintptr_t>(d_phi) & 15) == 0) {
        // warps per block: each warp's table is L x 32 pairs; at most 48 KB per block
        const int wpb = (int)std::max<int64_t>(1, std::min<int64_t>(kObsThreads / 32, 49152 / (256 * (int64_t)L)));
        const size_t smem = (size_t)wpb * L * 32 * sizeof(FF);
        const unsigned grid = (unsigned)std::min<int64_t>((B + wpb - 1) / wpb, (int64_t)num_sms() * 16);
        obs_warp_kernel<<<grid, 32 * wpb, smem, stream>>>(L, V, B, 1.0 / (double)V, d_phi, d_M_out, d_C_out);
    } else {
        const size_t smem = sizeof(FF) * (size_t)L;
        const unsigned grid = (unsigned)std::min<int64_t>(B, (int64_t)num_sms() * 8);
        obs_kernel<<<grid, kObsThreads, smem, stream>>>(L, V, B, 1.0 / (double)V, d_phi, d_M_out, d_C_out);
    }
    GF_CHECK_LAUNCH();
    return GF_OK;
}

gf_status gf_chain_gather(int64_t n, const int64_t* d_chain_idx, int64_t idx0, int64_t n_values,
                          const double* d_values, int32_t width, double* d_out, cudaStream_t stream) {
    if (n < 0 || width < 1 || n_values < 0) return GF_EINVAL;
    if (n > 0 && (!d_chain_idx || !d_values || !d_out)) return GF_EINVAL;
    if (n == 0) return GF_OK;
    const int64_t total = n * width;
    const unsigned grid = (unsigned)std::max<int64_t>(1, std::min<int64_t>((total + 255) / 256, num_sms() * 16LL));
    gather_kernel<<<grid, 256, 0, stream>>>(n, d_chain_idx, idx0, n_values, d_values, width, d_out, status_word(stream));
    GF_CHECK_LAUNCH();
    return GF_OK;
}

gf_status gf_autocorr(int64_t n, const double* d_y, int32_t t_max, double c_window, double* d_gamma_out,
                      double* d_tau_out, cudaStream_t stream) {
    if (n < 1 || t_max < 0 || t_max >= n || !(c_window > 0.0)) return GF_EINVAL;
    if (!d_y || !d_gamma_out || !d_tau_out) return GF_EINVAL;
    if (!launch_reduction(mean_dev_kernel, n, stream, n, d_y, d_tau_out)) return GF_ECUDA;
    const int lags = (int)(((int64_t)t_max + num_sms()) / num_sms());
    launch_gamma(std::min(lags, kGammaMaxLags), n, d_y, t_max, d_tau_out, d_gamma_out, stream);
    GF_CHECK_LAUNCH();
    window_kernel<<<1, 32, 0, stream>>>(n, d_y, d_gamma_out, t_max, c_window, d_tau_out);
    GF_CHECK_LAUNCH();
    return GF_OK;
}

gf_status gf_ess(int64_t n, const double* d_logw, double* d_ess_out, cudaStream_t stream) {
    if (n < 0 || !d_ess_out || (n > 0 && !d_logw)) return GF_EINVAL;
    if (!launch_reduction(ess_kernel, n, stream, n, d_logw, d_ess_out)) return GF_ECUDA;
    GF_CHECK_LAUNCH();
    return GF_OK;
}

}  // extern "C"
