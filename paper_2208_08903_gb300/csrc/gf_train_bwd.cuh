// gf_train_bwd.cuh -- the reverse pass of one coupling layer (paper
// arXiv:2208.08903 Sec. 1, the gradient of the shifted reverse KL divergence),
// two equal hidden widths C in {8, 16, 24, 32}, kernel size 3.  After the
// layer's h1, h2 and s have been recomputed and its affine adjoint has left
// g3 = (dL/ds_pre, dL/dt) (zero at the fixed sites):
//   k_back2  : gh2 = LReLU'(h2) conv3^T(g3), gh1 = LReLU'(h1) conv2^T(gh2)
//   k_wgrad2 : dW2, db2 from h1 and gh2
//   k_back1  : gx += conv1^T(gh1) at the fixed sites, dW1, db1
//   k_wgrad3 : dW3, db3 from h2 and g3
// Activations are [B][C/4][V][4];
// a work unit is G consecutive slices (outermost axis) of one configuration,
// its inputs staged in shared memory chunk-major with one halo slice on each
// side.  All sums are FP32 in a fixed order: convolutions one chain per output
// (taps, then channels), weight gradients as described below.
//
// Measured per layer at batch 1024 of 2D L=32 width 32, against one kernel per
// operation with its inputs read through L1: gh2 and gh1 592 -> 494 us, conv1's
// two 213 -> 80, dW3 103 -> 50, dW2 610 -> 569; at batch 64 of 2D L=16 width 16
// (12 layers) a whole step 1.89 -> 0.78 ms.
#pragma once

#include <algorithm>
#include <type_traits>

#include "gf_flow_fp32_kernel.cuh"

namespace gf {
namespace bwd {

using f32k::cp16;
using f32k::cp_wait;
using f32k::load_w;
using f32k::wrap;

constexpr int kBudget = 227 * 1024;

struct BwdArgs {
    int L, S, V, G, frozen;
    int64_t B;
    float slope;
    FastDiv fd_S, fd_L, fd_Sh, fd_Lh;
    const float* xl;            // the layer's input
    const float *h1, *h2, *g3;
    float *gh2, *gh1, *gx;
    const float *W1b, *W2b, *W3b;   // transposed, tap-flipped: [t][c], [t][o][i], [t][2][c]
    float* partial;             // [cta][T + 1][Cin][Cout]
};

// Stages slices s0 - halo .. s0 + G - 1 + halo (mod L) of a chunk-major tensor
// of C channels of configuration b: dst[c4 * pitch + site] float4.
template <int C>
__device__ __forceinline__ void stage_slab(float* dst, int pitch, const float* src, const BwdArgs& a, int64_t b, int s0,
                                           int halo) {
    const int ns = (a.G + 2 * halo) * a.S, first = (s0 - halo) * a.S;
    for (int c4 = 0; c4 < C / 4; ++c4) {
        const float* p = src + (b * (C / 4) + c4) * (int64_t)a.V * 4;
        for (int i = threadIdx.x; i < ns; i += blockDim.x)
            cp16(dst + (c4 * pitch + i) * 4, p + (int64_t)wrap(first + i, a.V) * 4);
    }
}

// ------------------------------------------------------------------ k_back2
// FP32-pipe bound (conv2^T): warp tile 32 NS sites x 8 channels of packed
// FMAs as in the sampler's conv2, W2b in shared memory for the CTA's life, two
// CTAs per SM where they fit so that one computes while the other stages.
constexpr int kBack2Threads = 256;

template <int ND, int C>
__host__ __device__ constexpr int back2_weights() { return (ND == 3 ? 27 : 9) * (C * C + 2 * C); }

template <int ND, int C>
size_t back2_smem(int S, int G) {
    return (size_t)(back2_weights<ND, C>() + (C / 4) * ((G + 2) * S + 1) * 4 + (G + 4) * S * 2) * 4;
}

template <int ND, int C, int NS>
__device__ __forceinline__ void back2_tile(const BwdArgs& a, const float* W2, const float* g_s, int pitch, int task,
                                           int64_t b, int s0) {
    constexpr int T = ND == 3 ? 27 : 9;
    const int L = a.L, S = a.S, nf = a.G * S, nblk = (nf + 32 * NS - 1) / (32 * NS);
    const int lane = threadIdx.x & 31, g = task / nblk, blk = task - g * nblk, co = g * 8;
    int at[NS];                                  // slice of the slab, y, x: 10 bits each
#pragma unroll
    for (int k = 0; k < NS; ++k) {
        const int f = min(blk * (32 * NS) + lane + 32 * k, nf - 1);
        const int r = fdiv(f, a.fd_S), j = f - r * S, y = ND == 3 ? fdiv(j, a.fd_L) : 0;
        at[k] = r << 20 | y << 10 | (j - y * L);
    }
    f32x2 acc[NS][4];
#pragma unroll
    for (int k = 0; k < NS; ++k)
#pragma unroll
        for (int i = 0; i < 4; ++i) acc[k][i] = 0ull;
#pragma unroll 1
    for (int t = 0; t < T; ++t) {
        const int ds = ND == 3 ? t / 9 : t / 3, dy = ND == 3 ? (t / 3) % 3 - 1 : 0, dx = t % 3 - 1;
        int row[NS];
#pragma unroll
        for (int k = 0; k < NS; ++k)
            row[k] = (((at[k] >> 20) + ds) * S + (ND == 3 ? wrap(((at[k] >> 10) & 1023) + dy, L) * L : 0) +
                      wrap((at[k] & 1023) + dx, L)) * 4;
        const float* wt = W2 + t * C * C + co;
#pragma unroll 1
        for (int c4 = 0; c4 < C / 4; ++c4) {
            float4 hv[NS];
#pragma unroll
            for (int k = 0; k < NS; ++k) hv[k] = *reinterpret_cast<const float4*>(g_s + row[k] + c4 * pitch * 4);
#pragma unroll
            for (int cc = 0; cc < 4; ++cc) {
                f32x2 ww[4];
                load_w<8, false>(ww, wt + (4 * c4 + cc) * C);
#pragma unroll
                for (int k = 0; k < NS; ++k) {
                    const f32x2 h = f2_splat(cc == 0 ? hv[k].x : cc == 1 ? hv[k].y : cc == 2 ? hv[k].z : hv[k].w);
#pragma unroll
                    for (int i = 0; i < 4; ++i) acc[k][i] = f2_fma(h, ww[i], acc[k][i]);
                }
            }
        }
    }
#pragma unroll
    for (int k = 0; k < NS; ++k) {
        if (blk * (32 * NS) + lane + 32 * k >= nf) continue;
        const int n = (s0 + (at[k] >> 20)) * S + (ND == 3 ? ((at[k] >> 10) & 1023) * L : 0) + (at[k] & 1023);
        const int64_t o = ((b * (C / 4) + (co >> 2)) * a.V + n) * 4;
#pragma unroll
        for (int h = 0; h < 2; ++h) {
            const int64_t oh = o + (int64_t)h * a.V * 4;
            const float4 r = __ldg(reinterpret_cast<const float4*>(a.h1 + oh));
            float4 v = make_float4(f2_lo(acc[k][2 * h]), f2_hi(acc[k][2 * h]), f2_lo(acc[k][2 * h + 1]), f2_hi(acc[k][2 * h + 1]));
            v.x *= r.x > 0.f ? 1.f : a.slope; v.y *= r.y > 0.f ? 1.f : a.slope;
            v.z *= r.z > 0.f ? 1.f : a.slope; v.w *= r.w > 0.f ? 1.f : a.slope;
            *reinterpret_cast<float4*>(a.gh1 + oh) = v;
        }
    }
}

template <int ND, int C, int NS>
__global__ void __launch_bounds__(kBack2Threads, 2) k_back2(const __grid_constant__ BwdArgs a) {
    constexpr int T = ND == 3 ? 27 : 9;
    extern __shared__ __align__(16) float smf[];
    const int L = a.L, S = a.S, G = a.G, pitch = (G + 2) * S + 1, nh = (G + 2) * S, hS = S >> 1;
    float* W2 = smf;                             // [t][o][i]
    float* W3 = W2 + T * C * C;                  // [t][2][c]
    float* g_s = W3 + 2 * T * C;                 // gh2, [c4][pitch] float4
    float2* g3s = reinterpret_cast<float2*>(g_s + (C / 4) * pitch * 4);   // slices s0 - 2 .. s0 + G + 1
    for (int i = threadIdx.x * 4; i < T * C * C; i += kBack2Threads * 4) cp16(W2 + i, a.W2b + i);
    for (int i = threadIdx.x * 4; i < 2 * T * C; i += kBack2Threads * 4) cp16(W3 + i, a.W3b + i);
    const int per_cfg = L / G;
    for (int64_t u = blockIdx.x; u < a.B * per_cfg; u += gridDim.x) {
        const int64_t b = u / per_cfg;
        const int s0 = (int)(u - b * per_cfg) * G;
        __syncthreads();
        const float2* g3 = reinterpret_cast<const float2*>(a.g3) + b * a.V;
        for (int i = threadIdx.x; i < (G + 4) * S; i += kBack2Threads)
            g3s[i] = __ldg(g3 + wrap(wrap((s0 - 2) * S + i, a.V), a.V));
        cp_wait();
        __syncthreads();
        // gh2 of slices s0 - 1 .. s0 + G, 8 channels per item, sites ordered by
        // parity (the taps that reach updated sites agree in a warp)
        const int half = nh >> 1;
        for (int it = threadIdx.x; it < nh * (C / 8); it += kBack2Threads) {
            int g = 0, f = it;
#pragma unroll
            for (int k = 1; k < C / 8; ++k)
                if (f >= nh) { f -= nh; ++g; }
            const int q = f >= half ? 1 : 0;
            f -= q * half;
            const int r = fdiv(f, a.fd_Sh), jj = f - r * hS, sl = wrap(s0 - 1 + r, L);
            const int y = ND == 3 ? fdiv(jj, a.fd_Lh) : 0;
            const int xc = 2 * (jj - y * (L >> 1)) + ((q + sl + y) & 1);
            const int j = (ND == 3 ? y * L : 0) + xc, co = 8 * g;
            const int64_t o = ((b * (C / 4) + 2 * g) * a.V + sl * S + j) * 4;
            const float4 ra = __ldg(reinterpret_cast<const float4*>(a.h2 + o));
            const float4 rb = __ldg(reinterpret_cast<const float4*>(a.h2 + o + (int64_t)a.V * 4));
            f32x2 acc[4] = {0ull, 0ull, 0ull, 0ull};
            const bool even = q != a.frozen;     // taps of even offset parity reach updated sites
#pragma unroll
            for (int t = 0; t < T; ++t) {
                const int ds = ND == 3 ? t / 9 : t / 3, dy = ND == 3 ? (t / 3) % 3 : 1, dx = t % 3;
                if (((ds + dy + dx + 1) & 1) == (even ? 1 : 0)) continue;
                const float2 gv = g3s[(r + ds) * S + (ND == 3 ? wrap(y + dy - 1, L) * L : 0) + wrap(xc + dx - 1, L)];
                f32x2 w0[4], w1[4];
                load_w<8, false>(w0, W3 + (2 * t) * C + co);
                load_w<8, false>(w1, W3 + (2 * t + 1) * C + co);
#pragma unroll
                for (int i = 0; i < 4; ++i) acc[i] = f2_fma(f2_splat(gv.y), w1[i], f2_fma(f2_splat(gv.x), w0[i], acc[i]));
            }
            const float hr[8] = {ra.x, ra.y, ra.z, ra.w, rb.x, rb.y, rb.z, rb.w};
            float v[8];
#pragma unroll
            for (int i = 0; i < 8; ++i)
                v[i] = ((i & 1) ? f2_hi(acc[i >> 1]) : f2_lo(acc[i >> 1])) * (hr[i] > 0.f ? 1.f : a.slope);
            float* d = g_s + ((2 * g) * pitch + r * S + j) * 4;
            *reinterpret_cast<float4*>(d) = make_float4(v[0], v[1], v[2], v[3]);
            *reinterpret_cast<float4*>(d + pitch * 4) = make_float4(v[4], v[5], v[6], v[7]);
            if (r >= 1 && r <= G) {              // the unit's own slices
                *reinterpret_cast<float4*>(a.gh2 + o) = make_float4(v[0], v[1], v[2], v[3]);
                *reinterpret_cast<float4*>(a.gh2 + o + (int64_t)a.V * 4) = make_float4(v[4], v[5], v[6], v[7]);
            }
        }
        __syncthreads();
        const int tasks = ((G * S + 32 * NS - 1) / (32 * NS)) * (C / 8);
        for (int task = threadIdx.x >> 5; task < tasks; task += kBack2Threads / 32)
            back2_tile<ND, C, NS>(a, W2, g_s, pitch, task, b, s0);
    }
}

// ------------------------------------------------------------------ weight gradients
// The order in which a weight's gradient is summed decides its last bits, and
// through Adam's normalised steps those of the next iteration's loss, so it is
// fixed by the shape and the batch alone: min(B, two per SM) CTAs take every
// so-manieth unit of wgrad_G consecutive slices, each sum is one FMA chain (or
// the stated number of chains) over the CTA's units, rows and columns in order,
// and k_wgrad_reduce adds the CTAs' partials.  Terms with a zero factor (the
// field at updated sites, g3 at fixed ones) leave a chain as it is and are
// skipped.
inline int wgrad_parts(int64_t B) { return (int)std::min<int64_t>(B, (int64_t)num_sms() * 2); }
// The largest divisor of L whose `bytes` are within `limit`, else 1.
template <typename F>
int wgrad_G(int L, size_t limit, F bytes) {
    int G = L;
    while (G > 1 && (bytes(G) > limit || L % G != 0)) --G;
    return G;
}

// ------------------------------------------------------------------ k_wgrad2
// dW2[t][i][o] = sum_n h1(n + delta(t))[i] gh2(n)[o], a GEMM over the sites; one
// chain per sum (2D C = 32: k_wgrad2_c32 below).  A thread holds the three
// x-taps of one (dz, dy) row offset, 2 input and OB output channels.  Walking a
// row along x, each h1 value is loaded and paired once and feeds three taps:
// per site one 8-byte and OB / 4 16-byte loads feed 3 OB packed FMAs.  Bound by
// the FP32 pipe for large batches, by the length of the chains for small ones,
// whose CTAs are split by row offset (gridDim.y).
inline int wgrad2_G(int L, int S, int C) {
    if (C == 32) return wgrad_G(L, 100 * 1024, [&](int g) { return (size_t)(2 * g + 2) * S * 36 * 4; });
    return wgrad_G(L, 96 * 1024, [&](int g) { return (size_t)(2 * g + 2) * S * C * 4; });
}
template <int ND, int C>
struct Wg2 {
    static constexpr int OB = ND == 3 && C >= 24 ? 8 : 4;
    static constexpr int TASKS = (ND == 3 ? 9 : 3) * (C / 2) * (C / OB), THREADS = (TASKS + 31) / 32 * 32;
    static size_t smem(int S, int G) { return (size_t)(C / 4) * (((G + 2) * S | 1) + (G * S | 1)) * 16; }
};

template <int ND, int C>
__global__ void __launch_bounds__(Wg2<ND, C>::THREADS, ND == 2 ? 2 : 1) k_wgrad2(const __grid_constant__ BwdArgs a) {
    constexpr int T = ND == 3 ? 27 : 9, OB = Wg2<ND, C>::OB, OP = OB / 2;
    extern __shared__ __align__(16) float smf[];
    const int L = a.L, S = a.S, G = a.G, px = (G + 2) * S | 1, pg = G * S | 1;   // odd: chunks on distinct banks
    const int per_part = Wg2<ND, C>::TASKS / gridDim.y;
    const bool active = (int)threadIdx.x < per_part;
    const int task = active ? (int)(blockIdx.y * per_part + threadIdx.x) : 0;
    const int og = task % (C / OB), ig = (task / (C / OB)) % (C / 2), nr = task / ((C / OB) * (C / 2));
    const int ds = ND == 3 ? nr / 3 : nr, dy = ND == 3 ? nr % 3 - 1 : 0;
    f32x2 acc[3][2][OP], accb[OP];               // [dx][input][output pair], bias
#pragma unroll
    for (int j = 0; j < OP; ++j) {
        accb[j] = 0ull;
#pragma unroll
        for (int d = 0; d < 6; ++d) acc[d / 2][d % 2][j] = 0ull;
    }
    const bool bias = active && nr == 0 && ig == 0;
    const f32x2 one = f2_splat(1.f);
    const int per_cfg = L / G, rows = G * (ND == 3 ? L : 1);
    const float* xs = smf + (ig >> 1) * px * 4 + (ig & 1) * 2;
    float* const g_s = smf + (C / 4) * px * 4;
    const float* gs = g_s + (OB / 4) * og * pg * 4;
    for (int64_t u = blockIdx.x; u < a.B * per_cfg; u += gridDim.x) {
        const int64_t b = u / per_cfg;
        const int s0 = (int)(u - b * per_cfg) * G;
        __syncthreads();
        stage_slab<C>(g_s, pg, a.gh2, a, b, s0, 0);
        stage_slab<C>(smf, px, a.h1, a, b, s0, 1);
        cp_wait();
        __syncthreads();
        if (!active) continue;
        for (int r = 0; r < rows; ++r) {
            const int rs = ND == 3 ? fdiv(r, a.fd_L) : r, y = ND == 3 ? r - rs * L : 0;
            const float* xr = xs + ((rs + ds) * S + (ND == 3 ? wrap(y + dy, L) * L : 0)) * 4;
            const float* gr = gs + (rs * S + y * L) * 4;
            f32x2 w0[2], w1[2], w2[2], w3[2];    // four columns of the window
            const auto load = [&](f32x2 (&w)[2], int x) {
                const float2 v = *reinterpret_cast<const float2*>(xr + x * 4);
                w[0] = f2_splat(v.x);
                w[1] = f2_splat(v.y);
            };
            load(w0, L - 1);
            load(w1, 0);
            const auto site = [&](int x, const f32x2 (&wm)[2], const f32x2 (&wc)[2], const f32x2 (&wp)[2]) {
                f32x2 gv[OP];
#pragma unroll
                for (int q = 0; q < OB / 4; ++q) {
                    const ulonglong2 g = *reinterpret_cast<const ulonglong2*>(gr + (q * pg + x) * 4);
                    gv[2 * q] = g.x;
                    gv[2 * q + 1] = g.y;
                }
#pragma unroll
                for (int i = 0; i < 2; ++i)
#pragma unroll
                    for (int j = 0; j < OP; ++j) {
                        acc[0][i][j] = f2_fma(wm[i], gv[j], acc[0][i][j]);
                        acc[1][i][j] = f2_fma(wc[i], gv[j], acc[1][i][j]);
                        acc[2][i][j] = f2_fma(wp[i], gv[j], acc[2][i][j]);
                    }
                if (bias)
#pragma unroll
                    for (int j = 0; j < OP; ++j) accb[j] = f2_fma(one, gv[j], accb[j]);
            };
            // columns x, x + 1 (L is even); the window moves by naming
            const auto two = [&](int x, f32x2 (&a0)[2], f32x2 (&a1)[2], f32x2 (&a2)[2], f32x2 (&a3)[2]) {
                load(a2, x + 1);
                load(a3, x + 2 == L ? 0 : x + 2);
                site(x, a0, a1, a2);
                site(x + 1, a1, a2, a3);
            };
            int x = 0;
#pragma unroll 1
            for (; x + 4 <= L; x += 4) {
                two(x, w0, w1, w2, w3);
                two(x + 2, w2, w3, w0, w1);
            }
            if (x < L) two(x, w0, w1, w2, w3);
        }
    }
    if (!active) return;
    // one partial per CTA
    float* P = a.partial + (int64_t)blockIdx.x * (T + 1) * C * C + OB * og;
#pragma unroll
    for (int d = 0; d < 3; ++d)
#pragma unroll
        for (int i = 0; i < 2; ++i)
#pragma unroll
            for (int j = 0; j < OP; ++j)
                *reinterpret_cast<f32x2*>(P + ((3 * nr + d) * C + 2 * ig + i) * C + 2 * j) = acc[d][i][j];
    if (bias)
#pragma unroll
        for (int j = 0; j < OP; ++j) *reinterpret_cast<f32x2*>(P + T * C * C + 2 * j) = accb[j];
}

// 2D, C = 32 (the training workload's flow): two chains per sum, over the even
// and the odd columns of every row, added at the end.  Each thread owns an 8 x 8
// tile (8 input channels of one tap x 8 output channels) and one column parity:
// per site two 16-byte loads each of h1 and gh2 (row pitch 36 floats) feed 64
// multiply-adds.  0.61 ms at batch 1024 (32 TFLOP/s).  Packed FMAs over output
// pairs (0.74 to 0.80 ms: an instruction and a register pair per h1 value), over
// the two column parities (0.86 ms) and staging by asynchronous copies with a
// tenth, idle warp to even out the schedulers (0.74 ms) were slower.
constexpr int kWg2c32Threads = 288;
inline size_t wg2c32_smem(int S, int G) {
    return std::max((size_t)((2 * G + 2) * S) * 36 * 4, (size_t)144 * 72 * 4);
}

template <int ND>
__global__ void __launch_bounds__(kWg2c32Threads, 2) k_wgrad2_c32(const __grid_constant__ BwdArgs a) {
    constexpr int T = 9, C = 32, P = 36, TILES = T * 4 * 4;   // (tap, input group) x output group
    static_assert(ND == 2, "two chains per sum in 2D only");
    extern __shared__ __align__(16) float smf[];
    const int L = a.L, V = a.V, G = a.G;
    const int half = threadIdx.x / TILES, r = threadIdx.x % TILES;
    const int og = r & 3, ig = (r >> 2) & 3, t = r >> 4, ds = t / 3, dx = t % 3 - 1;
    float* x_s = smf;                            // [(G+2) L][P]
    float* g_s = smf + (size_t)(G + 2) * L * P;  // [G L][P]
    float acc[8][8], accb[8];
#pragma unroll
    for (int j = 0; j < 8; ++j) {
        accb[j] = 0.f;
#pragma unroll
        for (int i = 0; i < 8; ++i) acc[i][j] = 0.f;
    }
    const bool bias = t == 0 && ig == 0;
    const int per_cfg = L / G;
    for (int64_t u = blockIdx.x; u < a.B * per_cfg; u += gridDim.x) {
        const int64_t b = u / per_cfg;
        const int s0 = (int)(u - b * per_cfg) * G;
        __syncthreads();
        const int nsx = (G + 2) * L, nsg = G * L;
        for (int e = threadIdx.x; e < nsx * 8; e += blockDim.x) {
            const int c4 = e / nsx, site = e % nsx;
            *reinterpret_cast<float4*>(x_s + (size_t)site * P + 4 * c4) = __ldg(reinterpret_cast<const float4*>(
                a.h1 + ((b * 8 + c4) * (int64_t)V + wrap((s0 - 1) * L + site, V)) * 4));
        }
        for (int e = threadIdx.x; e < nsg * 8; e += blockDim.x) {
            const int c4 = e / nsg, site = e % nsg;
            *reinterpret_cast<float4*>(g_s + (size_t)site * P + 4 * c4) =
                __ldg(reinterpret_cast<const float4*>(a.gh2 + ((b * 8 + c4) * (int64_t)V + s0 * L + site) * 4));
        }
        __syncthreads();
        for (int rs = 0; rs < G; ++rs) {
            const int in_row = (rs + ds) * L, g_row = rs * L;
            for (int x = half; x < L; x += 2) {
                const float* ap = x_s + (size_t)(in_row + wrap(x + dx, L)) * P + ig * 8;
                const float* bp = g_s + (size_t)(g_row + x) * P + og * 8;
                const float4 a0 = *reinterpret_cast<const float4*>(ap);
                const float4 a1 = *reinterpret_cast<const float4*>(ap + 4);
                const float4 b0 = *reinterpret_cast<const float4*>(bp);
                const float4 b1 = *reinterpret_cast<const float4*>(bp + 4);
                const float av[8] = {a0.x, a0.y, a0.z, a0.w, a1.x, a1.y, a1.z, a1.w};
                const float bv[8] = {b0.x, b0.y, b0.z, b0.w, b1.x, b1.y, b1.z, b1.w};
#pragma unroll
                for (int i = 0; i < 8; ++i)
#pragma unroll
                    for (int o = 0; o < 8; ++o) acc[i][o] = fmaf(av[i], bv[o], acc[i][o]);
                if (bias)
#pragma unroll
                    for (int o = 0; o < 8; ++o) accb[o] += bv[o];
            }
        }
    }
    // the halves' sums through shared memory, then one partial per CTA
    __syncthreads();
    float* red = smf;                            // [TILES][72]
    if (half == 1) {
#pragma unroll
        for (int i = 0; i < 8; ++i)
#pragma unroll
            for (int o = 0; o < 8; ++o) red[(size_t)r * 72 + i * 8 + o] = acc[i][o];
#pragma unroll
        for (int o = 0; o < 8; ++o) red[(size_t)r * 72 + 64 + o] = accb[o];
    }
    __syncthreads();
    if (half != 0) return;
    float* Pt = a.partial + (int64_t)blockIdx.x * (T + 1) * C * C + og * 8;
#pragma unroll
    for (int i = 0; i < 8; ++i)
#pragma unroll
        for (int o = 0; o < 8; ++o) Pt[(t * C + ig * 8 + i) * C + o] = acc[i][o] + red[(size_t)r * 72 + i * 8 + o];
    if (bias)
#pragma unroll
        for (int o = 0; o < 8; ++o) Pt[T * C * C + o] = accb[o] + red[(size_t)r * 72 + 64 + o];
}

// ------------------------------------------------------------------ k_back1
// Both uses of gh1 from one staging of it: gx += conv1^T(gh1) at the fixed
// sites (one thread per site, one chain over taps and channels) and dW1, db1
// (thread = channel and row group, a sliding window over x of the field at the
// fixed sites; the groups' sums are added in order).  Bound by reading gh1 and
// by the shared-memory reads.
constexpr int kThinThreads = 512;                // row groups: kThinThreads / C

template <int ND, int C>
struct Back1 {
    static constexpr int T = ND == 3 ? 27 : 9, GRP = kThinThreads / C;
    static int G(int L, int S) {
        return wgrad_G(L, 112 * 1024, [&](int g) { return (size_t)(g * S * (C + 4) + (g + 2) * S) * 4; });
    }
    // the row groups' sums reuse the staged gh1
    static size_t smem(int S, int G) {
        return ((size_t)std::max((C / 4) * ((G + 2) * S | 1) * 4, GRP * C * (T + 1)) + T * C + (G + 2) * S) * 4;
    }
};

template <int ND, int C>
__global__ void __launch_bounds__(kThinThreads) k_back1(const __grid_constant__ BwdArgs a) {
    constexpr int T = ND == 3 ? 27 : 9, NR = T / 3, GRP = kThinThreads / C;
    extern __shared__ __align__(16) float smf[];
    const int L = a.L, S = a.S, G = a.G, pitch = (G + 2) * S | 1, hS = S >> 1;
    const int nst = (C / 4) * pitch * 4;
    float* g_s = smf;                            // gh1, [c4][pitch] float4; at the end [GRP][T + 1][C]
    float* W1 = smf + (nst > GRP * C * (T + 1) ? nst : GRP * C * (T + 1));   // [t][c]
    float* x_s = W1 + T * C;                     // the field at the fixed sites, slices s0 - 1 .. s0 + G
    for (int i = threadIdx.x; i < T * C; i += kThinThreads) W1[i] = __ldg(a.W1b + i);
    const int ch = threadIdx.x % C, grp = threadIdx.x / C;
    float acc[T + 1];
#pragma unroll
    for (int t = 0; t <= T; ++t) acc[t] = 0.f;
    const int per_cfg = L / G, rps = ND == 3 ? L : 1;
    for (int64_t u = blockIdx.x; u < a.B * per_cfg; u += gridDim.x) {
        const int64_t b = u / per_cfg;
        const int s0 = (int)(u - b * per_cfg) * G;
        __syncthreads();
        stage_slab<C>(g_s, pitch, a.gh1, a, b, s0, 1);
        for (int i = threadIdx.x; i < (G + 2) * S; i += kThinThreads) {
            const int n = wrap((s0 - 1) * S + i, a.V), sl = fdiv(n, a.fd_S), j = n - sl * S;
            const int y = ND == 3 ? fdiv(j, a.fd_L) : 0;
            x_s[i] = ((sl + y + (j - y * L)) & 1) == a.frozen ? __ldg(a.xl + b * a.V + n) : 0.f;
        }
        cp_wait();
        __syncthreads();
        // gx at the unit's fixed sites
        for (int it = threadIdx.x; it < G * hS; it += kThinThreads) {
            const int r = fdiv(it, a.fd_Sh), jj = it - r * hS, sl = s0 + r;
            const int y = ND == 3 ? fdiv(jj, a.fd_Lh) : 0;
            const int xc = 2 * (jj - y * (L >> 1)) + ((a.frozen + sl + y) & 1);
            float v = 0.f;
#pragma unroll 1
            for (int k = 0; k < NR; ++k) {
                const int ds = ND == 3 ? k / 3 : k, dy = ND == 3 ? k % 3 - 1 : 0;
                const int row = (r + ds) * S + (ND == 3 ? wrap(y + dy, L) * L : 0);
#pragma unroll
                for (int dx = 0; dx < 3; ++dx) {
                    const float* p = g_s + (row + wrap(xc + dx - 1, L)) * 4;
                    const float* wt = W1 + (3 * k + dx) * C;
#pragma unroll
                    for (int c4 = 0; c4 < C / 4; ++c4) {
                        const float4 h = *reinterpret_cast<const float4*>(p + c4 * pitch * 4);
                        const float4 w = *reinterpret_cast<const float4*>(wt + 4 * c4);
                        v = fmaf(h.x, w.x, v); v = fmaf(h.y, w.y, v);
                        v = fmaf(h.z, w.z, v); v = fmaf(h.w, w.w, v);
                    }
                }
            }
            a.gx[b * a.V + sl * S + (ND == 3 ? y * L : 0) + xc] += v;
        }
        // dW1, db1
        if (grp < GRP) {
            const float* gc = g_s + (ch >> 2) * pitch * 4 + (ch & 3);
            for (int row = grp; row < G * rps; row += GRP) {
                const int rs = ND == 3 ? fdiv(row, a.fd_L) : row, y = ND == 3 ? row - rs * L : 0;
                int base[NR];
#pragma unroll
                for (int k = 0; k < NR; ++k)
                    base[k] = (rs + (ND == 3 ? k / 3 : k)) * S + (ND == 3 ? wrap(y + k % 3 - 1, L) * L : 0);
                const int gb = (rs + 1) * S + y * L;
                float wm[NR], w0[NR];
#pragma unroll
                for (int k = 0; k < NR; ++k) {
                    wm[k] = x_s[base[k] + L - 1];
                    w0[k] = x_s[base[k]];
                }
                for (int x = 0; x < L; ++x) {
                    const int xp = x + 1 == L ? 0 : x + 1;
                    const float g = gc[(gb + x) * 4];
#pragma unroll
                    for (int k = 0; k < NR; ++k) {
                        const float wp = x_s[base[k] + xp];
                        acc[3 * k] = fmaf(wm[k], g, acc[3 * k]);
                        acc[3 * k + 1] = fmaf(w0[k], g, acc[3 * k + 1]);
                        acc[3 * k + 2] = fmaf(wp, g, acc[3 * k + 2]);
                        wm[k] = w0[k];
                        w0[k] = wp;
                    }
                    acc[T] += g;
                }
            }
        }
    }
    __syncthreads();
    if (grp < GRP)
#pragma unroll
        for (int t = 0; t <= T; ++t) g_s[(grp * (T + 1) + t) * C + ch] = acc[t];
    __syncthreads();
    float* P = a.partial + (int64_t)blockIdx.x * (T + 1) * C;
    for (int e = threadIdx.x; e < (T + 1) * C; e += kThinThreads) {
        float sum = 0.f;
        for (int g = 0; g < GRP; ++g) sum += g_s[g * (T + 1) * C + e];
        P[e] = sum;
    }
}

// ------------------------------------------------------------------ k_wgrad3
// dW3[t][i][.] = sum over the updated sites of h2(n + delta(t))[i] g3(n)[.], the
// pair (s, t) packed.  Thread = input channel and row group; it walks the
// updated sites of a row (every other one) with a window of three columns; the
// groups' sums are added in order.
template <int ND, int C>
struct Wgrad3 {
    static constexpr int T = ND == 3 ? 27 : 9, GRP = kThinThreads / C;
    static int G(int L, int S) {
        return wgrad_G(L, 112 * 1024, [&](int g) { return (size_t)(g * S * 2 + (g + 2) * S * (C + 4)) * 4; });
    }
    static size_t smem(int S, int G) {
        return std::max((size_t)(C / 4) * ((G + 2) * S | 1) * 16 + (size_t)G * S * 8, (size_t)GRP * C * (T + 1) * 8);
    }
};

template <int ND, int C>
__global__ void __launch_bounds__(kThinThreads) k_wgrad3(const __grid_constant__ BwdArgs a) {
    constexpr int T = ND == 3 ? 27 : 9, NR = T / 3, GRP = kThinThreads / C;
    extern __shared__ __align__(16) float smf[];
    const int L = a.L, S = a.S, G = a.G, pitch = (G + 2) * S | 1;
    float* h_s = smf;                            // h2, [c4][pitch] float4
    f32x2* g_s = reinterpret_cast<f32x2*>(h_s + (C / 4) * pitch * 4);
    f32x2* red = reinterpret_cast<f32x2*>(smf);  // [GRP][T + 1][C], after the units
    const int ch = threadIdx.x % C, grp = threadIdx.x / C;
    f32x2 acc[T + 1];
#pragma unroll
    for (int t = 0; t <= T; ++t) acc[t] = 0ull;
    const f32x2 one = f2_splat(1.f);
    const int per_cfg = L / G, rps = ND == 3 ? L : 1;
    for (int64_t u = blockIdx.x; u < a.B * per_cfg; u += gridDim.x) {
        const int64_t b = u / per_cfg;
        const int s0 = (int)(u - b * per_cfg) * G;
        __syncthreads();
        stage_slab<C>(h_s, pitch, a.h2, a, b, s0, 1);
        const f32x2* g3 = reinterpret_cast<const f32x2*>(a.g3) + b * a.V + s0 * S;
        for (int i = threadIdx.x; i < G * S; i += kThinThreads) g_s[i] = __ldg(g3 + i);
        cp_wait();
        __syncthreads();
        if (grp >= GRP) continue;
        const float* hc = h_s + (ch >> 2) * pitch * 4 + (ch & 3);
        for (int row = grp; row < G * rps; row += GRP) {
            const int rs = ND == 3 ? fdiv(row, a.fd_L) : row, y = ND == 3 ? row - rs * L : 0;
            const float* base[NR];
#pragma unroll
            for (int k = 0; k < NR; ++k)
                base[k] = hc + ((rs + (ND == 3 ? k / 3 : k)) * S + (ND == 3 ? wrap(y + k % 3 - 1, L) * L : 0)) * 4;
            const f32x2* gr = g_s + rs * S + y * L;
            const int x0 = (a.frozen + 1 + s0 + rs + y) & 1;             // the row's first updated site
            float left[NR];
#pragma unroll
            for (int k = 0; k < NR; ++k) left[k] = base[k][(x0 == 0 ? L - 1 : 0) * 4];
            for (int x = x0; x < L; x += 2) {
                const int xp = x + 1 == L ? 0 : x + 1;
                const f32x2 g = gr[x];
#pragma unroll
                for (int k = 0; k < NR; ++k) {
                    const float mid = base[k][x * 4], right = base[k][xp * 4];
                    acc[3 * k] = f2_fma(f2_splat(left[k]), g, acc[3 * k]);
                    acc[3 * k + 1] = f2_fma(f2_splat(mid), g, acc[3 * k + 1]);
                    acc[3 * k + 2] = f2_fma(f2_splat(right), g, acc[3 * k + 2]);
                    left[k] = right;
                }
                if (ch == 0) acc[T] = f2_fma(one, g, acc[T]);
            }
        }
    }
    __syncthreads();
    if (grp < GRP)
#pragma unroll
        for (int t = 0; t <= T; ++t) red[(grp * (T + 1) + t) * C + ch] = acc[t];
    __syncthreads();
    f32x2* P = reinterpret_cast<f32x2*>(a.partial) + (int64_t)blockIdx.x * (T + 1) * C;
    for (int e = threadIdx.x; e < (T + 1) * C; e += kThinThreads) {
        f32x2 sum = 0ull;
        for (int g = 0; g < GRP; ++g) sum = f2_fma(one, red[g * (T + 1) * C + e], sum);
        P[e] = sum;
    }
}

// Slices per unit: the largest divisor of L whose units fit `fits` and number
// at least `want` (else the largest number of units that fits).
template <typename Fits>
int pick_G(int L, int64_t B, int64_t want, Fits fits) {
    int best = 0;
    for (int g = L; g >= 1; --g) {
        if (L % g || !fits(g)) continue;
        best = g;
        if (B * (L / g) >= want) break;
    }
    return best;                                 // 0: not even one slice fits
}

// Launches of one layer's reverse pass; all but back2 write wgrad_parts partials.
struct BwdOps {
    gf_status (*back2)(BwdArgs, cudaStream_t);
    gf_status (*wgrad2)(BwdArgs, cudaStream_t);
    gf_status (*back1)(BwdArgs, cudaStream_t);
    gf_status (*wgrad3)(BwdArgs, cudaStream_t);
};
BwdOps ops_2d(int C);       // gf_train_bwd_2d.cu
BwdOps ops_3d(int C);       // gf_train_bwd_3d.cu

template <typename K>
bool allow(K kern) {
    return cudaFuncSetAttribute(kern, cudaFuncAttributeMaxDynamicSharedMemorySize, kBudget) == cudaSuccess;
}

template <int ND, int C, int NS>
gf_status launch_back2_ns(BwdArgs a, cudaStream_t st) {
    if (!allow(k_back2<ND, C, NS>)) return GF_ECUDA;
    const size_t smem = back2_smem<ND, C>(a.S, a.G);
    const int per_sm = 2 * (smem + 1024) <= 228 * 1024 ? 2 : 1;
    const int64_t grid = std::min<int64_t>(a.B * (a.L / a.G), (int64_t)num_sms() * per_sm);
    k_back2<ND, C, NS><<<(unsigned)grid, kBack2Threads, smem, st>>>(a);
    GF_CHECK_LAUNCH();
    return GF_OK;
}
template <int ND, int C>
gf_status launch_back2(BwdArgs a, cudaStream_t st) {
    const int64_t sms = num_sms();
    // two CTAs per SM and at least as many units, else one
    a.G = pick_G(a.L, a.B, 2 * sms, [&](int g) { return 2 * (back2_smem<ND, C>(a.S, g) + 1024) <= 228 * 1024; });
    if (a.G == 0) a.G = pick_G(a.L, a.B, sms, [&](int g) { return back2_smem<ND, C>(a.S, g) <= (size_t)kBudget; });
    if (a.G == 0) return GF_EUNSUPPORTED;
    // tile: 4 sites per lane when that gives every warp one, else fewer
    const int nf = a.G * a.S, groups = C / 8;
    if ((nf + 127) / 128 * groups >= 8) return launch_back2_ns<ND, C, 4>(a, st);
    if ((nf + 63) / 64 * groups >= 8) return launch_back2_ns<ND, C, 2>(a, st);
    return launch_back2_ns<ND, C, 1>(a, st);
}
template <int ND, int C>
gf_status launch_wgrad2(BwdArgs a, cudaStream_t st) {
    a.G = wgrad2_G(a.L, a.S, C);
    const int64_t np = wgrad_parts(a.B), sms = num_sms();
    if constexpr (ND == 2 && C == 32) {
        const size_t smem = wg2c32_smem(a.S, a.G);
        if (smem > (size_t)kBudget) return GF_EUNSUPPORTED;
        if (!allow(k_wgrad2_c32<ND>)) return GF_ECUDA;
        k_wgrad2_c32<ND><<<(unsigned)np, kWg2c32Threads, smem, st>>>(a);
    } else {
        using P = Wg2<ND, C>;
        const size_t smem = P::smem(a.S, a.G);
        if (smem > (size_t)kBudget) return GF_EUNSUPPORTED;
        // batches that leave SMs idle: more, smaller CTAs (each stages the unit)
        const int parts = ND == 3 && 9 * np <= 2 * sms ? 9 : np <= sms ? 3 : 1;
        if (!allow(k_wgrad2<ND, C>)) return GF_ECUDA;
        k_wgrad2<ND, C><<<dim3((unsigned)np, (unsigned)parts), (P::TASKS / parts + 31) / 32 * 32, smem, st>>>(a);
    }
    GF_CHECK_LAUNCH();
    return GF_OK;
}
// k_back1 and k_wgrad3: Plan gives their G and shared memory.
template <typename Plan, typename K>
gf_status launch_thin(K kern, BwdArgs a, cudaStream_t st) {
    a.G = Plan::G(a.L, a.S);
    const size_t smem = Plan::smem(a.S, a.G);
    if (smem > (size_t)kBudget) return GF_EUNSUPPORTED;
    if (!allow(kern)) return GF_ECUDA;
    kern<<<wgrad_parts(a.B), kThinThreads, smem, st>>>(a);
    GF_CHECK_LAUNCH();
    return GF_OK;
}
template <int ND, int C>
gf_status launch_back1(BwdArgs a, cudaStream_t st) {
    return launch_thin<Back1<ND, C>>(k_back1<ND, C>, a, st);
}
template <int ND, int C>
gf_status launch_wgrad3(BwdArgs a, cudaStream_t st) {
    return launch_thin<Wgrad3<ND, C>>(k_wgrad3<ND, C>, a, st);
}
template <int ND, int C>
constexpr BwdOps make_ops() { return {launch_back2<ND, C>, launch_wgrad2<ND, C>, launch_back1<ND, C>, launch_wgrad3<ND, C>}; }

}  // namespace bwd
}  // namespace gf
