// gf_flow_fp32_kernel.cuh -- fused FP32 coupling-stack kernel (both
// directions) for two equal hidden widths C in {8, 16, 24, 32}, kernel size 3.
//
// Paper (arXiv:2208.08903) Sec. 1: prior sample, even/odd affine coupling
// layers x -> x*exp(s) + t with (s, t) a convolutional net of the fixed
// sites, composition of N_tri layers, Jacobian via the sum of s, model density
// log q = log r - log|det|, and the phi^4 action for log w = -S - log q.
//
// One CTA owns one configuration at a time (persistent grid-stride loop): the
// field x stays in shared memory through every layer, the hidden activations
// h1 / h2 live in a slot cache of slices (see gf_flow.cuh), channel-chunk
// major ([slot][C/4][site][4]: consecutive sites of one chunk are consecutive
// 16-byte words, so a warp's loads of 32 consecutive sites have no bank
// conflict for any C).  The kernel is bound by the FP32 pipe: conv2 is 85 % to
// 95 % of the FLOPs.  A warp's conv2 tile is 32 NS sites x CO channels (lane =
// site), accumulated as packed FP32 pairs of output channels (fma.rn.f32x2:
// half the issue slots); per input channel NS site values and CO weights
// (broadcast reads) feed NS CO multiply-adds, so at 4 x 8 and above the
// shared-memory reads take less time than the FMAs.  Weights never come from
// global memory inside the loops: a layer's W2 is staged through two buffers of
// whole taps by asynchronous copies, one buffer ahead, the other weights of a
// layer beside it.  Small lattices take several CTAs per SM or, when the batch
// leaves SMs idle, tiles of one site and two or four channels per lane.
//
// Measured against a kernel of 256 threads with scalar 4 x 8 tiles, weights read
// from global memory and the phase headers fetched one by one: 3D L=12 width
// 32, 16 couplings, batch 300: 42.7 -> 14.8 ms (32 TFLOP/s; issue slots 50 %
// active, the FMA pipe about 40 %); 2D L=64 width 32: 20.4 -> 40.5 TFLOP/s; 2D L=8 width 8, 64
// configurations: 100 -> 59 us, 16,384: 4.2 -> 12.9 TFLOP/s.  One kernel per
// tile: with the tile chosen inside one kernel the accumulators were spilled
// around every weight stage (41 ms).
//
// Sums: every output of a convolution is one FMA chain in tap and channel
// order from the bias (the same results for every tile and thread count); the
// head sums as described at head_split.  The log-det, sum z^2 and the action
// are FP32 pairs (gf_common.cuh) added as by 256 threads, whatever the CTA's
// size (order_sum): results depend on the shape alone.  Training's forward pass
// and recompute are instantiations of their own (kForward, kRecompute); its
// log-det is an FP64 sum (train_logdet).
#pragma once

#include "gf_f32x2.cuh"
#include "gf_flow.cuh"

namespace gf {
namespace f32k {

// What a kernel does: the flow in either direction; training's forward pass, which
// saves the field after every layer and the log-det; training's recompute of one
// layer (h1_out, h2_out, s_out), which does nothing else.
constexpr int kFlow = 0, kForward = 1, kRecompute = 2;

constexpr int kVT = 256;                   // threads of the sums' order; a CTA thread stands for up to 4

struct FlowArgs {
    const float* W;            // packed weights
    const Phase* sched;
    int n_phases, n_passes;    // n_passes: conv2 passes of one layer
    int64_t stride;
    PackedOffsets off;
    int L, S, V, layer0, n_layers, R;
    int stage_taps, n_stages;  // taps of W2 per staging buffer
    int two_small;             // second buffer for the layer's other weights
    int head_G, head_zb, head_a, head_b, head_train;   // see HeadSplit
    FastDiv fd_S, fd_L, fd_Sh, fd_Lh;
    float slope;
    int use_tanh, has_phi4;
    FF c2d_ff, lam_ff;         // 2 nd + m2 and lam as FP32 pairs
    int64_t B;
    uint64_t seed, counter0;
    const float* z_in;
    float* z_out;
    const float* phi_in;
    float* phi_out;
    double* logq_out;
    double* S_out;
    double* logw_out;
    float* xs_out;             // training: the field after l layers at xs_out + l xs_stride + b V
    int64_t xs_stride;
    double* logdet_out;
    // training's recompute of layer layer0 from its input (z_in), all three set:
    // h1, h2 [B][C/4][V][4] and s [B][V] at the updated sites; nothing else
    float* h1_out;
    float* h2_out;
    float* s_out;
    int off_h1, off_h2, off_small, off_w2, off_red, off_s, off_sched;   // shared memory (floats)
};

// conv2 tiles (sites per lane, output channels); the last is also the one of
// the kernels that read their weights from global memory.  (16 channels per
// tile need fewer loads per FMA but ran 5 % to 15 % slower at every shape.)
constexpr int kTiles = kF32Tiles;
constexpr int kTileNS[kTiles] = {1, 1, 2, 3, 5, 4};
constexpr int kTileCO[kTiles] = {2, 4, 8, 8, 8, 8};
constexpr int kTileGW = kTiles - 1;
// Tiles of two channels are never the cheapest above width 8.
constexpr int tile_first(int C) { return C > 8 ? 1 : 0; }

__device__ __forceinline__ int wrap(int v, int L) { return v < 0 ? v + L : (v >= L ? v - L : v); }
__device__ __forceinline__ float lrelu(float v, float a) { return v > 0.f ? v : a * v; }

// Weight reads: shared memory, or (GW, shapes whose activations leave no room
// for staged weights) global memory through the read-only path.
template <bool GW>
__device__ __forceinline__ ulonglong2 ldw2(const float* p) {
    if (GW) return __ldg(reinterpret_cast<const ulonglong2*>(p));
    return *reinterpret_cast<const ulonglong2*>(p);
}
template <bool GW>
__device__ __forceinline__ f32x2 ldw1(const float* p) {
    if (GW) return __ldg(reinterpret_cast<const unsigned long long*>(p));
    return *reinterpret_cast<const f32x2*>(p);
}
// acc[0 .. N/2) += splat(h) * w[0 .. N)
template <int N, bool GW>
__device__ __forceinline__ void load_w(f32x2 (&w)[N / 2], const float* p) {
    if constexpr (N == 2) {
        w[0] = ldw1<GW>(p);
    } else {
#pragma unroll
        for (int i = 0; i < N / 4; ++i) {
            const ulonglong2 u = ldw2<GW>(p + 4 * i);
            w[2 * i] = u.x;
            w[2 * i + 1] = u.y;
        }
    }
}

__device__ __forceinline__ void cp16(float* dst, const float* src) {
    asm volatile("cp.async.cg.shared.global [%0], [%1], 16;"
                 :: "r"(static_cast<uint32_t>(__cvta_generic_to_shared(dst))), "l"(src) : "memory");
}
__device__ __forceinline__ void cp_wait() { asm volatile("cp.async.wait_all;" ::: "memory"); }
__device__ __forceinline__ void cp_copy(float* dst, const float* src, int n) {
    for (int i = threadIdx.x * 4; i < n; i += blockDim.x * 4) cp16(dst + i, src + i);
}

// The staged weights: two buffers of stage_taps taps of W2, filled one ahead
// in the order the conv2 passes use them (a layer that fits one buffer is
// loaded once), and the layer's W1, b1 | b2, W3, b3.
template <int ND, int C, bool GW>
struct Weights {
    static constexpr int T = ND == 3 ? 27 : 9;
    static constexpr int kS1 = T * C + C, kS2 = C + 2 * T * C + 4, kSmall = kS1 + kS2;
    const FlowArgs& a;
    float* sm;
    int64_t left;              // layer applications after the current one
    int l, lnext;              // current and next layer
    int buf, sbuf;             // current W2 buffer and small buffer
    int passes;                // conv2 passes of this layer not yet begun
    bool first;                // no conv2 stage of this layer has begun

    __device__ const float* layer(int i) const { return a.W + (size_t)i * a.stride; }
    __device__ float* small_buf(int s) const { return sm + a.off_small + (a.two_small ? s * kSmall : 0); }
    __device__ float* w2_buf(int s) const { return sm + a.off_w2 + s * a.stage_taps * C * C; }
    __device__ void load_small(int s, int i) const {
        cp_copy(small_buf(s), layer(i), kS1);
        cp_copy(small_buf(s) + kS1, layer(i) + a.off.b2, kS2);
    }
    __device__ void load_w2(int s, int i, int st) const {
        const int t0 = st * a.stage_taps, t1 = min(T, t0 + a.stage_taps);
        cp_copy(w2_buf(s), layer(i) + a.off.W2 + (size_t)t0 * C * C, (t1 - t0) * C * C);
    }
    __device__ const float* W1() const { return GW ? layer(l) : small_buf(sbuf); }
    __device__ const float* b1() const { return W1() + T * C; }
    __device__ const float* b2() const { return GW ? layer(l) + a.off.b2 : small_buf(sbuf) + kS1; }
    __device__ const float* W3() const { return b2() + C; }
    __device__ const float* b3() const { return W3() + 2 * T * C; }
    // the weights of tap t (of the current stage)
    __device__ const float* W2(int t, int t0) const {
        return GW ? layer(l) + a.off.W2 + (size_t)t * C * C : w2_buf(buf) + (t - t0) * C * C;
    }
    __device__ void begin_layer() {
        passes = a.n_passes;
        first = true;
        if (GW) return;
        if (!a.two_small) load_small(0, l);
        cp_wait();                               // made visible by the next barrier
    }
    // before the taps of stage st: its weights have arrived, and the copies
    // of the stage after it go into the other buffer (whose readers have all
    // passed the barrier)
    __device__ void begin_stage(int st) {
        if (st == 0) --passes;
        if (!GW) cp_wait();
        __syncthreads();
        if (GW) return;
        if (a.n_stages > 1) {
            if (st > 0 || !first) buf ^= 1;
            if (st + 1 < a.n_stages) load_w2(buf ^ 1, l, st + 1);
            else if (passes > 0) load_w2(buf ^ 1, l, 0);
            else if (left > 0) load_w2(buf ^ 1, lnext, 0);
        } else if (first && left > 0) {
            load_w2(buf ^ 1, lnext, 0);
        }
        if (first && a.two_small && left > 0) load_small(sbuf ^ 1, lnext);
        first = false;
    }
    __device__ void end_layer() {
        if (GW) return;
        buf ^= 1;
        sbuf ^= 1;
    }
};

// ---------------------------------------------------------------- conv1
// h1 = LReLU(conv1(x at the sites of parity `frozen`)), 8 channels per thread,
// sites ordered by parity so that a warp's live taps agree (half of the taps
// reach fixed sites; the others add nothing).
template <int ND, int C, bool GW, int MODE>
__device__ void phase_h1(const FlowArgs& a, const Weights<ND, C, GW>& w, const Phase& ph, const float* x, float* h1,
                         int frozen, int64_t b) {
    const int L = a.L, S = a.S, hS = S >> 1, nf = ph.n * S, half = nf >> 1;
    const float* W1 = w.W1();
    const float* b1 = w.b1();
    for (int it = threadIdx.x; it < nf * (C / 8); it += blockDim.x) {
        int g = 0, f = it;
#pragma unroll
        for (int k = 1; k < C / 8; ++k)
            if (f >= nf) { f -= nf; ++g; }
        const int q = f >= half ? 1 : 0;
        f -= q * half;
        const int r = fdiv(f, a.fd_Sh), jj = f - r * hS;
        const int sl = wrap(ph.s0 + r, L);
        const int y = ND == 3 ? fdiv(jj, a.fd_Lh) : 0;
        const int xc = 2 * (jj - y * (L >> 1)) + ((q + sl + y) & 1);
        const int co = g << 3;
        f32x2 acc[4];
        load_w<8, GW>(acc, b1 + co);
        int xs[3], ys[3], zs[3];
        xs[0] = wrap(xc - 1, L); xs[1] = xc; xs[2] = wrap(xc + 1, L);
        zs[0] = wrap(sl - 1, L) * S; zs[1] = sl * S; zs[2] = wrap(sl + 1, L) * S;
        if (ND == 3) { ys[0] = wrap(y - 1, L) * L; ys[1] = y * L; ys[2] = wrap(y + 1, L) * L; }
        const bool even = q == frozen;           // taps of even offset parity are live
#pragma unroll
        for (int t = 0; t < (ND == 3 ? 27 : 9); ++t) {
            const int ds = ND == 3 ? t / 9 : t / 3, dy = ND == 3 ? (t / 3) % 3 : 1, dx = t % 3;
            if (((ds + dy + dx + 1) & 1) == (even ? 1 : 0)) continue;
            const f32x2 xv = f2_splat(x[zs[ds] + (ND == 3 ? ys[dy] : 0) + xs[dx]]);
            f32x2 ww[4];
            load_w<8, GW>(ww, W1 + t * C + co);
#pragma unroll
            for (int i = 0; i < 4; ++i) acc[i] = f2_fma(xv, ww[i], acc[i]);
        }
        float* o = h1 + (((size_t)ph.out[r] * (C / 4) + 2 * g) * S + (ND == 3 ? y * L : 0) + xc) * 4;
        float v[8];
#pragma unroll
        for (int i = 0; i < 4; ++i) { v[2 * i] = lrelu(f2_lo(acc[i]), a.slope); v[2 * i + 1] = lrelu(f2_hi(acc[i]), a.slope); }
        *reinterpret_cast<float4*>(o) = make_float4(v[0], v[1], v[2], v[3]);
        *reinterpret_cast<float4*>(o + 4 * S) = make_float4(v[4], v[5], v[6], v[7]);
        if constexpr (MODE == kRecompute) {
            float* go = a.h1_out + ((b * (C / 4) + 2 * g) * a.V + sl * S + (ND == 3 ? y * L : 0) + xc) * 4;
            *reinterpret_cast<float4*>(go) = make_float4(v[0], v[1], v[2], v[3]);
            *reinterpret_cast<float4*>(go + 4 * (int64_t)a.V) = make_float4(v[4], v[5], v[6], v[7]);
        }
    }
}

// ---------------------------------------------------------------- conv2
// One pass: warp `task` = 32 NS consecutive sites of the phase x CO channels.
template <int ND, int C, int NS, int CO, bool GW, int MODE>
__device__ __forceinline__ void conv2_pass(const FlowArgs& a, Weights<ND, C, GW>& w, const Phase& ph, const float* h1,
                                        float* h2, int pass, int64_t b) {
    const int L = a.L, S = a.S, nf = ph.n * S, nblk = (nf + 32 * NS - 1) / (32 * NS);
    const int lane = threadIdx.x & 31, task = pass * (int)(blockDim.x >> 5) + (int)(threadIdx.x >> 5);
    const int g = task / nblk, blk = task - g * nblk, co = g * CO;
    const bool active = g < C / CO;
    int at[NS];                                  // slice of the phase, y, x: 10 bits each
#pragma unroll
    for (int k = 0; k < NS; ++k) {
        const int f = min(blk * (32 * NS) + lane + 32 * k, nf - 1);
        const int r = fdiv(f, a.fd_S), j = f - r * S, y = ND == 3 ? fdiv(j, a.fd_L) : 0;
        at[k] = r << 20 | y << 10 | (j - y * L);
    }
    f32x2 acc[NS][CO / 2];
    for (int st = 0; st < a.n_stages; ++st) {
        w.begin_stage(st);
        if (!active) continue;
        if (st == 0) {
            f32x2 bias[CO / 2];
            load_w<CO, GW>(bias, w.b2() + co);
#pragma unroll
            for (int k = 0; k < NS; ++k)
#pragma unroll
                for (int i = 0; i < CO / 2; ++i) acc[k][i] = bias[i];
        }
        const auto tap = [&](int t, int t0) {
            const int ds = ND == 3 ? t / 9 - 1 : t / 3 - 1, dy = ND == 3 ? (t / 3) % 3 - 1 : 0, dx = t % 3 - 1;
            int row[NS];
#pragma unroll
            for (int k = 0; k < NS; ++k) {
                const int j2 = (ND == 3 ? wrap(((at[k] >> 10) & 1023) + dy, L) * L : 0) + wrap((at[k] & 1023) + dx, L);
                row[k] = ((int)ph.in[(at[k] >> 20) + 1 + ds] * (C / 4) * S + j2) * 4;
            }
            const float* wt = w.W2(t, t0) + co;
#pragma unroll (NS == 1 ? 2 : 1)
            for (int c4 = 0; c4 < C / 4; ++c4) {
                float4 hv[NS];
#pragma unroll
                for (int k = 0; k < NS; ++k) hv[k] = *reinterpret_cast<const float4*>(h1 + row[k] + c4 * S * 4);
#pragma unroll
                for (int cc = 0; cc < 4; ++cc) {
                    f32x2 ww[CO / 2];
                    load_w<CO, GW>(ww, wt + (4 * c4 + cc) * C);
#pragma unroll
                    for (int k = 0; k < NS; ++k) {
                        const f32x2 h = f2_splat(cc == 0 ? hv[k].x : cc == 1 ? hv[k].y : cc == 2 ? hv[k].z : hv[k].w);
#pragma unroll
                        for (int i = 0; i < CO / 2; ++i) acc[k][i] = f2_fma(h, ww[i], acc[k][i]);
                    }
                }
            }
        };
        if (NS == 1 && ND == 2 && C <= 16 && a.n_stages == 1) {   // latency-bound: every tap's loads in flight
#pragma unroll
            for (int t = 0; t < 9; ++t) tap(t, 0);
        } else {
            const int t0 = st * a.stage_taps, t1 = min(Weights<ND, C, GW>::T, t0 + a.stage_taps);
#pragma unroll (NS == 1 ? 3 : 1)
            for (int t = t0; t < t1; ++t) tap(t, t0);
        }
    }
    if (!active) return;
#pragma unroll
    for (int k = 0; k < NS; ++k) {
        if (blk * (32 * NS) + lane + 32 * k >= nf) continue;
        float* o = h2 + (((int)ph.out[at[k] >> 20] * (C / 4) + (co >> 2)) * S + (ND == 3 ? ((at[k] >> 10) & 1023) * L : 0) +
                         (at[k] & 1023)) * 4;
        float v[CO];
#pragma unroll
        for (int i = 0; i < CO / 2; ++i) {
            v[2 * i] = lrelu(f2_lo(acc[k][i]), a.slope);
            v[2 * i + 1] = lrelu(f2_hi(acc[k][i]), a.slope);
        }
        if constexpr (CO == 2) {
            *reinterpret_cast<float2*>(o + (co & 3)) = make_float2(v[0], v[1]);
        } else {
#pragma unroll
            for (int i = 0; i < CO / 4; ++i)
                *reinterpret_cast<float4*>(o + (size_t)i * S * 4) = make_float4(v[4 * i], v[4 * i + 1], v[4 * i + 2], v[4 * i + 3]);
        }
        if constexpr (MODE == kRecompute) {
            const int n = wrap(ph.s0 + (at[k] >> 20), L) * S + (ND == 3 ? ((at[k] >> 10) & 1023) * L : 0) + (at[k] & 1023);
            float* go = a.h2_out + ((b * (C / 4) + (co >> 2)) * a.V + n) * 4 + (co & 3);
#pragma unroll
            for (int i = 0; i < CO; i += 2)
                *reinterpret_cast<float2*>(go + (int64_t)(i / 4) * a.V * 4 + (i & 3)) = make_float2(v[i], v[i + 1]);
        }
    }
}

// ---------------------------------------------------------------- conv3 + affine update
// (s, t) at the updated sites of slices r0 .. r0 + nr - 1 of the phase as one
// packed pair; `tps` lanes share a site, each summing C / tps channels over all
// taps, combined with xor-shuffles.
template <int ND, int C, bool GW, int MODE>
__device__ void phase_c3(const FlowArgs& a, const Weights<ND, C, GW>& w, const Phase& ph, int r0, int nr, int tps,
                         const float* h2, float* x, float* s_site, int frozen, bool inverse, FF& logdet, int64_t b) {
    constexpr int T = ND == 3 ? 27 : 9;
    const int L = a.L, S = a.S, half = S >> 1;
    const int lt = 31 - __clz(tps), nchunk = (C / 4) >> lt;
    const int total = (nr * half) << lt;
    const float* W3 = w.W3();
    const float bs = GW ? __ldg(w.b3()) : w.b3()[0], bt = GW ? __ldg(w.b3() + 1) : w.b3()[1];
    const int iters = (total + blockDim.x - 1) / blockDim.x;
    for (int i = 0; i < iters; ++i) {
        const int it = i * blockDim.x + threadIdx.x;
        const bool valid = it < total;
        const int ai = valid ? it >> lt : 0, rk = it & (tps - 1);
        const int r = r0 + fdiv(ai, a.fd_Sh), aa = ai - (r - r0) * half;
        const int sl = wrap(ph.s0 + r, L);
        const int y = ND == 3 ? fdiv(aa, a.fd_Lh) : 0;
        const int xc = 2 * (aa - y * (L >> 1)) + ((frozen ^ 1 ^ sl ^ y) & 1);
        f32x2 p = a.head_train ? f2_make(bs, bt) : f2_make(0.f, 0.f);
        if (valid) {
            const int xs[3] = {wrap(xc - 1, L), xc, wrap(xc + 1, L)};
#pragma unroll (ND == 2 ? 3 : 1)
            for (int k = 0; k < T / 3; ++k) {
                const int ds = ND == 3 ? k / 3 : k, dy = ND == 3 ? k % 3 - 1 : 0;
                const float* row = h2 + ((int)ph.in[r + ds] * (C / 4) * S + (ND == 3 ? wrap(y + dy, L) * L : 0)) * 4;
#pragma unroll
                for (int dx = 0; dx < 3; ++dx) {
                    const float* wt = W3 + (3 * k + dx) * 2 * C;
#pragma unroll 2
                    for (int c = 0; c < nchunk; ++c) {
                        const int c4 = rk * nchunk + c;
                        const float4 hv = *reinterpret_cast<const float4*>(row + (c4 * S + xs[dx]) * 4);
                        f32x2 ww[4];
                        load_w<8, GW>(ww, wt + 8 * c4);
                        p = f2_fma(f2_splat(hv.x), ww[0], p);
                        p = f2_fma(f2_splat(hv.y), ww[1], p);
                        p = f2_fma(f2_splat(hv.z), ww[2], p);
                        p = f2_fma(f2_splat(hv.w), ww[3], p);
                    }
                }
            }
        }
        float ps = f2_lo(p), pt = f2_hi(p);
        for (int o = 1; o < tps; o <<= 1) {
            ps += __shfl_xor_sync(0xffffffffu, ps, o);
            pt += __shfl_xor_sync(0xffffffffu, pt, o);
        }
        if (valid && rk == 0) {
            const float spre = a.head_train ? ps : ps + bs, tt = a.head_train ? pt : pt + bt;
            const float s = a.use_tanh ? tanhf(spre) : spre;
            const int n = sl * S + (ND == 3 ? y * L : 0) + xc;
            if constexpr (MODE == kRecompute) {
                a.s_out[b * a.V + n] = s;
                continue;
            }
            if (!inverse) x[n] = fmaf(x[n], expf(s), tt);
            else x[n] = (x[n] - tt) * expf(-s);
            if (GW) ff_add(logdet, s);             // (256 threads and the blocks of head_split: the same order)
            else s_site[(ph.s0 + r) * half + aa] = s;
        }
    }
}

// Adds the s of one layer to the log-det of each of the kVT threads that the
// order of the sums stands for: site u (of the V/2 updated ones, in order) of a
// block of head_G slices starting at a, with tps lanes to a site, belongs to
// thread ((u - a) tps) mod kVT.
__device__ __forceinline__ void add_logdet(const FlowArgs& a, const float* s_site, FF (&ld)[4]) {
    const int half = a.S >> 1;
#pragma unroll
    for (int j = 0; j < 4; ++j) {
        const int vt = threadIdx.x + j * blockDim.x;
        if (vt >= kVT) break;
        for (int s0 = 0; s0 < a.L; s0 += a.head_G) {
            const int tps = s0 < a.head_zb ? a.head_a : a.head_b, n = min(a.head_G, a.L - s0) * half;
            if (vt & (tps - 1)) continue;
            const int lt = 31 - __clz(tps);
            for (int u = vt >> lt; u < n; u += kVT >> lt) ff_add(ld[j], s_site[s0 * half + u]);
        }
    }
}

// Training's log-det in FP64, added as k_couple_fwd of the layer-by-layer form
// does, so that a configuration's log q does not depend on which form its batch
// takes: thread vt of kVT takes the updated sites n = vt (mod kVT) of every layer
// in order, then block_sum's order.  FP64 instructions are slow, so a thread
// stands for vt = 2 i and 2 i + 1, of which one updates each of its site pairs,
// and FP32 is widened by integer instructions: one FP64 addition per 32 updated
// sites.  A training step takes 0.986 to 1.007 of its time with FP32 pairs (24 shapes).
struct TrainLogdet {
    double acc[2][2];                          // [i = thread + j CTA size][vt & 1]
};
__device__ __forceinline__ double widen(float f) {
    const uint32_t u = __float_as_uint(f), e = u & 0x7f800000u;
    if (e == 0u || e == 0x7f800000u) return (double)f;       // zero, subnormal, infinite, NaN
    return __hiloint2double((int)((u & 0x80000000u) | (((u & 0x7fffffffu) >> 3) + 0x38000000u)), (int)(u << 29));
}
// adds one layer (fixed sites of parity `frozen`)
template <int ND>
__device__ __forceinline__ void train_logdet(const FlowArgs& a, const float* s_site, int frozen, TrainLogdet& t) {
#pragma unroll
    for (int j = 0; j < 2; ++j) {
#pragma unroll 1
        for (int i = threadIdx.x + j * blockDim.x, u = i; i < kVT / 2 && u < (a.V >> 1); u += kVT / 2) {
            const int sl = fdiv(2 * u, a.fd_S), row = ND == 3 ? fdiv(2 * u, a.fd_L) + sl : sl;   // (L is even)
            const bool odd = ((frozen + 1 + row) & 1) != 0;            // x of the pair's updated site
            const double v = (odd ? t.acc[j][1] : t.acc[j][0]) + widen(s_site[u]);
            t.acc[j][0] = odd ? t.acc[j][0] : v;
            t.acc[j][1] = odd ? v : t.acc[j][1];
        }
    }
}
// the sum over the threads (valid in thread 0); buf: kVT doubles (V when that is less)
__device__ __forceinline__ double train_logdet_sum(const FlowArgs& a, const TrainLogdet& t, double* buf, double* red) {
#pragma unroll
    for (int j = 0; j < 2; ++j) {
        const int i = threadIdx.x + j * blockDim.x;
        if (i >= kVT / 2 || 2 * i >= a.V) continue;
        buf[2 * i] = t.acc[j][0];
        buf[2 * i + 1] = t.acc[j][1];
    }
    __syncthreads();
    for (int vt = threadIdx.x; vt < kVT; vt += blockDim.x) {           // (uniform in a warp)
        const double w = warp_sum(vt < a.V ? buf[vt] : 0.0);
        if ((vt & 31) == 0) red[vt >> 5] = w;
    }
    __syncthreads();
    double r = 0.0;
    for (int i = 0; i < kVT / 32; ++i) r += red[i];
    return r;
}

// FP64 value of the sum of part(j, vt) over vt < kVT in the order of kVT
// threads (a butterfly in each warp of 32, then one over the warps); valid in
// every thread.
template <typename F>
__device__ double order_sum(FF* red, F part) {
    const int lane = threadIdx.x & 31;
#pragma unroll
    for (int j = 0; j < 4; ++j) {
        const int vt = threadIdx.x + j * blockDim.x;
        if (vt >= kVT) break;                      // (uniform in a warp: kVT and the CTA size are multiples of 32)
        const FF v = warp_sum_ff(part(j, vt));
        if (lane == 0) red[vt >> 5] = v;
    }
    __syncthreads();
    FF r = lane < kVT / 32 ? red[lane] : FF{0.f, 0.f};
    r = warp_sum_ff(r);
    __syncthreads();
    return ff_to_double(r);
}

// (kFlow keeps its tests of xs_out and logdet_out, which are null there: without
// them ptxas orders conv2's loop in the 5 x 8 tiles, at the limit of registers,
// 4 % to 8 % slower; 3D L = 12, hidden 32, 8 layers, 300 configurations 7.45 -> 8.07 ms.)
template <int ND, int C, int NS, int CO, bool GW, int MODE>
__global__ void __launch_bounds__(512, 1) flow_fp32_kernel(const __grid_constant__ FlowArgs a, int inverse) {
    extern __shared__ __align__(16) float smf[];
    const int V = a.V;
    float* x = smf;
    float* h1 = smf + a.off_h1;
    float* h2 = smf + a.off_h2;
    FF* red = reinterpret_cast<FF*>(smf + a.off_red);
    float* s_site = smf + a.off_s;
    const Phase* sched = GW ? a.sched : reinterpret_cast<const Phase*>(smf + a.off_sched);
    if (!GW)
        for (int i = threadIdx.x; i < a.n_phases * (int)(sizeof(Phase) / 4); i += blockDim.x)
            reinterpret_cast<uint32_t*>(smf + a.off_sched)[i] = __ldg(reinterpret_cast<const uint32_t*>(a.sched) + i);
    const int64_t n_cfg = a.B > (int64_t)blockIdx.x ? (a.B - 1 - (int64_t)blockIdx.x) / gridDim.x + 1 : 0;
    const int N = a.n_layers;
    Weights<ND, C, GW> w{a, smf, n_cfg * N - 1, inverse ? N - 1 : a.layer0, 0, 0, 0, 0, true};
    if (!GW && n_cfg * N > 0) {
        w.load_small(0, w.l);
        w.load_w2(0, w.l, 0);
    }
    const auto square = [](float v) { const float p = v * v; return FF{p, fmaf(v, v, -p)}; };

    for (int64_t b = blockIdx.x; b < a.B; b += gridDim.x) {
        if (!inverse) {
            if (a.z_in) {
                for (int n = threadIdx.x; n < V; n += blockDim.x) x[n] = __ldg(a.z_in + b * V + n);
            } else {
                for (int j = threadIdx.x; 4 * j < V; j += blockDim.x) {
                    const u64x4 r = philox4x64_10(a.seed, 0ull,
                                                  u64x4{a.counter0 + (uint64_t)b, (uint64_t)j, 0ull, TAG_PRIOR});
                    float zz[4];
                    normals4_f32(r, zz);
#pragma unroll
                    for (int q = 0; q < 4; ++q)
                        if (4 * j + q < V) x[4 * j + q] = zz[q];
                }
            }
        } else {
            for (int n = threadIdx.x; n < V; n += blockDim.x) x[n] = __ldg(a.phi_in + b * V + n);
        }
        __syncthreads();
        FF logdet[4] = {{0.f, 0.f}, {0.f, 0.f}, {0.f, 0.f}, {0.f, 0.f}};
        TrainLogdet tld = {};                      // (kForward)
        double z2 = 0.0;
        const auto sum_squares = [&](int, int vt) {   // each square exactly as a pair
            FF v{0.f, 0.f};
            if (!inverse && !a.z_in) {                // drawn: four sites to a Philox block
                for (int n = 4 * vt; n < V; n += 4 * kVT)
                    for (int q = 0; q < 4 && n + q < V; ++q) ff_add(v, square(x[n + q]));
            } else {
                for (int n = vt; n < V; n += kVT) ff_add(v, square(x[n]));
            }
            return v;
        };
        if (!inverse && MODE != kRecompute) {
            if constexpr (MODE == kFlow) z2 = order_sum(red, sum_squares);
            for (int n = threadIdx.x; n < V; n += blockDim.x) {
                const float v = x[n];
                if (a.z_out) a.z_out[b * V + n] = v;
                if (a.xs_out) a.xs_out[b * V + n] = v;
            }
        }

        for (int li = 0; li < N; ++li) {
            w.lnext = inverse ? (w.l == 0 ? N - 1 : w.l - 1) : (w.l + 1 == a.layer0 + N ? a.layer0 : w.l + 1);
            const int frozen = w.l & 1;
            if (a.xs_out && li > 0) {
                __syncthreads();
                for (int n = threadIdx.x; n < V; n += blockDim.x) a.xs_out[li * a.xs_stride + b * V + n] = x[n];
            }
            if (!GW && !a.two_small) __syncthreads();   // the previous layer's weights are no longer read
            w.begin_layer();
            for (int p = 0; p < a.n_phases; ++p) {
                const Phase& ph = sched[p];
                if (ph.type == PH_H2) {            // begins with a barrier of its own (begin_stage)
                    const int tasks = ((ph.n * a.S + 32 * NS - 1) / (32 * NS)) * (C / CO), nw = (int)(blockDim.x >> 5);
                    for (int q = 0; q * nw < tasks; ++q) conv2_pass<ND, C, NS, CO, GW, MODE>(a, w, ph, h1, h2, q, b);
                    continue;
                }
                __syncthreads();
                if (ph.type == PH_H1) {
                    if constexpr (MODE == kForward) {
                        if (p == 0 && li > 0) train_logdet<ND>(a, s_site, frozen ^ 1, tld);
                    } else {
                        if (!GW && p == 0 && li > 0) add_logdet(a, s_site, logdet);
                    }
                    phase_h1<ND, C, GW, MODE>(a, w, ph, x, h1, frozen, b);
                } else {
                    const int na = max(0, min((int)ph.n, a.head_zb - (int)ph.s0));
                    if (na > 0) phase_c3<ND, C, GW, MODE>(a, w, ph, 0, na, a.head_a, h2, x, s_site, frozen, inverse, logdet[0], b);
                    if (na < ph.n)
                        phase_c3<ND, C, GW, MODE>(a, w, ph, na, ph.n - na, a.head_b, h2, x, s_site, frozen, inverse, logdet[0], b);
                }
            }
            w.end_layer();
            w.l = w.lnext;
            --w.left;
        }
        __syncthreads();
        if constexpr (MODE == kForward) {
            for (int n = threadIdx.x; n < V; n += blockDim.x) a.phi_out[b * V + n] = x[n];
            if (N > 0) train_logdet<ND>(a, s_site, (N - 1) & 1, tld);
            const double ld = train_logdet_sum(a, tld, reinterpret_cast<double*>(h1), reinterpret_cast<double*>(red));
            if (threadIdx.x == 0) a.logdet_out[b] = ld;
        }
        if constexpr (MODE != kFlow) continue;     // (the next configuration's x may be written now)

        for (int n = threadIdx.x; n < V; n += blockDim.x) {
            if (!inverse) a.phi_out[b * V + n] = x[n];
            else if (a.z_out) a.z_out[b * V + n] = x[n];
        }
        if (!GW && N > 0) add_logdet(a, s_site, logdet);
        const double ld = order_sum(red, [&](int j, int) { return logdet[j]; });
        if (inverse) z2 = order_sum(red, sum_squares);
        double S = 0.0;
        if (!inverse && a.has_phi4)
            S = order_sum(red, [&](int, int vt) { return action_part<ND>(x, a.L, V, a.c2d_ff, a.lam_ff, vt, kVT); });
        if (threadIdx.x == 0) {
            if (a.logdet_out) a.logdet_out[b] = ld;
            const double logr = -0.5 * z2 - 0.5 * (double)V * LOG_2PI;
            const double logq = logr - ld;
            a.logq_out[b] = logq;
            if (!inverse && a.has_phi4) {
                if (a.S_out) a.S_out[b] = S;
                if (a.logw_out) a.logw_out[b] = -S - logq;
            }
        }
        __syncthreads();
    }
    if (!GW) cp_wait();
}

using FlowKernel = void (*)(const FlowArgs, int);
// the kernel of a lattice dimension, width, tile and mode (gf_flow_fp32_*d_w*.cu);
// the recompute has tiles from kTileRec on, weights in global memory are for
// kFlow alone
constexpr int kTileRec = 2;
template <int ND, int C>
FlowKernel kernel_of(int tile, bool gw, int mode);

template <int ND, int C, int I = 0>
FlowKernel pick_kernel(int tile, bool gw, int mode) {
    if constexpr (I == kTiles) {
        return nullptr;
    } else if constexpr (I < tile_first(C)) {
        return pick_kernel<ND, C, I + 1>(tile, gw, mode);
    } else {
        if (gw) return flow_fp32_kernel<ND, C, kTileNS[kTileGW], kTileCO[kTileGW], true, kFlow>;
        if (tile == I && mode == kFlow) return flow_fp32_kernel<ND, C, kTileNS[I], kTileCO[I], false, kFlow>;
        if (tile == I && mode == kForward) return flow_fp32_kernel<ND, C, kTileNS[I], kTileCO[I], false, kForward>;
        if constexpr (I >= kTileRec)
            if (tile == I && mode == kRecompute) return flow_fp32_kernel<ND, C, kTileNS[I], kTileCO[I], false, kRecompute>;
        return pick_kernel<ND, C, I + 1>(tile, gw, mode);
    }
}

}  // namespace f32k
}  // namespace gf
