// gf_flow_variant.cu -- fused FP32 coupling-stack kernel for the general s/t
// network of the paper's model section (Sec. 3, model parameters
// hidden_sizes and kernel_size): any list of up to GF_MAX_HIDDEN hidden
// convolutions of any width (LeakyReLU after each), an odd kernel size
// (k^nd taps, circular padding (k-1)/2), then the head conv(-> 2) giving s
// (tanh when use_final_tanh) and t.  The coupling layers, log-det, log q, the
// action and log w are those of Sec. 1, as in gf_flow_fp32.cu.
//
// One CTA owns one configuration at a time (persistent grid-stride loop).
// The whole lattice stays in shared memory through every layer: the field x
// and two ping-pong activation buffers [V][Cp], Cp = the widest hidden layer
// rounded up to an odd number of floats, so that lanes reading consecutive
// sites' rows hit distinct banks.  A thread computes up to 8 output channels
// of 1, 2 or 4 sites V / NS apart (the same x coordinate, so one wrap in x for
// all of them) as packed FMAs over channel pairs: per input channel 2 weight
// loads that a whole warp shares and NS site loads feed 4 NS packed FMAs.  The
// layer's weights stream through two shared-memory stages of whole (tap, input
// channel) rows, the next chunk copied (cp.async) while this one is used; one
// barrier per chunk.  Supported while x and both buffers fit in the 227 KB of
// shared memory (gf_flow_create_ex returns GF_EUNSUPPORTED otherwise); where
// the stages don't fit beside them, the weights are read through L1.
//
// What bounds it: the latency of shared-memory loads and barriers with few warps
// (registers, or the buffers' shared memory, allow 16 to 24 an SM), and registers:
// one kernel holds up to three forms of the hidden convolution and of the head, and
// each of the six instantiations spills 1.2 to 1.9 KB of stores and 0.6 to 1.3 KB of
// loads a thread at 80 or 128 registers (the former one-site kernel up to 32 bytes).  One site per
// thread with the weights through L1 was bound by load issue (8 FMAs to 3 loads)
// and waited for L2 at the start of every convolution: 2D L = 16, 12 layers,
// widths 16, 16, 8, 5 taps, 500 configurations 3004 us, now 1319 (23 TFLOP/s);
// 3D L = 8, widths 16, 8, 16, 4 layers, 300 configurations 1291 -> 419.
//
// Each sum runs over taps, then input channels, from the bias, and the lattice
// sums are added as by `vthreads` threads whatever the CTA's size, so results
// depend on the shape alone.
#include <algorithm>
#include <cstring>
#include <type_traits>

#include "gf_flow_fp32_kernel.cuh"

namespace gf {

namespace {

struct VarArgs {
    const float* W;                        // packed weights, layer stride `stride`
    int64_t stride;
    int32_t woff[GF_MAX_HIDDEN + 1];       // conv j: W[t][cin][cop] (layer-relative)
    int32_t boff[GF_MAX_HIDDEN + 1];       // conv j: bias[cop]
    int32_t cin[GF_MAX_HIDDEN + 1], cout[GF_MAX_HIDDEN + 1], cop[GF_MAX_HIDDEN + 1];
    int32_t rows[GF_MAX_HIDDEN + 1];       // conv j: (tap, input channel) rows per staged chunk
    int32_t ns[GF_MAX_HIDDEN + 1];         // conv j: sites per thread
    int nh, K, L, V, Cp, n_layers;
    int vt;                                // threads of the sums' order (at most 4 per CTA thread)
    int stage;                             // floats of a stage's rows; its bias follows
    int stage_stride;
    int off_stage;
    float slope;
    int use_tanh, has_phi4;
    FF c2d_ff, lam_ff;
    int64_t B;
    uint64_t seed, counter0;
    const float* z_in;
    float* z_out;
    const float* phi_in;
    float* phi_out;
    double* logq_out;
    double* S_out;
    double* logw_out;
};

// v mod L for -L <= v < 2 L, and any v for L = 2 (the offsets are at most 3 from
// a site, and L is even).
__device__ __forceinline__ int wrapv(int v, int L) {
    if (L == 2) return v & 1;
    v += v < 0 ? L : 0;
    return v - (v >= L ? L : 0);
}
__device__ __forceinline__ float lrelu(float v, float a) { return v > 0.f ? v : a * v; }

extern __shared__ __align__(16) float smv[];

// The chunks of weights in the order of use: for every configuration, layer
// and convolution, its rows (once per pass over its items if they need more
// than one chunk).  Advanced alike by every thread.
struct Stream {
    int64_t b;
    int li, j, p, c, passes, buf;
};

// passes over conv j's items: NT threads, ns sites each (the head: the sites of
// the virtual threads that a thread stands for)
__device__ __forceinline__ int conv_passes(const VarArgs& a, int j) {
    const int nt = blockDim.x;
    if (j == a.nh) return ((a.vt + nt - 1) / nt) * (((a.V >> 1) + a.vt * a.ns[j] - 1) / (a.vt * a.ns[j]));
    const int items = (a.V / a.ns[j]) * ((a.cop[j] + 7) >> 3);
    return (items + nt - 1) / nt;
}
__device__ __forceinline__ int conv_rows(const VarArgs& a, int j, int taps) { return taps * a.cin[j]; }

// Copies the stream's next chunk into its stage and advances the stream.
__device__ __forceinline__ void issue_chunk(const VarArgs& a, Stream& s, int taps, bool inverse) {
    if (s.b >= a.B || a.n_layers == 0) return;
    const int l = inverse ? a.n_layers - 1 - s.li : s.li, total = conv_rows(a, s.j, taps), per = a.rows[s.j];
    const float* W = a.W + (size_t)l * a.stride;
    float* dst = smv + a.off_stage + s.buf * a.stage_stride;
    const int cop = a.cop[s.j], r0 = s.c * per, n = min(per, total - r0) * cop;
    f32k::cp_copy(dst, W + a.woff[s.j] + (size_t)r0 * cop, n);
    if (s.c == 0) f32k::cp_copy(dst + a.stage, W + a.boff[s.j], cop);
    s.buf ^= 1;
    ++s.c;
    if (s.c * per < total) return;
    s.c = 0;
    ++s.p;
    if (per < total && s.p < s.passes) return;
    s.p = 0;
    if (++s.j > a.nh) {
        s.j = 0;
        if (++s.li == a.n_layers) {
            s.li = 0;
            s.b += gridDim.x;
        }
    }
    s.passes = conv_passes(a, s.j);
}

// Waits for the chunk in flight, starts the next one, returns the chunk's stage.
__device__ __forceinline__ int next_chunk(const VarArgs& a, Stream& s, int taps, bool inverse) {
    const int at = a.off_stage + (s.buf ^ 1) * a.stage_stride;
    f32k::cp_wait();
    __syncthreads();
    issue_chunk(a, s, taps, inverse);
    return at;
}

// Tap and input channel of the next row.
struct Walk { int kx, ky, kz, ci; };

// acc += weights of `rows` rows (CO of their cop channels) times the sites'
// inputs.  Site s is at (xc[s], y[s], z[s]), or all at xc[0] (NX = 1); its row of `stride` floats starts at
// in + site * stride.  zero >= 0: a masked input (one channel), read at the
// sites of parity `frozen` and as the zero at smv[zero] elsewhere.
template <int ND, int NS, int NX, int CO, bool STAGED, bool ONE>
__device__ __forceinline__ void add_rows(const VarArgs& a, f32x2 (&acc)[NS][CO / 2], Walk& w, const int (&xc)[NX], const int (&y)[NS],
                                         const int (&z)[NS], const float* wg, int ws, int cop, int rows, int cin, int in,
                                         int stride, int zero, int frozen) {
    const int K = a.K, L = a.L, h = (K - 1) >> 1;
    int at[NS], odd[NS];                           // start and parity of each site's row of this (ky, kz)
    bool moved = true;
    while (rows > 0) {
        if (moved) {
#pragma unroll
            for (int s = 0; s < NS; ++s) {
                const int yy = wrapv(y[s] + w.ky - h, L), zz = ND == 3 ? wrapv(z[s] + w.kz - h, L) : 0;
                at[s] = in + (zz * L + yy) * L * stride;
                odd[s] = yy + zz + frozen;
            }
            moved = false;
        }
        int xx[NX], q[NS];
#pragma unroll
        for (int s = 0; s < NX; ++s) xx[s] = wrapv(xc[s] + w.kx - h, L);
#pragma unroll
        for (int s = 0; s < NS; ++s) {
            const int X = xx[NX == 1 ? 0 : s];
            q[s] = ONE ? at[s] + X * stride : at[s] + X * stride + w.ci;
            if (ONE && zero >= 0 && ((X + odd[s]) & 1)) q[s] = zero;
        }
        const int e = ONE ? 1 : min(cin - w.ci, rows);
#pragma unroll (ONE ? 1 : 4)
        for (int i = 0; i < e; ++i) {
            f32x2 wv[CO / 2], v[NS];
            if constexpr (CO == 2) {
                wv[0] = STAGED ? *reinterpret_cast<const f32x2*>(smv + ws) : __ldg(reinterpret_cast<const f32x2*>(wg));
            } else {
#pragma unroll
                for (int c = 0; c < CO / 4; ++c) {
                    const ulonglong2 u = STAGED ? *reinterpret_cast<const ulonglong2*>(smv + ws + 4 * c)
                                                : __ldg(reinterpret_cast<const ulonglong2*>(wg + 4 * c));
                    wv[2 * c] = u.x;
                    wv[2 * c + 1] = u.y;
                }
            }
#pragma unroll
            for (int s = 0; s < NS; ++s) v[s] = f2_splat(smv[q[s] + i]);
#pragma unroll
            for (int s = 0; s < NS; ++s)
#pragma unroll
                for (int c = 0; c < CO / 2; ++c) acc[s][c] = f2_fma(v[s], wv[c], acc[s][c]);
            if (STAGED) ws += cop;
            else wg += cop;
        }
        rows -= e;
        if (!ONE) w.ci += e;
        if (ONE || w.ci == cin) {
            w.ci = 0;
            if (++w.kx == K) {
                w.kx = 0;
                moved = true;
                if (++w.ky == K) { w.ky = 0; ++w.kz; }
            }
        }
    }
}

// conv j of the hidden chain: out = LReLU(conv_j(in)), rows of Cp floats.  conv
// 0 reads the field at the sites of parity `frozen` and zero elsewhere.
template <int ND, int NS, bool STAGED>
__device__ void hidden_conv(const VarArgs& a, Stream& st, const float* __restrict__ Wl, int j, int in, int stride, int zero,
                            int frozen, int out, int taps, bool inverse) {
    const int cin = a.cin[j], cout = a.cout[j], cop = a.cop[j], L = a.L, total = conv_rows(a, j, taps);
    const int chunk = STAGED ? a.rows[j] : total;
    const int per = a.V / NS, items = per * ((cop + 7) >> 3), rows_s = per / L;   // lattice rows between a thread's sites
    int ws = 0;
    if (!STAGED) __syncthreads();
    for (int it0 = 0; it0 < items; it0 += blockDim.x) {
        const int it = it0 + threadIdx.x, g = it / per, k = it - g * per, co = g << 3;
        const bool act = it < items, eight = co + 4 < cop;
        const int xc[1] = {k % L}, row = k / L;
        int y[NS], z[NS];
#pragma unroll
        for (int s = 0; s < NS; ++s) {
            const int r = row + s * rows_s;
            z[s] = ND == 3 ? r / L : 0;
            y[s] = r - z[s] * L;
        }
        f32x2 acc[NS][4];
        Walk w{0, 0, 0, 0};
        for (int r0 = 0; r0 < total; r0 += chunk) {
            if (STAGED && (it0 == 0 || chunk < total)) ws = next_chunk(a, st, taps, inverse);
            if (!act) continue;
            const int n = min(chunk, total - r0);
            if (r0 == 0) {
                const float* bg = Wl + a.boff[j] + co;
#pragma unroll
                for (int c = 0; c < 4; ++c) {
                    const bool on = c < 2 || eight;
                    const float lo = on ? (STAGED ? smv[ws + a.stage + co + 2 * c] : __ldg(bg + 2 * c)) : 0.f;
                    const float hi = on ? (STAGED ? smv[ws + a.stage + co + 2 * c + 1] : __ldg(bg + 2 * c + 1)) : 0.f;
#pragma unroll
                    for (int s = 0; s < NS; ++s) acc[s][c] = f2_make(lo, hi);
                }
            }
            const float* wg = Wl + a.woff[j] + (size_t)r0 * cop + co;
            if (eight) {
                if (cin == 1)
                    add_rows<ND, NS, 1, 8, STAGED, true>(a, acc, w, xc, y, z, wg, ws + co, cop, n, cin, in, stride, zero, frozen);
                else
                    add_rows<ND, NS, 1, 8, STAGED, false>(a, acc, w, xc, y, z, wg, ws + co, cop, n, cin, in, stride, zero, frozen);
            } else {
                f32x2 four[NS][2];
#pragma unroll
                for (int s = 0; s < NS; ++s) { four[s][0] = acc[s][0]; four[s][1] = acc[s][1]; }
                if (cin == 1)
                    add_rows<ND, NS, 1, 4, STAGED, true>(a, four, w, xc, y, z, wg, ws + co, cop, n, cin, in, stride, zero, frozen);
                else
                    add_rows<ND, NS, 1, 4, STAGED, false>(a, four, w, xc, y, z, wg, ws + co, cop, n, cin, in, stride, zero, frozen);
#pragma unroll
                for (int s = 0; s < NS; ++s) { acc[s][0] = four[s][0]; acc[s][1] = four[s][1]; }
            }
        }
        if (!act) continue;
#pragma unroll
        for (int s = 0; s < NS; ++s) {
            float* o = smv + out + (size_t)(k + s * per) * a.Cp + co;
#pragma unroll
            for (int c = 0; c < 4; ++c) {
                if (co + 2 * c < cout) o[2 * c] = lrelu(f2_lo(acc[s][c]), a.slope);
                if (co + 2 * c + 1 < cout) o[2 * c + 1] = lrelu(f2_hi(acc[s][c]), a.slope);
            }
        }
    }
}

// Head conv(-> s, t) at the updated sites of this layer and the affine
// update of x there (x * e^s + t, or (x - t) e^-s inverting), log-det += s.
// Its input is the last hidden activation, or the masked field when the net
// has no hidden layer (the head then reads only fixed sites, which this
// layer does not change).  Virtual thread v takes the updated sites v, v + vt,
// ..., NS of them at a time.
template <int ND, int NS, bool STAGED>
__device__ void head_conv(const VarArgs& a, Stream& st, const float* __restrict__ Wl, int in, int stride, int zero,
                          int frozen, int taps, bool inverse, FF (&logdet)[4]) {
    const int j = a.nh, cin = a.cin[j], L = a.L, half = L >> 1, n_upd = a.V >> 1, total = conv_rows(a, j, taps);
    const int chunk = STAGED ? a.rows[j] : total;
    const int pa = frozen ^ 1;                        // parity of the updated sites
    int ws = 0;
    bool first = true;
    if (!STAGED) __syncthreads();
#pragma unroll
    for (int jv = 0; jv < 4; ++jv) {
        const int v = threadIdx.x + jv * blockDim.x;
        if (jv * (int)blockDim.x >= a.vt) break;
        for (int a0 = 0; a0 < n_upd; a0 += NS * a.vt) {
            const bool act = v < a.vt && a0 + v < n_upd;
            int xc[NS], y[NS], z[NS];
#pragma unroll
            for (int s = 0; s < NS; ++s) {            // (beyond the last site: the first again, not stored)
                const int at = a0 + v + s * a.vt, ai = at < n_upd ? at : 0;
                const int r = ai / half, k = ai - r * half;   // row r = y + L z, k-th updated site in it
                z[s] = ND == 3 ? r / L : 0;
                y[s] = r - z[s] * L;
                xc[s] = 2 * k + ((pa ^ y[s] ^ z[s]) & 1);
            }
            f32x2 acc[NS][1];
            Walk w{0, 0, 0, 0};
            for (int r0 = 0; r0 < total; r0 += chunk) {
                if (STAGED && (first || chunk < total)) ws = next_chunk(a, st, taps, inverse);
                first = false;
                if (!act) continue;
                if (r0 == 0) {
                    const float* bg = Wl + a.boff[j];
                    const f32x2 b = STAGED ? f2_make(smv[ws + a.stage], smv[ws + a.stage + 1]) : f2_make(__ldg(bg), __ldg(bg + 1));
#pragma unroll
                    for (int s = 0; s < NS; ++s) acc[s][0] = b;
                }
                const float* wg = Wl + a.woff[j] + (size_t)r0 * 4;
                const int n = min(chunk, total - r0);
                if (cin == 1)
                    add_rows<ND, NS, NS, 2, STAGED, true>(a, acc, w, xc, y, z, wg, ws, 4, n, cin, in, stride, zero, frozen);
                else
                    add_rows<ND, NS, NS, 2, STAGED, false>(a, acc, w, xc, y, z, wg, ws, 4, n, cin, in, stride, zero, frozen);
            }
            if (!act) continue;
#pragma unroll
            for (int s = 0; s < NS; ++s) {
                if (a0 + v + s * a.vt >= n_upd) break;
                const float ps = f2_lo(acc[s][0]), pt = f2_hi(acc[s][0]), sc = a.use_tanh ? tanhf(ps) : ps;
                float& xv = smv[(z[s] * L + y[s]) * L + xc[s]];
                if (!inverse) xv = fmaf(xv, expf(sc), pt);
                else xv = (xv - pt) * expf(-sc);
                ff_add(logdet[jv], sc);
            }
        }
    }
}

// Sum of one pair per virtual thread (part(j, v) of thread v = threadIdx.x + j
// blockDim.x), in the order of block_sum_ff of a block of vt threads.
template <typename F>
__device__ double order_sum(FF* red, int vt, F part) {
    const int lane = threadIdx.x & 31;
#pragma unroll
    for (int j = 0; j < 4; ++j) {
        const int v = threadIdx.x + j * blockDim.x;
        if (v >= vt) break;                        // (uniform in a warp: multiples of 32)
        const FF r = warp_sum_ff(part(j, v));
        if (lane == 0) red[v >> 5] = r;
    }
    __syncthreads();
    FF r = lane < (vt >> 5) ? red[lane] : FF{0.f, 0.f};
    r = warp_sum_ff(r);
    __syncthreads();
    return ff_to_double(r);
}

template <int ND, int NSMAX, bool STAGED>
__global__ void __launch_bounds__(256, NSMAX == 4 ? 2 : 3) flow_variant_kernel(const __grid_constant__ VarArgs a, int inverse) {
    const int V = a.V, vt = a.vt;
    const int Vpad = (V + 3) & ~3;
    int taps = a.K * a.K;
    if (ND == 3) taps *= a.K;
    float* x = smv;
    const int bufA = Vpad, bufB = bufA + V * a.Cp, red_at = (Vpad + 2 * V * a.Cp + 1) & ~1;
    FF* red = reinterpret_cast<FF*>(smv + red_at);
    const int zero_at = red_at + 32;               // (a sum uses at most 8 pairs)
    if (threadIdx.x == 0) smv[zero_at] = 0.f;

    Stream st{blockIdx.x, 0, 0, 0, 0, conv_passes(a, 0), 0};
    if (STAGED) issue_chunk(a, st, taps, inverse);
    for (int64_t b = blockIdx.x; b < a.B; b += gridDim.x) {
        if (inverse || a.z_in) {
            const float* src = (inverse ? a.phi_in : a.z_in) + b * V;
            for (int n = threadIdx.x; n < V; n += blockDim.x) x[n] = __ldg(src + n);
        } else {
            for (int jq = threadIdx.x; 4 * jq < V; jq += blockDim.x) {
                const u64x4 w = philox4x64_10(a.seed, 0ull,
                                              u64x4{a.counter0 + (uint64_t)b, (uint64_t)jq, 0ull, TAG_PRIOR});
                float zz[4];
                normals4_f32(w, zz);
#pragma unroll
                for (int q = 0; q < 4; ++q)
                    if (4 * jq + q < V) x[4 * jq + q] = zz[q];
            }
        }
        __syncthreads();
        const auto square = [](float v) {
            const float p = v * v;
            return FF{p, fmaf(v, v, -p)};
        };
        const auto sum_squares = [&](int, int v) {
            FF r{0.f, 0.f};
            if (!inverse && !a.z_in) {                 // drawn: four sites to a Philox block
                for (int n = 4 * v; n < V; n += 4 * vt)
                    for (int q = 0; q < 4 && n + q < V; ++q) ff_add(r, square(x[n + q]));
            } else {
                for (int n = v; n < V; n += vt) ff_add(r, square(x[n]));
            }
            return r;
        };
        double z2 = 0.0;
        if (!inverse) {
            z2 = order_sum(red, vt, sum_squares);
            if (a.z_out)
                for (int n = threadIdx.x; n < V; n += blockDim.x) a.z_out[b * V + n] = x[n];
        }

        FF logdet[4] = {{0.f, 0.f}, {0.f, 0.f}, {0.f, 0.f}, {0.f, 0.f}};
        for (int li = 0; li < a.n_layers; ++li) {
            const int l = inverse ? a.n_layers - 1 - li : li;
            const int frozen = l & 1;
            const float* Wl = a.W + (size_t)l * a.stride;
            int in = 0, stride = 1, zero = zero_at;
            for (int j = 0; j < a.nh; ++j) {
                const int out = j & 1 ? bufB : bufA;
                if (NSMAX == 4 && a.ns[j] == 4)
                    hidden_conv<ND, NSMAX, STAGED>(a, st, Wl, j, in, stride, zero, frozen, out, taps, inverse);
                else if (a.ns[j] == 2)
                    hidden_conv<ND, 2, STAGED>(a, st, Wl, j, in, stride, zero, frozen, out, taps, inverse);
                else
                    hidden_conv<ND, 1, STAGED>(a, st, Wl, j, in, stride, zero, frozen, out, taps, inverse);
                in = out;
                stride = a.Cp;
                zero = -1;
            }
            if (a.ns[a.nh] == 4) head_conv<ND, 4, STAGED>(a, st, Wl, in, stride, zero, frozen, taps, inverse, logdet);
            else if (a.ns[a.nh] == 2) head_conv<ND, 2, STAGED>(a, st, Wl, in, stride, zero, frozen, taps, inverse, logdet);
            else head_conv<ND, 1, STAGED>(a, st, Wl, in, stride, zero, frozen, taps, inverse, logdet);
        }
        __syncthreads();

        float* dst = inverse ? a.z_out : a.phi_out;
        if (dst)
            for (int n = threadIdx.x; n < V; n += blockDim.x) dst[b * V + n] = x[n];
        const double ld = order_sum(red, vt, [&](int j, int) { return logdet[j]; });
        if (inverse) z2 = order_sum(red, vt, sum_squares);
        double S = 0.0;
        if (!inverse && a.has_phi4)
            S = order_sum(red, vt, [&](int, int v) { return action_part<ND>(x, a.L, V, a.c2d_ff, a.lam_ff, v, vt); });
        if (threadIdx.x == 0) {
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
}

// Canonical FP32 weights -> variant packed layout.  Canonical per layer, for
// each conv j: W_j[o][i][t] then b_j[o]; packed: W_j[t][i][cop] at woff[j]
// (o fastest, zero-padded to cop) and b_j[cop] at boff[j].
struct VarRepack {
    int32_t coff[GF_MAX_HIDDEN + 2];       // canonical start of conv j in a layer (j = nh+1: end)
    int32_t woff[GF_MAX_HIDDEN + 1], boff[GF_MAX_HIDDEN + 1];
    int32_t cin[GF_MAX_HIDDEN + 1], cout[GF_MAX_HIDDEN + 1], cop[GF_MAX_HIDDEN + 1];
    int nh, T, n_layers;
    int64_t cstride, pstride;
};

__global__ void repack_variant_kernel(const float* __restrict__ canon, float* __restrict__ packed, const VarRepack r) {
    const int64_t total = (int64_t)r.n_layers * r.cstride;
    for (int64_t i = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; i < total;
         i += (int64_t)gridDim.x * blockDim.x) {
        const int l = (int)(i / r.cstride);
        const int q = (int)(i - (int64_t)l * r.cstride);
        int j = 0;
        while (j < r.nh && q >= r.coff[j + 1]) ++j;
        const int k = q - r.coff[j];
        const int nw = r.cout[j] * r.cin[j] * r.T;
        float* P = packed + (int64_t)l * r.pstride;
        if (k < nw) {
            const int o = k / (r.cin[j] * r.T), ci = (k / r.T) % r.cin[j], t = k % r.T;
            P[r.woff[j] + ((int64_t)t * r.cin[j] + ci) * r.cop[j] + o] = canon[i];
        } else {
            P[r.boff[j] + (k - nw)] = canon[i];
        }
    }
}

VarRepack repack_plan(const gf_flow* f) {
    VarRepack r;
    std::memset(&r, 0, sizeof(r));
    r.nh = f->n_hidden;
    r.T = f->T;
    r.n_layers = f->shape.n_layers;
    r.cstride = f->canon_stride;
    r.pstride = f->vstride;
    int32_t c = 0;
    for (int j = 0; j <= f->n_hidden; ++j) {
        r.coff[j] = c;
        r.cin[j] = f->vcin[j];
        r.cout[j] = f->vcout[j];
        r.cop[j] = f->vcop[j];
        r.woff[j] = f->vwoff[j];
        r.boff[j] = f->vboff[j];
        c += r.cout[j] * r.cin[j] * r.T + r.cout[j];
    }
    r.coff[f->n_hidden + 1] = c;
    return r;
}

constexpr size_t kBudget = 227 * 1024;

// Shared memory of the staged form with `stage` floats per stage (16-byte
// aligned offsets), and its layout.
size_t staged_smem(const gf_flow* f, int stage, VarArgs* a) {
    int cop = 4;
    for (int j = 0; j <= f->n_hidden; ++j) cop = std::max(cop, f->vcop[j]);
    const int at = (int)((f->smem_bytes / 4 + 3) & ~size_t(3)), each = stage + cop;
    if (a) { a->off_stage = at; a->stage = stage; a->stage_stride = each; }
    return (size_t)(at + 2 * each) * 4;
}

template <int ND, int NSMAX, bool STAGED>
gf_status launch_v(const gf_flow* f, const VarArgs& a, bool inverse, size_t smem, int threads, int per_sm,
                   cudaStream_t stream) {
    auto kern = flow_variant_kernel<ND, NSMAX, STAGED>;
    if (cudaFuncSetAttribute(kern, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem) != cudaSuccess)
        return GF_ECUDA;
    const int64_t grid = std::min<int64_t>(a.B, (int64_t)num_sms() * per_sm);
    if (grid <= 0) return GF_OK;
    kern<<<(unsigned)grid, threads, smem, stream>>>(a, inverse ? 1 : 0);
    GF_CHECK_LAUNCH();
    return GF_OK;
}

}  // namespace

// Plans the variant network: packed offsets, shared-memory size and block size.
gf_status variant_configure(gf_flow* f) {
    const int nh = f->n_hidden;
    int cmax = 1;
    int64_t off = 0;
    for (int j = 0; j <= nh; ++j) {
        f->vcin[j] = j == 0 ? 1 : f->hidden[j - 1];
        f->vcout[j] = j == nh ? 2 : f->hidden[j];
        f->vcop[j] = (f->vcout[j] + 3) & ~3;
        f->vwoff[j] = (int32_t)off;
        off += (int64_t)f->T * f->vcin[j] * f->vcop[j];
        f->vboff[j] = (int32_t)off;
        off += f->vcop[j];
        if (j < nh) cmax = std::max(cmax, f->hidden[j]);
    }
    f->vstride = (off + 3) & ~int64_t(3);
    f->Cp = nh == 0 ? 1 : (cmax | 1);
    const size_t Vpad = (f->V + 3) & ~3;
    const size_t floats = ((Vpad + 2 * (size_t)f->V * f->Cp + 1) & ~size_t(1)) + 2 * 32;
    f->smem_bytes = floats * 4;
    if (f->smem_bytes > kBudget) return GF_EUNSUPPORTED;
    // threads: enough for the widest conv's (site, channel-group) items, 64..256
    int items = f->V / 2;
    for (int j = 0; j < nh; ++j) items = std::max(items, f->V * ((f->vcop[j] + 7) / 8));
    f->vthreads = std::max(64, std::min(256, (items + 31) & ~31));
    return GF_OK;
}

gf_status repack_variant(gf_flow* f, cudaStream_t stream) {
    const VarRepack r = repack_plan(f);
    const int64_t total = f->n_params;
    if (total == 0) return GF_OK;
    const int grid = (int)std::min<int64_t>((total + 255) / 256, 4096);
    repack_variant_kernel<<<grid, 256, 0, stream>>>(f->d_canon, f->d_vpacked, r);
    GF_CHECK_LAUNCH();
    return GF_OK;
}

gf_status launch_flow_variant(const gf_flow* f, bool inverse, const gf_phi4* phi4, int64_t B,
                              uint64_t seed, uint64_t counter0, const float* z_in, float* z_out,
                              const float* phi_in, float* phi_out, double* logq_out,
                              double* S_out, double* logw_out, cudaStream_t stream) {
    VarArgs a;
    std::memset(&a, 0, sizeof(a));
    a.W = f->d_vpacked;
    a.stride = f->vstride;
    for (int j = 0; j <= f->n_hidden; ++j) {
        a.woff[j] = f->vwoff[j];
        a.boff[j] = f->vboff[j];
        a.cin[j] = f->vcin[j];
        a.cout[j] = f->vcout[j];
        a.cop[j] = f->vcop[j];
    }
    a.nh = f->n_hidden;
    a.K = f->K;
    a.L = f->shape.L;
    a.V = f->V;
    a.Cp = f->Cp;
    a.n_layers = f->shape.n_layers;
    a.slope = (float)f->shape.leaky_slope;
    a.use_tanh = f->shape.use_final_tanh;
    a.has_phi4 = phi4 != nullptr;
    ff_split(2.0 * f->shape.nd + (phi4 ? phi4->m2 : 0.0), &a.c2d_ff.hi, &a.c2d_ff.lo);
    ff_split(phi4 ? phi4->lam : 0.0, &a.lam_ff.hi, &a.lam_ff.lo);
    a.B = B;
    a.seed = seed;
    a.counter0 = counter0;
    a.z_in = z_in; a.z_out = z_out; a.phi_in = phi_in; a.phi_out = phi_out;
    a.logq_out = logq_out; a.S_out = S_out; a.logw_out = logw_out;

    // Stages of 8 KB, or less where that is all that fits; none: weights through L1.
    int cop = 4, longest = 0;
    for (int j = 0; j <= f->n_hidden; ++j) {
        cop = std::max(cop, f->vcop[j]);
        longest = std::max(longest, f->T * f->vcin[j] * f->vcop[j]);
    }
    size_t smem = f->smem_bytes;
    bool staged = false;
    for (int stage : {2048, 1024, 512}) {
        stage = std::min(stage, longest);
        if (stage < cop || staged_smem(f, stage, nullptr) > kBudget) continue;
        smem = staged_smem(f, stage, &a);
        staged = true;
        break;
    }
    a.vt = f->vthreads;
    for (int j = 0; j <= f->n_hidden; ++j) {
        const int total = f->T * f->vcin[j];
        int n = 1;                                         // equal chunks
        if (staged) n = (total + a.stage / f->vcop[j] - 1) / (a.stage / f->vcop[j]);
        a.rows[j] = (total + n - 1) / n;
    }
    // CTA size and sites per thread (at most 4 with 128 registers to a thread, 2
    // with 80): those that finish the batch soonest, estimated in cycles of a
    // layer on an SM of r CTAs as what one CTA alone takes (a row, one input channel
    // of one tap, takes a warp 4 + 7 ns issue slots or 8 ns cycles of its
    // scheduler's FMA pipe; a pass no less than its latencies, 24 cycles a row and 60
    // a tap; 400 for every barrier) plus the others' issue time.  Fitted to 27
    // networks at 37 to 8000 configurations: the pick is mostly within 5 % of the
    // best, at worst 12 % (2D L = 16, widths 16, 16, 8, 5 taps: 256 threads 1820 us,
    // 128 threads 1310, 64 threads 1690 for 500).
    const int64_t sms = num_sms(), by_smem = (int64_t)(228 * 1024 / (smem + 1024));
    double best = 0;
    int threads = 0, nsmax = 0, per_sm = 1;
    for (int most : {staged ? 2 : 4, 4})              // (without stages the buffers leave room for one CTA)
        for (int nt : {64, 128, 256}) {
            nt = std::min(nt, f->vthreads);
            const int64_t fit = std::max<int64_t>(1, std::min<int64_t>(by_smem, 65536 / ((most == 4 ? 128 : 80) * nt)));
            const int64_t r = std::max<int64_t>(1, std::min((B + sms - 1) / sms, fit));
            double lat = 0, eff = 0;
            int32_t ns[GF_MAX_HIDDEN + 1];
            for (int j = 0; j <= f->n_hidden; ++j) {
                const bool head = j == f->n_hidden;
                const int groups = (f->vcop[j] + 7) / 8, items = head ? f->V / 2 : f->V * groups;
                ns[j] = 1;
                if (head) ns[j] = items >= 4 * f->vthreads ? 4 : items > f->vthreads ? 2 : 1;
                if (!head && items / 2 >= nt) ns[j] = 2;
                if (!head && most == 4 && items / 4 >= nt && (f->shape.nd == 3 || f->shape.L % 4 == 0)) ns[j] = 4;
                const int tasks = (items / ns[j] + 31) / 32, warps = nt / 32, total = f->T * f->vcin[j];
                const double c = head ? 4.0 + 4.0 * ns[j] : std::max(8.0 * ns[j], 4.0 + 7.0 * ns[j]);
                const double tap = f->T * (20.0 + 5.0 * ns[j]);
                eff += tasks / 4.0 * (c * total + tap);
                const double issue = (c + 3.0 * ns[j]) * total + tap, stall = 24.0 * total + 60.0 * f->T;
                for (int left = tasks; left > 0; left -= warps)
                    lat += std::max((std::min(left, warps) + 3) / 4 * issue, issue + stall) +
                           400.0 * (total + a.rows[j] - 1) / a.rows[j];
            }
            const double cost = (double)((B + sms * r - 1) / (sms * r)) * (lat + (r - 0.5) * eff);
            if (threads && cost >= best) continue;
            best = cost; threads = nt; nsmax = most; per_sm = (int)fit;
            std::copy(ns, ns + f->n_hidden + 1, a.ns);
        }
    const auto go = [&](auto nd) -> gf_status {
        constexpr int ND = decltype(nd)::value;
        if (!staged) return launch_v<ND, 4, false>(f, a, inverse, smem, threads, per_sm, stream);
        return nsmax == 4 ? launch_v<ND, 4, true>(f, a, inverse, smem, threads, per_sm, stream)
                          : launch_v<ND, 2, true>(f, a, inverse, smem, threads, per_sm, stream);
    };
    return f->shape.nd == 3 ? go(std::integral_constant<int, 3>()) : go(std::integral_constant<int, 2>());
}

}  // namespace gf
