// gf_train.cu -- reverse-KL self-training step of the coupling stack.
//
// Paper arXiv:2208.08903 Sec. 1 (shifted reverse Kullback-Leibler divergence
// as the training objective) and Sec. 3 (training loop: sample z from the
// prior, gradient of the loss, Adam update).  Loss per configuration:
// log q(phi) + S(phi) = log r(z) - sum_l sum_{updated} s + S(F^{-1}(z)),
// differentiated by a hand-written reverse pass:
//   forward  : the fused FP32 kernel over all layers, saving each layer's input
//              x_l (layer by layer where `layerwise` says so)
//   backward : per layer (last first) recompute h1, h2, s from x_l, then
//              affine adjoint -> conv3^T -> LReLU' -> conv2^T -> LReLU'
//              -> conv1^T onto the fixed sites, and the weight gradients
//              (gf_train_bwd.cuh).
// Activations go through HBM in a channel-chunk-major layout,
// [B][C/4][V][4] FP32 (chunk width min(C, 4)), so that lanes working on
// consecutive sites load consecutive 16-byte words; the step is bound by FP32
// FMA throughput and the extra traffic is a few percent of its time.  Weight
// gradients: each CTA accumulates its configurations in registers and
// writes a partial; one kernel per layer sums the partials of its three
// convolutions in a fixed order (deterministic, no atomics).
#include <algorithm>
#include <cstring>

#include "gf_flow.cuh"
#include "gf_train_bwd.cuh"

namespace gf {
namespace {

constexpr int kThreads = 256;

__device__ __forceinline__ int wrapi(int v, int L) { return v < 0 ? v + L : (v >= L ? v - L : v); }
__device__ __forceinline__ float lrelu(float v, float a) { return v > 0.f ? v : a * v; }

template <int ND>
__device__ __forceinline__ void tap_delta(int t, int& ds, int& dy, int& dx) {
    if (ND == 3) { ds = t / 9 - 1; dy = (t / 3) % 3 - 1; dx = t % 3 - 1; }
    else { ds = t / 3 - 1; dy = 0; dx = t % 3 - 1; }
}

// Site n + delta(t) on the periodic lattice (n = x + L*(y + L*z)).
template <int ND>
__device__ __forceinline__ int nbr(int n, int t, int L) {
    int ds, dy, dx;
    tap_delta<ND>(t, ds, dy, dx);
    const int x = n % L;
    if (ND == 3) {
        const int y = (n / L) % L, z = n / (L * L);
        return (wrapi(z + ds, L) * L + wrapi(y + dy, L)) * L + wrapi(x + dx, L);
    }
    const int y = n / L;
    return wrapi(y + ds, L) * L + wrapi(x + dx, L);
}

template <int ND>
__device__ __forceinline__ int parity(int n, int L) {
    const int x = n % L, y = (n / L) % L;
    return (ND == 3 ? (x + y + n / (L * L)) : (x + y)) & 1;
}

// Element (b, n, c) of a C-channel activation tensor: chunk width W = min(C, 4),
// offset ((b * (C / W) + c / W) * V + n) * W + c % W.  This returns the start of
// chunk c / W (c a multiple of W).
__device__ __forceinline__ int64_t chunk_at(int64_t b, int n, int c, int C, int V) {
    const int W = C < 4 ? C : 4;
    return ((b * (C / W) + c / W) * (int64_t)V + n) * W;
}

// ------------------------------------------------------------------ prior
__global__ void k_prior(int V, int64_t B, uint64_t seed, uint64_t counter0, const float* __restrict__ zin,
                        float* __restrict__ z) {
    const int64_t groups = (int64_t)B * ((V + 3) / 4);
    for (int64_t g = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; g < groups;
         g += (int64_t)gridDim.x * blockDim.x) {
        const int64_t b = g / ((V + 3) / 4);
        const int j = (int)(g - b * ((V + 3) / 4));
        if (zin) {
            for (int q = 0; q < 4 && 4 * j + q < V; ++q) z[b * V + 4 * j + q] = zin[b * V + 4 * j + q];
            continue;
        }
        const u64x4 w = philox4x64_10(seed, 0ull, u64x4{counter0 + (uint64_t)b, (uint64_t)j, 0ull, TAG_PRIOR});
        float zz[4];
        normals4_f32(w, zz);
        for (int q = 0; q < 4 && 4 * j + q < V; ++q) z[b * V + 4 * j + q] = zz[q];
    }
}

// ------------------------------------------------------------------ generic periodic conv
// out(b, n, co..co+8) = LReLU( bias + sum_t sum_ci W[t][ci][co] * in'(b, nbr(n,t), ci) )
// in' = in, or in masked to sites of parity `mask` (mask >= 0).
// Warp task = (configuration, 128 sites, 8 output channels); lane owns sites
// lane + 32k (k < 4).  The conv's weights [T][Cin][Cout] are staged in shared
// memory once per CTA (warp-uniform broadcast reads).
struct ConvArgs {
    const float* in; int Cin; int mask;
    const float* W; const float* bias; int Cout;
    float* out; float slope;
    int L, V; int64_t B;
};

template <int ND, int VEC, bool MASKED>
__global__ void __launch_bounds__(kThreads) k_conv(const ConvArgs a) {
    extern __shared__ __align__(16) float wsm[];
    const int T = ND == 3 ? 27 : 9;
    {
        const int n4 = T * a.Cin * a.Cout / 4;
        for (int i = threadIdx.x; i < n4; i += blockDim.x)
            reinterpret_cast<float4*>(wsm)[i] = __ldg(reinterpret_cast<const float4*>(a.W) + i);
        __syncthreads();
    }
    const int lane = threadIdx.x & 31;
    const int nblk = (a.V + 127) >> 7, ngrp = a.Cout >> 3;
    const int64_t tasks = a.B * nblk * ngrp;
    const int64_t cstride = (int64_t)a.V * VEC;            // floats between input chunks
    for (int64_t task = (blockIdx.x * (int64_t)blockDim.x + threadIdx.x) >> 5; task < tasks;
         task += ((int64_t)gridDim.x * blockDim.x) >> 5) {
        const int g = (int)(task % ngrp);
        const int64_t rest = task / ngrp;
        const int blk = (int)(rest % nblk);
        const int64_t b = rest / nblk;
        const int co = g << 3;
        int n[4];
        bool valid[4];
#pragma unroll
        for (int k = 0; k < 4; ++k) {
            n[k] = (blk << 7) + lane + 32 * k;
            valid[k] = n[k] < a.V;
            if (!valid[k]) n[k] = a.V - 1;
        }
        float acc[4][8];
#pragma unroll
        for (int k = 0; k < 4; ++k)
#pragma unroll
            for (int c = 0; c < 8; ++c) acc[k][c] = __ldg(a.bias + co + c);
        const float* inb = a.in + chunk_at(b, 0, 0, a.Cin, a.V);
        for (int t = 0; t < T; ++t) {
            int m[4];
            float msk[4];
#pragma unroll
            for (int k = 0; k < 4; ++k) {
                m[k] = nbr<ND>(n[k], t, a.L);
                msk[k] = (!MASKED || parity<ND>(m[k], a.L) == a.mask) ? 1.f : 0.f;
            }
            const float* Wt = wsm + t * a.Cin * a.Cout + co;
            for (int c0 = 0; c0 < a.Cin; c0 += VEC) {
                float hv[4][VEC];
                const float* pc = inb + (int64_t)(c0 / VEC) * cstride;
#pragma unroll
                for (int k = 0; k < 4; ++k) {
                    const float* p = pc + (int64_t)m[k] * VEC;
                    if (VEC == 4) {
                        const float4 v = __ldg(reinterpret_cast<const float4*>(p));
                        hv[k][0] = v.x; hv[k][VEC > 1 ? 1 : 0] = v.y;
                        hv[k][VEC > 2 ? 2 : 0] = v.z; hv[k][VEC > 3 ? 3 : 0] = v.w;
                    } else {
                        hv[k][0] = __ldg(p);
                    }
                    if constexpr (MASKED) {
#pragma unroll
                        for (int q = 0; q < VEC; ++q) hv[k][q] *= msk[k];
                    }
                }
#pragma unroll
                for (int q = 0; q < VEC; ++q) {
                    const float* wp = Wt + (c0 + q) * a.Cout;
                    const float4 wa = *reinterpret_cast<const float4*>(wp);
                    const float4 wb = *reinterpret_cast<const float4*>(wp + 4);
#pragma unroll
                    for (int k = 0; k < 4; ++k) {
                        const float h = hv[k][q];
                        acc[k][0] = fmaf(h, wa.x, acc[k][0]); acc[k][1] = fmaf(h, wa.y, acc[k][1]);
                        acc[k][2] = fmaf(h, wa.z, acc[k][2]); acc[k][3] = fmaf(h, wa.w, acc[k][3]);
                        acc[k][4] = fmaf(h, wb.x, acc[k][4]); acc[k][5] = fmaf(h, wb.y, acc[k][5]);
                        acc[k][6] = fmaf(h, wb.z, acc[k][6]); acc[k][7] = fmaf(h, wb.w, acc[k][7]);
                    }
                }
            }
        }
#pragma unroll
        for (int k = 0; k < 4; ++k) {
            if (!valid[k]) continue;
            float* o0 = a.out + chunk_at(b, n[k], co, a.Cout, a.V);
            float* o1 = a.out + chunk_at(b, n[k], co + 4, a.Cout, a.V);
            float r[8];
#pragma unroll
            for (int c = 0; c < 8; ++c) r[c] = lrelu(acc[k][c], a.slope);
            *reinterpret_cast<float4*>(o0) = make_float4(r[0], r[1], r[2], r[3]);
            *reinterpret_cast<float4*>(o1) = make_float4(r[4], r[5], r[6], r[7]);
        }
    }
}

// ------------------------------------------------------------------ conv3 + affine (forward)
// One CTA per configuration: (s, t) at the updated sites, x_out = x_in*e^s + t
// there, x_out = x_in on fixed sites; s saved for the reverse pass;
// logdet[b] += sum s (FP64, fixed-order block reduction) unless logdet is null
// (then a configuration may be split over gridDim.y CTAs).  PARTS: the threads'
// sums run on over the layers in part[b][kThreads] (from zero at layer 0) and
// logdet[b] is their sum after the last one: the order of the fused forward pass.
template <int ND, bool PARTS>
__global__ void __launch_bounds__(kThreads) k_couple_fwd(const float* __restrict__ h2, int C2,
                                                        const float* __restrict__ W3, const float* __restrict__ b3,
                                                        int use_tanh, int frozen, int L, int V, int64_t B,
                                                        const float* __restrict__ xin, float* __restrict__ xout,
                                                        float* __restrict__ s_save, double* __restrict__ logdet,
                                                        double* __restrict__ part, int layer, int n_layers) {
    __shared__ double red[32];
    const int T = ND == 3 ? 27 : 9;
    for (int64_t b = blockIdx.x; b < B; b += gridDim.x) {
        double ld = PARTS && layer > 0 ? part[b * kThreads + threadIdx.x] : 0.0;
        for (int n = blockIdx.y * blockDim.x + threadIdx.x; n < V; n += blockDim.x * gridDim.y) {
            const float xv = xin[b * V + n];
            if (parity<ND>(n, L) == frozen) { xout[b * V + n] = xv; s_save[b * V + n] = 0.f; continue; }
            float ps = __ldg(b3), pt = __ldg(b3 + 1);
            for (int t = 0; t < T; ++t) {
                const int m = nbr<ND>(n, t, L);
                const float* wp = W3 + (int64_t)t * C2 * 2;
                for (int c = 0; c < C2; c += 4) {
                    const float4 h = __ldg(reinterpret_cast<const float4*>(h2 + chunk_at(b, m, c, C2, V)));
                    const float4 w01 = __ldg(reinterpret_cast<const float4*>(wp + 2 * c));
                    const float4 w23 = __ldg(reinterpret_cast<const float4*>(wp + 2 * c + 4));
                    ps = fmaf(h.x, w01.x, ps); pt = fmaf(h.x, w01.y, pt);
                    ps = fmaf(h.y, w01.z, ps); pt = fmaf(h.y, w01.w, pt);
                    ps = fmaf(h.z, w23.x, ps); pt = fmaf(h.z, w23.y, pt);
                    ps = fmaf(h.w, w23.z, ps); pt = fmaf(h.w, w23.w, pt);
                }
            }
            const float s = use_tanh ? tanhf(ps) : ps;
            xout[b * V + n] = fmaf(xv, expf(s), pt);
            s_save[b * V + n] = s;
            ld += (double)s;
        }
        if (PARTS) part[b * kThreads + threadIdx.x] = ld;
        if (logdet && (!PARTS || layer == n_layers - 1)) {   // uniform over the block
            const double tot = block_sum(ld, red);
            if (threadIdx.x == 0) logdet[b] = PARTS ? tot : logdet[b] + tot;
        }
        __syncthreads();
    }
}

// ------------------------------------------------------------------ affine adjoint
// At updated sites: g3 = (dL/ds_pre, dL/dt), gx <- gx*e^s.  Fixed sites: g3 = 0.
template <int ND>
__global__ void k_couple_bwd(int frozen, int use_tanh, int L, int V, int64_t B, const float* __restrict__ xin,
                             const float* __restrict__ s_save, const double* __restrict__ glq, float glq_const,
                             float* __restrict__ gx, float* __restrict__ g3) {
    const int64_t total = B * (int64_t)V;
    for (int64_t i = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; i < total;
         i += (int64_t)gridDim.x * blockDim.x) {
        const int n = (int)(i % V);
        float2 o = make_float2(0.f, 0.f);
        if (parity<ND>(n, L) != frozen) {
            const float s = s_save[i], e = expf(s), g = gx[i];
            // d/ds of x*e^s, and of log q = log r - logdet (dLoss/dlog q per configuration)
            const float gq = glq ? (float)glq[i / V] : glq_const;
            const float gs = g * xin[i] * e - gq;
            o.x = use_tanh ? gs * (1.f - s * s) : gs;
            o.y = g;
            gx[i] = g * e;
        }
        reinterpret_cast<float2*>(g3)[i] = o;
    }
}

// ------------------------------------------------------------------ weight gradients (gf_train_bwd.cuh)
// Partial sums [part][T + 1][Cin][Cout] (tap T: the bias, i = 0) of the three
// convolutions of a layer -> their canonical gradients W[o][i][t] and b[o], times
// scale, in one launch.
struct ReduceSet {
    const float* partial;
    int nparts, Cin, Cout, blocks;
    float *gW, *gb;
};
struct ReduceArgs {
    ReduceSet set[3];
    int T;
    float scale;
};
__global__ void __launch_bounds__(256) k_wgrad_reduce(const __grid_constant__ ReduceArgs a) {
    // block = 32 outputs (lane); its 8 warps sum interleaved eighths of the
    // partials, combined in warp order (fixed: deterministic)
    __shared__ float part[8][32];
    int blk = blockIdx.x, i = 0;               // (unused sets have no blocks)
    while (i < 2 && blk >= a.set[i].blocks) blk -= a.set[i++].blocks;
    const ReduceSet& s = a.set[i];
    const int per = (a.T + 1) * s.Cin * s.Cout;
    const int lane = threadIdx.x & 31, wid = threadIdx.x >> 5;
    const int p = blk * 32 + lane;
    float sum = 0.f;
    if (p < per)
        for (int k = wid; k < s.nparts; k += 8) sum += s.partial[(int64_t)k * per + p];
    part[wid][lane] = sum;
    __syncthreads();
    if (wid == 0 && p < per) {
        float t = 0.f;
        for (int w = 0; w < 8; ++w) t += part[w][lane];
        const int o = p % s.Cout, c = (p / s.Cout) % s.Cin, tt = p / (s.Cout * s.Cin);
        if (tt < a.T) s.gW[((int64_t)o * s.Cin + c) * a.T + tt] = t * a.scale;
        else if (c == 0) s.gb[o] = t * a.scale;
    }
}

// ------------------------------------------------------------------ loss, force
// loss_b = log r(z_b) - logdet_b + S(phi_b); gx = dS/dphi (FP64 terms, FP32 out).
template <int ND>
__global__ void __launch_bounds__(kThreads) k_loss_force(const float* __restrict__ z, const float* __restrict__ phi,
                                                        const double* __restrict__ logdet, double m2, double lam,
                                                        int L, int V, int64_t B, double* __restrict__ loss_b,
                                                        float* __restrict__ gx) {
    __shared__ double red[32];
    for (int64_t b = blockIdx.x; b < B; b += gridDim.x) {
        const float* p = phi + b * V;
        double acc = 0.0, z2 = 0.0;
        for (int n = threadIdx.x; n < V; n += blockDim.x) {
            const double c = p[n];
            acc += c * lap_minus(p, n, ND, L) + m2 * c * c + lam * c * c * c * c;
            gx[b * V + n] = (float)phi4_force_site(p, n, ND, L, m2, lam);
            const double zz = z[b * V + n];
            z2 += zz * zz;
        }
        const double S = block_sum(acc, red);
        const double Z2 = block_sum(z2, red);
        if (threadIdx.x == 0) loss_b[b] = (-0.5 * Z2 - 0.5 * (double)V * LOG_2PI) - logdet[b] + S;
        __syncthreads();
    }
}

__global__ void k_mean(const double* __restrict__ v, int64_t n, double* __restrict__ out) {
    __shared__ double red[32];
    double s = 0.0;
    for (int64_t i = threadIdx.x; i < n; i += blockDim.x) s += v[i];
    s = block_sum(s, red);
    if (threadIdx.x == 0) *out = s / (double)n;
}

// ------------------------------------------------------------------ unfused sampler epilogue
// log r(z), S(phi) (FP64 site terms), log q = log r - logdet, log w = -S - log q.
template <int ND>
__global__ void __launch_bounds__(kThreads) k_finish(const float* __restrict__ z, const float* __restrict__ phi,
                                                    const double* __restrict__ logdet, int has_phi4, double m2,
                                                    double lam, int L, int V, int64_t B, float* __restrict__ phi_out,
                                                    float* __restrict__ z_out, double* __restrict__ logq,
                                                    double* __restrict__ S_out, double* __restrict__ logw) {
    __shared__ double red[32];
    for (int64_t b = blockIdx.x; b < B; b += gridDim.x) {
        const float* p = phi + b * V;
        double acc = 0.0, z2 = 0.0;
        for (int n = threadIdx.x; n < V; n += blockDim.x) {
            const double c = p[n];
            if (has_phi4) {
                double k = 0.0;
                for (int mu = 0; mu < ND; ++mu) {
                    const int t_plus = (mu == 0) ? (ND == 3 ? 14 : 5) : (mu == 1) ? (ND == 3 ? 16 : 7) : 22;
                    const int t_minus = (ND == 3 ? 26 : 8) - t_plus;
                    k += 2.0 * c - (double)p[nbr<ND>(n, t_plus, L)] - (double)p[nbr<ND>(n, t_minus, L)];
                }
                acc += c * k + m2 * c * c + lam * c * c * c * c;
            }
            const double zz = z[b * V + n];
            z2 += zz * zz;
            phi_out[b * V + n] = p[n];
            if (z_out) z_out[b * V + n] = z[b * V + n];
        }
        const double S = block_sum(acc, red);
        const double Z2 = block_sum(z2, red);
        if (threadIdx.x == 0) {
            const double lq = (-0.5 * Z2 - 0.5 * (double)V * LOG_2PI) - logdet[b];
            logq[b] = lq;
            if (has_phi4 && S_out) S_out[b] = S;
            if (has_phi4 && logw) logw[b] = -S - lq;
        }
        __syncthreads();
    }
}

// ------------------------------------------------------------------ weights for the reverse pass
// Transposed + tap-flipped copies: Wb[t][o][i] = W[o][i][T-1-t] (delta(T-1-t) = -delta(t)).
__global__ void k_pack_bwd(const float* __restrict__ canon, int64_t cstride, int n_layers, int T, int C1, int C2,
                           float* __restrict__ out, int64_t ostride) {
    const int64_t total = (int64_t)n_layers * ostride;
    const int64_t n1 = (int64_t)T * C1, n2 = (int64_t)T * C2 * C1, n3 = (int64_t)T * 2 * C2;
    for (int64_t i = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; i < total;
         i += (int64_t)gridDim.x * blockDim.x) {
        const int l = (int)(i / ostride);
        int64_t r = i - l * ostride;
        const float* W = canon + l * cstride;
        float v = 0.f;
        if (r < n1) {                                    // W1b[t][c] = W1[c][0][T-1-t]
            const int t = (int)(r / C1), c = (int)(r % C1);
            v = W[(int64_t)c * T + (T - 1 - t)];
        } else if ((r -= n1) < n2) {                     // W2b[t][o][i] = W2[o][i][T-1-t]
            const int t = (int)(r / ((int64_t)C2 * C1));
            const int o = (int)((r / C1) % C2), ii = (int)(r % C1);
            v = W[n1 + C1 + ((int64_t)o * C1 + ii) * T + (T - 1 - t)];
        } else if ((r -= n2) < n3) {                     // W3b[t][o][i] = W3[o][i][T-1-t]
            const int t = (int)(r / (2 * C2));
            const int o = (int)((r / C2) % 2), ii = (int)(r % C2);
            v = W[n1 + C1 + n2 + C2 + ((int64_t)o * C2 + ii) * T + (T - 1 - t)];
        }
        out[i] = v;
    }
}

// ------------------------------------------------------------------ Adam (Kingma & Ba)
__global__ void k_adam(int64_t n, float* __restrict__ w, const float* __restrict__ g, float* __restrict__ m,
                       float* __restrict__ v, float lr, float b1, float b2, float eps, float c1, float c2) {
    for (int64_t i = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; i < n; i += (int64_t)gridDim.x * blockDim.x) {
        const float gi = g[i];
        const float mi = b1 * m[i] + (1.f - b1) * gi;
        const float vi = b2 * v[i] + (1.f - b2) * gi * gi;
        m[i] = mi;
        v[i] = vi;
        w[i] -= lr * (mi / c1) / (sqrtf(vi / c2) + eps);
    }
}

// ------------------------------------------------------------------ workspace
struct TrainWs {
    float *xs, *h1, *h2, *s, *gx, *g3, *gh2, *gh1, *wb, *partial, *grad;
    double *logdet, *loss_b;
    size_t bytes;
};

int wgrad_grid() { return num_sms() * 2; }

TrainWs carve(const gf_flow* f, int64_t B, char* base) {
    TrainWs w;
    std::memset(&w, 0, sizeof(w));
    size_t off = 0;
    auto take = [&](size_t bytes) -> char* {
        char* p = base ? base + off : nullptr;
        off += (bytes + 255) & ~size_t(255);
        return p;
    };
    const int64_t BV = B * (int64_t)f->V;
    const int N = f->shape.n_layers, C = std::max(f->C1, f->C2);
    const int64_t obstride = (int64_t)f->T * f->C1 + (int64_t)f->T * f->C2 * f->C1 + 2LL * f->T * f->C2;
    w.xs = (float*)take(sizeof(float) * BV * (N + 1));
    w.h1 = (float*)take(sizeof(float) * BV * f->C1);
    w.h2 = (float*)take(sizeof(float) * BV * f->C2);
    w.s = (float*)take(sizeof(float) * BV);
    w.gx = (float*)take(sizeof(float) * BV);
    w.g3 = (float*)take(sizeof(float) * BV * 2);
    w.gh2 = (float*)take(sizeof(float) * BV * f->C2);
    w.gh1 = (float*)take(sizeof(float) * BV * f->C1);
    w.wb = (float*)take(sizeof(float) * obstride * std::max(N, 1));
    w.partial = (float*)take(sizeof(float) * (size_t)wgrad_grid() * (f->T + 1) * C * C);
    w.grad = (float*)take(sizeof(float) * std::max<int64_t>(f->n_params, 1));
    w.logdet = (double*)take(sizeof(double) * std::max<int64_t>(B, 1));
    w.loss_b = (double*)take(sizeof(double) * std::max<int64_t>(B, 1));
    w.bytes = off;
    return w;
}

int64_t grid1d(int64_t n) { return std::max<int64_t>(1, std::min<int64_t>((n + kThreads - 1) / kThreads, (int64_t)num_sms() * 16)); }

template <int ND>
gf_status conv(const ConvArgs& a, cudaStream_t st) {
    const int64_t warps = a.B * ((a.V + 127) / 128) * (a.Cout / 8);
    const int64_t grid = std::max<int64_t>(1, std::min<int64_t>((warps + 7) / 8, (int64_t)num_sms() * 8));
    const int T = ND == 3 ? 27 : 9;
    const size_t smem = (size_t)T * a.Cin * a.Cout * sizeof(float);
    auto go = [&](auto kern) -> bool {
        if (cudaFuncSetAttribute(kern, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem) != cudaSuccess)
            return false;
        kern<<<(unsigned)grid, kThreads, smem, st>>>(a);
        return true;
    };
    bool ok;
    if (a.mask >= 0) {      // masked input (conv1 of a coupling): parity test per neighbour
        if (a.Cin % 4 == 0) ok = go(k_conv<ND, 4, true>);
        else ok = go(k_conv<ND, 1, true>);
    } else {
        if (a.Cin % 4 == 0) ok = go(k_conv<ND, 4, false>);
        else ok = go(k_conv<ND, 1, false>);
    }
    if (!ok) return GF_ECUDA;
    GF_CHECK_LAUNCH();
    return GF_OK;
}

// conv1 + LReLU and conv2 + LReLU of layer l on x_l (FP32, activations in the workspace).
template <int ND>
gf_status net_fwd(const gf_flow* f, int l, const float* xl, int64_t B, const TrainWs& w, cudaStream_t st) {
    const PackedOffsets po = packed_offsets(f->T, f->C1, f->C2);
    const float slope = (float)f->shape.leaky_slope;
    const float* P = f->d_packed + (int64_t)l * f->packed_stride;
    ConvArgs c1{xl, 1, l & 1, P + po.W1, P + po.b1, f->C1, w.h1, slope, f->shape.L, f->V, B};
    gf_status s = conv<ND>(c1, st);
    if (s != GF_OK) return s;
    ConvArgs c2{w.h1, f->C1, -1, P + po.W2, P + po.b2, f->C2, w.h2, slope, f->shape.L, f->V, B};
    return conv<ND>(c2, st);
}

// kThreads FP64 partial sums of the log-det per configuration: the forward pass
// has no use for gh1 (layer-by-layer lattices have far more than 512 values of it
// a configuration).
double* logdet_parts(const TrainWs& w) { return reinterpret_cast<double*>(w.gh1); }

// One layer forward with a kernel per convolution: h1, h2, s and the field after
// the layer (and, unless null, `logdet` after the last one).
template <int ND>
gf_status layer_fwd(const gf_flow* f, int l, int64_t B, const float* xl, float* xout, double* logdet, const TrainWs& w,
                    cudaStream_t st) {
    const gf_status s = net_fwd<ND>(f, l, xl, B, w, st);
    if (s != GF_OK) return s;
    const PackedOffsets po = packed_offsets(f->T, f->C1, f->C2);
    const float* P = f->d_packed + (int64_t)l * f->packed_stride;
    const dim3 grid((unsigned)std::min<int64_t>(B, (int64_t)num_sms() * 8), logdet ? 1u : (unsigned)((f->V + kThreads - 1) / kThreads));
    const auto kern = logdet ? k_couple_fwd<ND, true> : k_couple_fwd<ND, false>;
    kern<<<grid, kThreads, 0, st>>>(w.h2, f->C2, P + po.W3, P + po.b3, f->shape.use_final_tanh, l & 1, f->shape.L,
                                    f->V, B, xl, xout, w.s, logdet, logdet_parts(w), l, f->shape.n_layers);
    GF_CHECK_LAUNCH();
    return GF_OK;
}

// Whether training runs the network layer by layer, a kernel per convolution
// over all configurations, instead of fused with a CTA per configuration (every
// sum has one order in both, so the field, log q, loss and gradient are the same
// to the bit whichever a batch takes; the kernels of 2D L=32 and 3D L=16 with
// width 32 always run the forward pass fused): where the fused kernel has no room to stage weights,
// and for lattices that do not fit a CTA at once when the batch leaves half of
// the SMs idle (3D L=12 width 32, batch 64: 0.48 ms a layer fused).
bool layerwise(const gf_flow* f, int64_t B) {
    if (fp32_c32_recompute_supported(f)) return false;
    return f->weights_global || (!f->full && 2 * B < num_sms());
}

// Forward pass of training: z -> x_1 .. x_N saved in the workspace, logdet per
// configuration.
template <int ND>
gf_status forward_pass(const gf_flow* f, int64_t B, uint64_t seed, uint64_t counter0, const float* z_in,
                       const TrainWs& w, cudaStream_t st) {
    const int N = f->shape.n_layers;
    const int64_t BV = B * (int64_t)f->V;
    if (fp32_c32_supported(f) || !layerwise(f, B))
        // one fused launch: z (or the prior) -> every layer's input x_l and the
        // log-det, with the FP32 weights (the kernels of gf_flow_fp32_c32.cu form
        // log q too, into a scratch buffer)
        return launch_flow_fp32(f, false, nullptr, B, seed, counter0, z_in, w.xs, nullptr, w.xs + (int64_t)N * BV, w.loss_b,
                                nullptr, nullptr, st, w.xs, BV, w.logdet);
    k_prior<<<(unsigned)grid1d(BV / 4 + 1), kThreads, 0, st>>>(f->V, B, seed, counter0, z_in, w.xs);
    GF_CHECK_LAUNCH();
    if (cudaMemsetAsync(w.logdet, 0, sizeof(double) * B, st) != cudaSuccess) return GF_ECUDA;
    for (int l = 0; l < N; ++l) {
        const gf_status s = layer_fwd<ND>(f, l, B, w.xs + (int64_t)l * BV, w.xs + (int64_t)(l + 1) * BV, w.logdet, w, st);
        if (s != GF_OK) return s;
    }
    return GF_OK;
}

// Reverse pass: with w.gx = dLoss/dphi seeded and dLoss/dlog q = glq[b] (or
// glq_const when glq is null), writes dLoss/dtheta * scale to grad (canonical
// order).  Needs the x_l saved by forward_pass with the same weights.
template <int ND>
gf_status reverse_pass(const gf_flow* f, int64_t B, const double* glq, float glq_const, float scale, float* grad,
                       const TrainWs& w, cudaStream_t st) {
    const int L = f->shape.L, V = f->V, N = f->shape.n_layers, T = f->T;
    const int C1 = f->C1, C2 = f->C2;
    const int64_t BV = B * (int64_t)V;
    const float slope = (float)f->shape.leaky_slope;
    const int use_tanh = f->shape.use_final_tanh;
    const int64_t obstride = (int64_t)T * C1 + (int64_t)T * C2 * C1 + 2LL * T * C2;
    if (N > 0) {
        k_pack_bwd<<<(unsigned)grid1d(obstride * N), kThreads, 0, st>>>(f->d_canon, f->canon_stride, N, T, C1, C2,
                                                                        w.wb, obstride);
        GF_CHECK_LAUNCH();
    }
    for (int l = N - 1; l >= 0; --l) {
        const float* xl = w.xs + (int64_t)l * BV;
        const float* Wb = w.wb + (int64_t)l * obstride;
        float* G = grad + (int64_t)l * f->canon_stride;
        float* gW1 = G;
        float* gb1 = gW1 + (int64_t)C1 * T;
        float* gW2 = gb1 + C1;
        float* gb2 = gW2 + (int64_t)C2 * C1 * T;
        float* gW3 = gb2 + C2;
        float* gb3 = gW3 + 2LL * C2 * T;
        gf_status s;
        if (layerwise(f, B)) s = layer_fwd<ND>(f, l, B, xl, w.g3 /* scratch for x_out */, nullptr, w, st);
        else s = launch_recompute(f, l, B, xl, w.h1, w.h2, w.s, st);         // h1, h2, s in one launch
        if (s != GF_OK) return s;
        k_couple_bwd<ND><<<(unsigned)grid1d(BV), kThreads, 0, st>>>(l & 1, use_tanh, L, V, B, xl, w.s, glq,
                                                                   glq_const, w.gx, w.g3);
        GF_CHECK_LAUNCH();
        // The data gradients stay on `st`; the weight gradients of conv3 and
        // conv2 run on the flow's side stream as soon as their inputs exist and
        // overlap them (which fills the SMs at small batches).  The side stream
        // only reads activations and writes partial sums; the reduction waits
        // for it.
        const bwd::BwdOps ops = ND == 3 ? bwd::ops_3d(C1) : bwd::ops_2d(C1);
        bwd::BwdArgs ba;
        std::memset(&ba, 0, sizeof(ba));
        ba.L = L; ba.S = f->S; ba.V = V; ba.frozen = l & 1; ba.B = B; ba.slope = slope;
        ba.fd_S = make_fastdiv((uint32_t)f->S); ba.fd_L = make_fastdiv((uint32_t)L);
        ba.fd_Sh = make_fastdiv((uint32_t)(f->S / 2)); ba.fd_Lh = make_fastdiv((uint32_t)(L / 2));
        ba.xl = xl; ba.h1 = w.h1; ba.h2 = w.h2; ba.g3 = w.g3; ba.gh2 = w.gh2; ba.gh1 = w.gh1; ba.gx = w.gx;
        ba.W1b = Wb; ba.W2b = Wb + (int64_t)T * C1; ba.W3b = ba.W2b + (int64_t)T * C2 * C1;
        // Room for the partials of conv3 and conv1 beside conv2's: the buffers of s
        // and of the next layer's input, both used up by now, or what a small
        // batch leaves of conv2's; else (tiny lattices at some batches) the
        // three share one buffer, one after the other.
        const int np = bwd::wgrad_parts(B);
        const int64_t n1 = (int64_t)np * (T + 1) * C1, n2 = n1 * C2, n3 = 2 * n1;
        const int64_t have = (int64_t)wgrad_grid() * (T + 1) * C1 * C2;
        float *p3 = w.partial, *p1 = w.partial;
        const bool apart = n3 <= BV || n1 + n2 + n3 <= have;
        if (n3 <= BV) { p3 = w.s; p1 = w.xs + (int64_t)(l + 1) * BV; }
        else if (apart) { p3 = w.partial + n2; p1 = p3 + n3; }
        const ReduceSet sets[3] = {{w.partial, np, C1, C2, ((T + 1) * C1 * C2 + 31) / 32, gW2, gb2},
                                   {p3, np, C2, 2, ((T + 1) * C2 * 2 + 31) / 32, gW3, gb3},
                                   {p1, np, 1, C1, ((T + 1) * C1 + 31) / 32, gW1, gb1}};
        const auto reduce = [&](int first, int count) {
            ReduceArgs ra;
            std::memset(&ra, 0, sizeof(ra));
            ra.T = T; ra.scale = scale;
            int blocks = 0;
            for (int i = 0; i < count; ++i) { ra.set[i] = sets[first + i]; blocks += ra.set[i].blocks; }
            k_wgrad_reduce<<<blocks, 256, 0, st>>>(ra);
            return cudaGetLastError() == cudaSuccess;
        };
        cudaStream_t side = apart ? f->side : st;
        const auto fork = [&](cudaEvent_t e) {
            return !apart || (cudaEventRecord(e, st) == cudaSuccess && cudaStreamWaitEvent(side, e, 0) == cudaSuccess);
        };
        if (!fork(f->ev_fork[0])) return GF_ECUDA;
        ba.partial = p3;
        if ((s = ops.wgrad3(ba, side)) != GF_OK) return s;
        if (!apart && !reduce(1, 1)) return GF_ECUDA;
        if ((s = ops.back2(ba, st)) != GF_OK) return s;               // gh2, gh1
        if (!fork(f->ev_fork[1])) return GF_ECUDA;
        ba.partial = w.partial;
        if ((s = ops.wgrad2(ba, side)) != GF_OK) return s;
        if (!apart && !reduce(0, 1)) return GF_ECUDA;
        ba.partial = p1;
        if ((s = ops.back1(ba, st)) != GF_OK) return s;               // gx
        if (apart && (cudaEventRecord(f->ev_join, side) != cudaSuccess || cudaStreamWaitEvent(st, f->ev_join, 0) != cudaSuccess))
            return GF_ECUDA;
        if (!reduce(apart ? 0 : 2, apart ? 3 : 1)) return GF_ECUDA;
    }
    return GF_OK;
}

template <int ND>
gf_status train_step(gf_flow* f, const gf_phi4* phi4, int64_t B, uint64_t seed, uint64_t counter0,
                     const float* z_in, double* loss_out, float* grad_out, float lr, float beta1,
                     float beta2, float adam_eps, float* adam_m, float* adam_v, int64_t adam_t,
                     const TrainWs& w, cudaStream_t st) {
    const int L = f->shape.L, V = f->V, N = f->shape.n_layers;
    const int64_t BV = B * (int64_t)V;
    float* grad = grad_out ? grad_out : w.grad;
    gf_status s = forward_pass<ND>(f, B, seed, counter0, z_in, w, st);
    if (s != GF_OK) return s;
    const unsigned cfg_grid = (unsigned)std::min<int64_t>(B, (int64_t)num_sms() * 8);
    // per-configuration loss log r - logdet + S and the seed dS/dphi; the loss
    // is the mean, so every configuration's gradient is scaled by 1/B
    k_loss_force<ND><<<cfg_grid, kThreads, 0, st>>>(w.xs, w.xs + (int64_t)N * BV, w.logdet, phi4->m2, phi4->lam,
                                                    L, V, B, w.loss_b, w.gx);
    GF_CHECK_LAUNCH();
    k_mean<<<1, kThreads, 0, st>>>(w.loss_b, B, loss_out);
    GF_CHECK_LAUNCH();
    if ((s = reverse_pass<ND>(f, B, nullptr, 1.0f, 1.0f / (float)B, grad, w, st)) != GF_OK) return s;
    if (lr > 0.f) {
        const float c1 = 1.f - powf(beta1, (float)adam_t), c2 = 1.f - powf(beta2, (float)adam_t);
        k_adam<<<(unsigned)grid1d(f->n_params), kThreads, 0, st>>>(f->n_params, f->d_canon, grad, adam_m, adam_v,
                                                                    lr, beta1, beta2, adam_eps, c1, c2);
        GF_CHECK_LAUNCH();
        return repack_weights(f, st);
    }
    return GF_OK;
}

// Forward half for autograd: phi = x_N and log q = log r(z) - logdet.
template <int ND>
gf_status forward_train(const gf_flow* f, int64_t B, uint64_t seed, uint64_t counter0, const float* z_in,
                        float* phi_out, double* logq_out, const TrainWs& w, cudaStream_t st) {
    gf_status s = forward_pass<ND>(f, B, seed, counter0, z_in, w, st);
    if (s != GF_OK) return s;
    const int64_t BV = B * (int64_t)f->V;
    const unsigned cfg_grid = (unsigned)std::min<int64_t>(B, (int64_t)num_sms() * 8);
    k_finish<ND><<<cfg_grid, kThreads, 0, st>>>(w.xs, w.xs + (int64_t)f->shape.n_layers * BV, w.logdet, 0, 0.0,
                                               0.0, f->shape.L, f->V, B, phi_out, nullptr, logq_out, nullptr,
                                               nullptr);
    GF_CHECK_LAUNCH();
    return GF_OK;
}

// Backward half: gx <- dLoss/dphi (zero when null), then the reverse pass.
template <int ND>
gf_status backward(const gf_flow* f, int64_t B, const float* gphi, const double* glogq, float* grad,
                   const TrainWs& w, cudaStream_t st) {
    const size_t bytes = sizeof(float) * (size_t)B * f->V;
    const cudaError_t e = gphi ? cudaMemcpyAsync(w.gx, gphi, bytes, cudaMemcpyDeviceToDevice, st)
                               : cudaMemsetAsync(w.gx, 0, bytes, st);
    if (e != cudaSuccess) return GF_ECUDA;
    return reverse_pass<ND>(f, B, glogq, 0.0f, 1.0f, grad, w, st);
}

// Unfused FP32 sampler: one kernel per convolution, activations through HBM.
// Workspace: z, two x buffers, h1, h2, s [B][V](x C), logdet [B].
struct PlainWs { float *z, *xa, *xb, *h1, *h2, *s; double* logdet; size_t bytes; };

PlainWs carve_plain(const gf_flow* f, int64_t B, char* base) {
    PlainWs w;
    size_t off = 0;
    auto take = [&](size_t bytes) -> char* {
        char* p = base ? base + off : nullptr;
        off += (bytes + 255) & ~size_t(255);
        return p;
    };
    const int64_t BV = B * (int64_t)f->V;
    w.z = (float*)take(sizeof(float) * BV);
    w.xa = (float*)take(sizeof(float) * BV);
    w.xb = (float*)take(sizeof(float) * BV);
    w.h1 = (float*)take(sizeof(float) * BV * f->C1);
    w.h2 = (float*)take(sizeof(float) * BV * f->C2);
    w.s = (float*)take(sizeof(float) * BV);
    w.logdet = (double*)take(sizeof(double) * std::max<int64_t>(B, 1));
    w.bytes = off;
    return w;
}

template <int ND>
gf_status sample_unfused(const gf_flow* f, const gf_phi4* phi4, int64_t B, uint64_t seed, uint64_t counter0,
                         const float* z_in, float* z_out, float* phi_out, double* logq, double* S_out,
                         double* logw, const PlainWs& w, cudaStream_t st) {
    const int L = f->shape.L, V = f->V, N = f->shape.n_layers;
    const int C1 = f->C1, C2 = f->C2;
    const int64_t BV = B * (int64_t)V;
    const float slope = (float)f->shape.leaky_slope;
    const PackedOffsets po = packed_offsets(f->T, C1, C2);
    k_prior<<<(unsigned)grid1d(BV / 4 + 1), kThreads, 0, st>>>(V, B, seed, counter0, z_in, w.z);
    GF_CHECK_LAUNCH();
    if (cudaMemsetAsync(w.logdet, 0, sizeof(double) * B, st) != cudaSuccess) return GF_ECUDA;
    const unsigned cfg_grid = (unsigned)std::min<int64_t>(B, (int64_t)num_sms() * 8);
    const float* xin = w.z;
    float* bufs[2] = {w.xa, w.xb};
    for (int l = 0; l < N; ++l) {
        const float* P = f->d_packed + (int64_t)l * f->packed_stride;
        ConvArgs c1{xin, 1, l & 1, P + po.W1, P + po.b1, C1, w.h1, slope, L, V, B};
        gf_status s = conv<ND>(c1, st);
        if (s != GF_OK) return s;
        ConvArgs c2{w.h1, C1, -1, P + po.W2, P + po.b2, C2, w.h2, slope, L, V, B};
        if ((s = conv<ND>(c2, st)) != GF_OK) return s;
        float* xout = bufs[l & 1];
        k_couple_fwd<ND, false><<<cfg_grid, kThreads, 0, st>>>(w.h2, C2, P + po.W3, P + po.b3, f->shape.use_final_tanh,
                                                       l & 1, L, V, B, xin, xout, w.s, w.logdet, nullptr, l, N);
        GF_CHECK_LAUNCH();
        xin = xout;
    }
    k_finish<ND><<<cfg_grid, kThreads, 0, st>>>(w.z, xin, w.logdet, phi4 != nullptr, phi4 ? phi4->m2 : 0.0,
                                               phi4 ? phi4->lam : 0.0, L, V, B, phi_out, z_out, logq, S_out, logw);
    GF_CHECK_LAUNCH();
    return GF_OK;
}

}  // namespace
}  // namespace gf

using namespace gf;

extern "C" {

size_t gf_train_workspace_bytes(const gf_flow* flow, int64_t B) {
    if (!flow || B < 0 || flow->variant) return 0;
    return carve(flow, B, nullptr).bytes;
}

gf_status gf_flow_train_step(gf_flow* flow, const gf_phi4* phi4, int64_t B, uint64_t seed,
                             uint64_t counter0, const float* d_z_in, double* d_loss_out,
                             float* d_grad_out, float lr, float beta1, float beta2,
                             float adam_eps, float* d_adam_m, float* d_adam_v,
                             int64_t adam_t, void* d_workspace, size_t workspace_bytes,
                             cudaStream_t stream) {
    if (!flow || !phi4 || B <= 0 || !d_loss_out) return GF_EINVAL;
    if (flow->variant) return GF_EUNSUPPORTED;
    if (!(lr >= 0.f)) return GF_EINVAL;
    if (lr > 0.f && (!d_adam_m || !d_adam_v || adam_t < 1)) return GF_EINVAL;
    const TrainWs w = carve(flow, B, static_cast<char*>(d_workspace));
    if (!d_workspace || workspace_bytes < w.bytes) return GF_EINVAL;
    if ((reinterpret_cast<uintptr_t>(d_workspace) & 255) != 0) return GF_EINVAL;
    if (flow->shape.nd == 3)
        return train_step<3>(flow, phi4, B, seed, counter0, d_z_in, d_loss_out, d_grad_out, lr, beta1, beta2,
                             adam_eps, d_adam_m, d_adam_v, adam_t, w, stream);
    return train_step<2>(flow, phi4, B, seed, counter0, d_z_in, d_loss_out, d_grad_out, lr, beta1, beta2,
                         adam_eps, d_adam_m, d_adam_v, adam_t, w, stream);
}

gf_status gf_flow_forward_train(const gf_flow* flow, int64_t B, uint64_t seed, uint64_t counter0,
                                const float* d_z_in, float* d_phi_out, double* d_logq_out, void* d_workspace,
                                size_t workspace_bytes, cudaStream_t stream) {
    if (!flow || B <= 0 || !d_phi_out || !d_logq_out) return GF_EINVAL;
    if (flow->variant) return GF_EUNSUPPORTED;
    const TrainWs w = carve(flow, B, static_cast<char*>(d_workspace));
    if (!d_workspace || workspace_bytes < w.bytes) return GF_EINVAL;
    if ((reinterpret_cast<uintptr_t>(d_workspace) & 255) != 0) return GF_EINVAL;
    if (flow->shape.nd == 3)
        return forward_train<3>(flow, B, seed, counter0, d_z_in, d_phi_out, d_logq_out, w, stream);
    return forward_train<2>(flow, B, seed, counter0, d_z_in, d_phi_out, d_logq_out, w, stream);
}

gf_status gf_flow_backward(const gf_flow* flow, int64_t B, const float* d_gphi, const double* d_glogq,
                           float* d_grad_out, void* d_workspace, size_t workspace_bytes, cudaStream_t stream) {
    if (!flow || B <= 0 || !d_grad_out) return GF_EINVAL;
    if (flow->variant) return GF_EUNSUPPORTED;
    const TrainWs w = carve(flow, B, static_cast<char*>(d_workspace));
    if (!d_workspace || workspace_bytes < w.bytes) return GF_EINVAL;
    if ((reinterpret_cast<uintptr_t>(d_workspace) & 255) != 0) return GF_EINVAL;
    if (flow->shape.nd == 3) return backward<3>(flow, B, d_gphi, d_glogq, d_grad_out, w, stream);
    return backward<2>(flow, B, d_gphi, d_glogq, d_grad_out, w, stream);
}

gf_status gf_flow_adam_step(gf_flow* flow, const float* d_grad, float lr, float beta1, float beta2,
                            float adam_eps, float* d_adam_m, float* d_adam_v, int64_t adam_t,
                            cudaStream_t stream) {
    if (!flow || !d_grad || !d_adam_m || !d_adam_v || adam_t < 1 || !(lr >= 0.f)) return GF_EINVAL;
    if (flow->n_params == 0) return GF_OK;
    const float c1 = 1.f - powf(beta1, (float)adam_t), c2 = 1.f - powf(beta2, (float)adam_t);
    k_adam<<<(unsigned)grid1d(flow->n_params), kThreads, 0, stream>>>(flow->n_params, flow->d_canon, d_grad,
                                                                       d_adam_m, d_adam_v, lr, beta1, beta2,
                                                                       adam_eps, c1, c2);
    GF_CHECK_LAUNCH();
    if (flow->variant) return repack_variant(flow, stream);
    return repack_weights(flow, stream);
}

size_t gf_unfused_workspace_bytes(const gf_flow* flow, int64_t B) {
    if (!flow || B < 0 || flow->variant) return 0;
    return carve_plain(flow, B, nullptr).bytes;
}

gf_status gf_flow_sample_unfused(const gf_flow* flow, const gf_phi4* phi4, int64_t B, uint64_t seed,
                                 uint64_t counter0, const float* d_z_in, float* d_z_out, float* d_phi_out,
                                 double* d_logq_out, double* d_S_out, double* d_logw_out, void* d_workspace,
                                 size_t workspace_bytes, cudaStream_t stream) {
    if (!flow || B < 0 || (B > 0 && (!d_phi_out || !d_logq_out))) return GF_EINVAL;
    if (!phi4 && (d_S_out || d_logw_out)) return GF_EINVAL;
    if (flow->variant) return GF_EUNSUPPORTED;
    if (B == 0) return GF_OK;
    const PlainWs w = carve_plain(flow, B, static_cast<char*>(d_workspace));
    if (!d_workspace || workspace_bytes < w.bytes) return GF_EINVAL;
    if ((reinterpret_cast<uintptr_t>(d_workspace) & 255) != 0) return GF_EINVAL;
    if (flow->shape.nd == 3)
        return sample_unfused<3>(flow, phi4, B, seed, counter0, d_z_in, d_z_out, d_phi_out, d_logq_out, d_S_out,
                                 d_logw_out, w, stream);
    return sample_unfused<2>(flow, phi4, B, seed, counter0, d_z_in, d_z_out, d_phi_out, d_logq_out, d_S_out,
                             d_logw_out, w, stream);
}

}  // extern "C"
