// gf_hmc.cu -- FP64 HMC trajectories for lattice phi^4 (the comparison
// sampler of paper arXiv:2208.08903 Sec. 2.2, for the same action).
//
// One CTA per chain.  The field lives in shared memory for the whole
// trajectory (the force needs neighbours); each thread keeps the momenta of
// its own sites (n = tid + k*blockDim) in registers.  HBM is touched once at
// the start (phi) and once at the end (phi on accept, dH, accept flag).
//
// The FP64 pipe bounds it: a warp's FP64 instruction takes about 19 cycles of
// an SM (1.057 TFLOP/s on the chip), so what counts is FP64 instructions, of any
// kind.  A site's kick is 2 nd - 1 additions of its neighbours, phi^2, and three
// multiply-adds, its drift one: 10 in 3D.  The energies ride on the first and the
// last kick: the hopping part as the squares of the nd forward differences (each
// exact or nearly so, all of one sign), 2 nd + 3 instructions more.  From the
// neighbour sums, in 4, two sums far larger than their difference cancelled: dH
// of a smooth field of size 50 lost two digits.  Each FP64 Box-Muller block (about 150
// instructions) is evaluated once, by one lane of the four whose sites it
// serves, and exchanged by shuffles.  Measured, 20 steps, against the form with
// the Laplacian, force and energies written out (18 FP64 instructions a step)
// and four lanes evaluating every block: 512 chains of 3D L=16 2.39 -> 1.18 ms,
// 152 chains 0.60 -> 0.30 ms, 400 chains of 2D L=64 1.58 -> 0.73 ms.  What is
// left above the instruction count is the SMs that hold 4 of the 512 chains
// while others hold 3.
#include <algorithm>
#include <type_traits>

#include "gf_common.cuh"

namespace gf {
namespace {

constexpr int kHmcThreads = 256;
constexpr int kMaxSitesPerThread = 16;    // V <= 4096

// POW2: L = 2^lg, neighbour indices by bit operations instead of runtime
// divisions.
template <int ND, bool POW2>
__global__ void __launch_bounds__(kHmcThreads, 2) hmc_kernel(int L, int lg, int V, double m2, double lam,
                                                          int64_t n_chains, double* __restrict__ phi_g,
                                                          int n_steps, double eps, uint64_t seed,
                                                          uint64_t traj, double* __restrict__ dH_out,
                                                          uint8_t* __restrict__ acc_out) {
    const auto nbrs = [&](int n) { return POW2 ? site_nbrs_pow2(n, ND, lg) : site_nbrs(n, ND, L); };
    extern __shared__ __align__(16) unsigned char smem_raw[];
    double* p = reinterpret_cast<double*>(smem_raw);
    double* red = p + V;                        // 8 warps' sums of H before, 8 after, then the accept flag
    const int tid = threadIdx.x, lane = tid & 31;
    const int nper = (V + kHmcThreads - 1) / kHmcThreads;
    for (int64_t c = blockIdx.x; c < n_chains; c += gridDim.x) {
        double* g = phi_g + c * V;
        for (int n = tid; n < V; n += kHmcThreads) p[n] = g[n];
        // momenta: sites 4j..4j+3 from one Philox block (FP64 Box-Muller); lane r
        // of a quad evaluates the block of the quad's sites in row k0 + r
        double pi[kMaxSitesPerThread];
#pragma unroll
        for (int k0 = 0; k0 < kMaxSitesPerThread; k0 += 4) {
#pragma unroll
            for (int q = 0; q < 4; ++q) pi[k0 + q] = 0.0;
            if (k0 >= nper) continue;
            const int j = ((tid & ~3) + (k0 + (tid & 3)) * kHmcThreads) >> 2;
            double nn[4] = {0.0, 0.0, 0.0, 0.0};
            if (4 * j < V)
                normals4_f64(philox4x64_10(seed, 0ull, u64x4{(uint64_t)c, traj, (uint64_t)j, TAG_HMC_P}), nn);
#pragma unroll
            for (int q = 0; q < 4; ++q)
#pragma unroll
                for (int i = 0; i < 4; ++i) {
                    const double v = __shfl_sync(0xffffffffu, nn[i], (lane & ~3) + q);
                    if (i == (tid & 3)) pi[k0 + q] = v;
                }
#pragma unroll
            for (int q = 0; q < 4; ++q)
                if (tid + (k0 + q) * kHmcThreads >= V) pi[k0 + q] = 0.0;
        }
        __syncthreads();
        // pi -= h dS/dphi = h (2 (2 nd + m2) phi - 2 sum of neighbours + 4 lam phi^3);
        // E = -1: returns this thread's part of H before the kick, E = 1: after it.
        // H = sum 1/2 pi^2 + sum over mu (phi - phi(n+mu))^2 + m2 phi^2 + lam phi^4
        const auto kick = [&](double h, auto with_energy) -> double {
            constexpr int E = decltype(with_energy)::value;
            const Phi4Kick kk = phi4_kick(h, ND, m2, lam);
            double kin = 0.0, pot = 0.0;
#pragma unroll
            for (int k = 0; k < kMaxSitesPerThread; ++k) {
                const int n = tid + k * kHmcThreads;
                if (k < nper && n < V) {
                    const SiteNbrs b = nbrs(n);
                    const double f = p[n], f2 = f * f;
                    double s = (p[b.xp] + p[b.xm]) + (p[b.yp] + p[b.ym]);
                    if (ND == 3) s += p[b.zp] + p[b.zm];
                    if (E < 0) kin = fma(pi[k], pi[k], kin);
                    pi[k] = phi4_force_at(kk, f, f2, s, pi[k]);
                    if (E > 0) kin = fma(pi[k], pi[k], kin);
                    if (E != 0) {
                        const double dx = f - p[b.xp], dy = f - p[b.yp], dz = ND == 3 ? f - p[b.zp] : 0.0;
                        pot = fma(dy, dy, fma(dx, dx, pot));
                        if (ND == 3) pot = fma(dz, dz, pot);
                        pot = fma(f2, fma(lam, f2, m2), pot);
                    }
                }
            }
            return E != 0 ? fma(0.5, kin, pot) : 0.0;
        };
        const double h0 = kick(0.5 * eps, std::integral_constant<int, -1>());
        double h1 = 0.0;
        for (int i = 1; i <= n_steps; ++i) {
            __syncthreads();     // all kicks read p before it moves
#pragma unroll
            for (int k = 0; k < kMaxSitesPerThread; ++k) {
                const int n = tid + k * kHmcThreads;
                if (k < nper && n < V) p[n] = fma(eps, pi[k], p[n]);
            }
            __syncthreads();
            if (i < n_steps) kick(eps, std::integral_constant<int, 0>());
            else h1 = kick(0.5 * eps, std::integral_constant<int, 1>());
        }
        // the two energies are added up separately: their difference is small
        const double w0 = warp_sum(h0), w1 = warp_sum(h1);
        if (lane == 0) {
            red[tid >> 5] = w0;
            red[8 + (tid >> 5)] = w1;
        }
        __syncthreads();
        if (tid < 32) {
            double H0 = 0.0, H1 = 0.0;
            for (int i = 0; i < kHmcThreads / 32; ++i) {
                H0 += red[i];
                H1 += red[8 + i];
            }
            if (tid == 0) {
                const u64x4 w = philox4x64_10(seed, 0ull, u64x4{(uint64_t)c, traj, 0ull, TAG_HMC_U});
                const double dH = H1 - H0;
                const bool acc = (-dH) > log(u53(w.x));
                red[16] = acc ? 1.0 : 0.0;
                if (dH_out) dH_out[c] = dH;
                if (acc_out) acc_out[c] = acc ? 1 : 0;
            }
        }
        __syncthreads();
        if (red[16] != 0.0)
            for (int n = tid; n < V; n += kHmcThreads) g[n] = p[n];
        __syncthreads();
    }
}

}  // namespace
}  // namespace gf

using namespace gf;

extern "C" gf_status gf_hmc_trajectory(int32_t nd, int32_t L, const gf_phi4* phi4, int64_t n_chains,
                                       double* d_phi, int32_t n_steps, double eps, uint64_t seed,
                                       uint64_t traj_index, double* d_dH_out, uint8_t* d_acc_out,
                                       cudaStream_t stream) {
    if (!phi4 || (nd != 2 && nd != 3) || L < 1 || n_chains < 0 || n_steps < 1 || !(eps == eps))
        return GF_EINVAL;
    int64_t V = 1;
    for (int i = 0; i < nd; ++i) V *= L;
    if (V > (int64_t)kHmcThreads * kMaxSitesPerThread) return GF_EUNSUPPORTED;
    if (n_chains == 0) return GF_OK;
    if (!d_phi) return GF_EINVAL;
    const size_t smem = (size_t)V * 8 + 32 * 8;
    int lg = 0;
    while ((1 << lg) < L) ++lg;
    const bool pow2 = (1 << lg) == L;
    auto kern = nd == 3 ? (pow2 ? hmc_kernel<3, true> : hmc_kernel<3, false>)
                        : (pow2 ? hmc_kernel<2, true> : hmc_kernel<2, false>);
    if (cudaFuncSetAttribute(kern, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem) != cudaSuccess)
        return GF_ECUDA;
    int per_sm = 0;
    if (cudaOccupancyMaxActiveBlocksPerMultiprocessor(&per_sm, kern, kHmcThreads, smem) != cudaSuccess ||
        per_sm < 1)
        per_sm = 1;
    const int64_t grid = std::min<int64_t>(n_chains, (int64_t)num_sms() * per_sm);
    kern<<<(unsigned)grid, kHmcThreads, smem, stream>>>(L, lg, (int)V, phi4->m2, phi4->lam, n_chains, d_phi,
                                                        n_steps, eps, seed, traj_index, d_dH_out, d_acc_out);
    GF_CHECK_LAUNCH();
    return GF_OK;
}
