// gf_flow_fp32.cu -- host side of the fused FP32 coupling-stack kernel: the
// shared-memory plan of a shape, the split of the head's sums, and the CTA
// size and conv2 tiles of a launch.
#include <algorithm>
#include <cstring>

#include "gf_flow_fp32_kernel.cuh"

namespace gf {

using namespace f32k;

namespace {

constexpr size_t kBudget = 227 * 1024;

// Which lanes sum the head (conv3) is part of the results: with `tps` lanes to
// a site, each sums C / tps channels over all taps and the lanes' sums are
// added pairwise.  tps is the largest power of two that divides C / 4 and
// gives the updated sites of a block of slices at most 256 lanes; the blocks
// are runs of as many slices (G) as two hidden tensors of G + 2 slices (all
// slices: L) leave within 227 KB.  It depends on the shape only, so results
// are the same whatever slices, tiles and threads a launch works with.
// Shapes for which not even a block of one slice fits are not supported.
struct HeadSplit {
    int G, zb, a, b;   // lanes per site: a in slices < zb, b from there on
};
bool head_split(int L, int S, int V, int C, HeadSplit* out) {
    const auto fits = [&](int slots) {
        return (size_t)((V + 3) & ~3) * 4 + (size_t)slots * S * 2 * C * 4 + 400 <= kBudget;
    };
    int G = L;
    if (L > MAX_PHASE_SLICES || !fits(L)) {
        G = std::min(MAX_PHASE_SLICES, L - 3);
        while (G >= 1 && !fits(G + 2)) --G;
        if (G < 1) return false;
    }
    const auto lanes = [&](int n) {
        int tps = 1;
        while (tps * 2 <= C / 4 && (C / 4) % (tps * 2) == 0 && n * (S / 2) * tps * 2 <= 256) tps *= 2;
        return tps;
    };
    const int rem = L % G;
    *out = HeadSplit{G, L - rem, lanes(G), rem ? lanes(rem) : 1};
    return true;
}

int64_t small_floats(int T, int C) { return 3LL * T * C + 2 * C + 4; }

// Shared memory (bytes) of a plan, filling the offsets when a != null.
size_t plan_smem(const gf_flow* f, int R, int n_phases, bool gw, int stage_taps, bool two_small, FlowArgs* a) {
    const int64_t C = f->C1, slot = (int64_t)f->S * C;
    int64_t o = (f->V + 3) & ~3;
    const int64_t h1 = o; o += R * slot;
    const int64_t h2 = o; o += R * slot;
    const int64_t sml = o; if (!gw) o += small_floats(f->T, f->C1) * (two_small ? 2 : 1);
    const int64_t w2 = o; if (!gw) o += 2LL * stage_taps * C * C;
    const int64_t red = o; o += 64;
    const int64_t ss = o; if (!gw) o += (f->V / 2 + 3) & ~3;
    const int64_t sch = o; if (!gw) o += (int64_t)n_phases * (int64_t)(sizeof(Phase) / 4);
    if (a) {
        a->off_h1 = (int)h1; a->off_h2 = (int)h2; a->off_small = (int)sml; a->off_w2 = (int)w2;
        a->off_red = (int)red; a->off_s = (int)ss; a->off_sched = (int)sch;
    }
    return (size_t)o * 4;
}

// Cost model of a conv2 phase of n slices, in cycles per input channel: with
// `resident` CTAs on an SM the FMA pipe (128 per cycle) or the shared-memory
// reads (one 128-byte wavefront per cycle: NS for the sites, CO / 4 for the
// weights) bound it, plus the issue slots that pairing a site's value with itself
// takes; one CTA alone needs its warps' issue time on the busiest of the four
// schedulers and, per pass, the latencies that nothing hides: about 20 cycles
// and 0.4 of a warp's time, and no less than the arrival of a stage of weights
// (800 cycles) over its `stage` channels.
struct TileCost { double eff, lat; int passes; };
TileCost tile_cost(int nf, int C, int tile, int warps, int stage) {
    const int ns = kTileNS[tile], co = kTileCO[tile];
    const int tasks = (nf + 32 * ns - 1) / (32 * ns) * (C / co);
    TileCost t;
    t.passes = (tasks + warps - 1) / warps;
    t.eff = tasks * (std::max(ns * co / 4.0, ns + std::max(1.0, co / 4.0)) + 0.5 + 0.4 * ns);
    const double c = ns * co + 1.6 * ns + 2.0;
    t.lat = 0;
    for (int left = tasks; left > 0; left -= warps)
        t.lat += std::max(((std::min(left, warps) + 3) / 4 + 0.4) * c + 20.0, 800.0 / stage);
    return t;
}
// The conv2 phases of one layer with one tile.
TileCost layer_cost(const gf_flow* f, int tile, int warps, int taps) {
    TileCost sum{0, 0, 0};
    for (int i = 0; i < f->n_h2; ++i) {
        const TileCost t = tile_cost(f->h2_n[i] * f->S, f->C1, tile, warps, taps * f->C1);
        sum.eff += f->h2_count[i] * t.eff;
        sum.lat += f->h2_count[i] * t.lat;
        sum.passes += f->h2_count[i] * t.passes;
    }
    return sum;
}
// Sets the flow's list of conv2 phases (false: more kinds than it holds).
bool set_h2(gf_flow* f, const std::vector<Phase>& s) {
    f->n_h2 = 0;
    for (const Phase& p : s) {
        if (p.type != PH_H2) continue;
        int i = 0;
        while (i < f->n_h2 && f->h2_n[i] != p.n) ++i;
        if (i == kMaxPhaseKinds) return false;
        if (i == f->n_h2) { f->h2_n[i] = p.n; f->h2_count[i] = 0; ++f->n_h2; }
        ++f->h2_count[i];
    }
    return true;
}

FlowKernel kernel_for(const gf_flow* f, int tile, int mode) {
    const bool gw = f->weights_global;
    switch (f->shape.nd * 100 + f->C1) {
        case 208: return kernel_of<2, 8>(tile, gw, mode);
        case 216: return kernel_of<2, 16>(tile, gw, mode);
        case 224: return kernel_of<2, 24>(tile, gw, mode);
        case 232: return kernel_of<2, 32>(tile, gw, mode);
        case 308: return kernel_of<3, 8>(tile, gw, mode);
        case 316: return kernel_of<3, 16>(tile, gw, mode);
        case 324: return kernel_of<3, 24>(tile, gw, mode);
        default: return kernel_of<3, 32>(tile, gw, mode);
    }
}

// CTAs of nt threads per SM: 228 KB of shared memory (1 KB per CTA reserved)
// and 64 K registers, 128 to a thread (the kernels' launch bound).
int ctas_per_sm(size_t smem, int nt) {
    return std::min((int)(228 * 1024 / (smem + 1024)), 65536 / (128 * nt));
}

}  // namespace

gf_status flow_fp32_configure(gf_flow* f) {
    const int L = f->shape.L, C = f->C1;
    HeadSplit hs;
    if (!head_split(L, f->S, f->V, C, &hs)) return GF_EUNSUPPORTED;
    f->head_G = hs.G; f->head_zb = hs.zb; f->head_a = hs.a; f->head_b = hs.b;
    // staged taps of W2 per buffer: all of them up to 12 KB, else about 8 KB
    const int tap = C * C * 4;
    f->stage_taps = f->T * tap <= 12 * 1024 ? f->T : std::max(1, 8192 / tap);
    f->weights_global = false;
    if (fp32_c32_recompute_supported(f)) {               // (kernels of its own for everything: no plan needed)
        f->full = true; f->G = L; f->R = L; f->n_phases = 3;
        return GF_OK;
    }
    // the whole lattice when it fits with a second buffer for the small weights
    if (L <= MAX_PHASE_SLICES && plan_smem(f, L, 3, false, f->stage_taps, true, nullptr) <= kBudget) {
        f->full = true; f->two_small = true; f->G = L; f->R = L; f->n_phases = 3;
        f->smem_bytes = plan_smem(f, f->R, f->n_phases, false, f->stage_taps, true, nullptr);
        f->n_h2 = 1; f->h2_n[0] = (int16_t)L; f->h2_count[0] = 1;
        return GF_OK;
    }
    // else G slices at a time: the cheapest G that fits, staging one tap per
    // buffer when the activations are large
    f->full = false; f->two_small = false;
    double best = 0;
    int bestG = 0, best_taps = 0, best_phases = 0;
    for (int taps : {f->stage_taps, 1}) {
        int top = std::min(MAX_PHASE_SLICES, L - 3);
        while (top >= 1 && plan_smem(f, top + 2, 0, false, taps, false, nullptr) > kBudget) --top;
        for (int G = top; G >= std::max(1, top - 7); --G) {
            // the schedule's conv2 phases: the first block needs two slices more
            // than it has, a short last one finds two in the cache
            f->n_h2 = 0;
            const auto add = [&](int n) {
                int i = 0;
                while (i < f->n_h2 && f->h2_n[i] != n) ++i;
                if (i == f->n_h2) { f->h2_n[i] = (int16_t)n; f->h2_count[i] = 0; ++f->n_h2; }
                ++f->h2_count[i];
            };
            for (int extra = 2; extra > 0; extra -= G) add(std::min(G, extra));
            for (int a = 0; a < L; a += G)
                if (L - a >= G) add(G);
                else if (L - a > 2) add(L - a - 2);
            double c = 0;
            for (int t = tile_first(C); t < kTiles; ++t) {
                const TileCost tc = layer_cost(f, t, 16, taps);
                const double ct = std::max(tc.eff, tc.lat) + 12.0 * ((L + G - 1) / G + 1);   // phase overhead: barriers, tails
                if (c == 0 || ct < c) c = ct;
            }
            if (bestG && c >= 0.98 * best) continue;
            const int phases = (int)build_schedule(L, G, false).size();
            if (plan_smem(f, G + 2, phases, false, taps, false, nullptr) > kBudget) continue;
            best = c; bestG = G; best_taps = taps; best_phases = phases;
        }
        if (taps == 1) break;
    }
    if (!bestG) {                                        // weights read from global memory
        f->weights_global = true;
        bestG = hs.G;                                    // (the sums' order is that of these blocks and 256 threads)
        best_phases = (int)build_schedule(L, bestG, false).size();
        if (plan_smem(f, bestG + 2, best_phases, true, f->T, false, nullptr) > kBudget) return GF_EUNSUPPORTED;
        best_taps = f->T;
    }
    f->G = bestG; f->R = bestG + 2; f->stage_taps = best_taps; f->n_phases = best_phases;
    f->smem_bytes = plan_smem(f, f->R, f->n_phases, f->weights_global, best_taps, false, nullptr);
    return set_h2(f, build_schedule(L, f->G, false)) ? GF_OK : GF_EUNSUPPORTED;
}

namespace {

// Fills in the plan of a launch over a.B configurations, chooses its CTA size
// and tile and launches it.
gf_status launch_plan(const gf_flow* f, FlowArgs& a, bool inverse, cudaStream_t stream) {
    const int64_t B = a.B;
    if (B <= 0) return GF_OK;
    const int L = f->shape.L, C = f->C1;
    const bool gw = f->weights_global, rec = a.s_out != nullptr;
    const int mode = rec ? kRecompute : a.xs_out ? kForward : kFlow;
    if (gw && mode != kFlow) return GF_EUNSUPPORTED;
    a.W = f->d_packed;
    a.sched = f->d_sched;
    a.n_phases = f->n_phases;
    a.stride = f->packed_stride;
    a.off = packed_offsets(f->T, C, C);
    a.L = L; a.S = f->S; a.V = f->V;
    a.R = f->R;
    a.stage_taps = f->stage_taps;
    a.n_stages = (f->T + f->stage_taps - 1) / f->stage_taps;
    a.two_small = f->two_small;
    a.head_G = f->head_G;
    a.head_zb = a.head_train ? L : f->head_zb;
    a.head_a = a.head_train ? 1 : f->head_a;
    a.head_b = f->head_b;
    a.fd_S = make_fastdiv((uint32_t)f->S);
    a.fd_L = make_fastdiv((uint32_t)L);
    a.fd_Sh = make_fastdiv((uint32_t)(f->S / 2));
    a.fd_Lh = make_fastdiv((uint32_t)(L / 2));
    a.slope = (float)f->shape.leaky_slope;
    a.use_tanh = f->shape.use_final_tanh;
    const size_t smem = plan_smem(f, f->R, f->n_phases, gw, f->stage_taps, f->two_small, &a);

    // CTA size and tile: those that finish the batch soonest (estimated: conv2
    // at its bound plus a fixed time per layer for the phases' latencies; against
    // every tile and CTA size on 50 lattices and widths at 64 to 4000 configurations
    // the pick takes 1.00 of the best one's time at the median, 1.13 at the 90th
    // percentile and 1.31 at worst, large batches of small lattices, which run best
    // with 4 x 8 tiles and fewer threads: 3D L = 8, hidden 8, 4000 1575 against
    // 1202 us);
    // 512 threads where the slices leave room for one CTA (256 with weights in
    // global memory, where the order of the sums is the CTA's own).
    int nti = -1, tile = 0;
    const int64_t sms = num_sms();
    double best = 0;
    for (int t = gw ? kTileGW : rec ? kTileRec : tile_first(C); t < kTiles; ++t)
        for (int i = gw ? kCtaSizes - 2 : f->full ? 0 : kCtaSizes - 1; i < (gw ? kCtaSizes - 1 : kCtaSizes); ++i) {
            const int nt = 64 << i, r = (int)std::min<int64_t>((B + sms - 1) / sms, ctas_per_sm(smem, nt));
            const TileCost c = layer_cost(f, t, nt / 32, f->stage_taps);
            const double items = (double)f->V * (C / 8 * 2 + 2) / nt;            // conv1 and head items per thread
            const double lat = c.lat * f->T * C + 2500.0 + 1.2 * nt + 60.0 * f->T / 9 * items, eff = 1.2 * c.eff * f->T * C;
            const double cost = (double)((B + sms * r - 1) / (sms * r)) * std::max(lat, r * eff);
            if (nti < 0 || cost < best) { best = cost; nti = i; tile = t; }
        }
    if (nti < 0) return GF_ECUDA;
    // (on every launch: a limit remembered from an earlier context does not hold
    // after a device reset)
    const FlowKernel kern = kernel_for(f, tile, mode);
    if (cudaFuncSetAttribute(kern, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)kBudget) != cudaSuccess)
        return GF_ECUDA;
    const int NT = 64 << nti;
    a.n_passes = layer_cost(f, tile, NT / 32, f->stage_taps).passes;
    const int64_t grid = std::min<int64_t>(B, sms * ctas_per_sm(smem, NT));
    kern<<<(unsigned)grid, NT, smem, stream>>>(a, inverse ? 1 : 0);
    GF_CHECK_LAUNCH();
    return GF_OK;
}

}  // namespace

gf_status launch_flow_fp32(const gf_flow* f, bool inverse, const gf_phi4* phi4, int64_t B,
                           uint64_t seed, uint64_t counter0, const float* z_in, float* z_out,
                           const float* phi_in, float* phi_out, double* logq_out,
                           double* S_out, double* logw_out, cudaStream_t stream, float* xs_out, int64_t xs_stride,
                           double* logdet_out) {
    if (fp32_c32_supported(f))
        return launch_flow_fp32_c32(f, inverse, phi4, B, seed, counter0, z_in, z_out, phi_in, phi_out, logq_out,
                                    S_out, logw_out, stream, xs_out, xs_stride, logdet_out);
    FlowArgs a;
    std::memset(&a, 0, sizeof(a));
    a.n_layers = f->shape.n_layers;
    a.head_train = xs_out != nullptr;
    a.has_phi4 = phi4 != nullptr;
    ff_split(2.0 * f->shape.nd + (phi4 ? phi4->m2 : 0.0), &a.c2d_ff.hi, &a.c2d_ff.lo);
    ff_split(phi4 ? phi4->lam : 0.0, &a.lam_ff.hi, &a.lam_ff.lo);
    a.B = B; a.seed = seed; a.counter0 = counter0;
    a.z_in = z_in; a.z_out = z_out; a.phi_in = phi_in; a.phi_out = phi_out;
    a.logq_out = logq_out; a.S_out = S_out; a.logw_out = logw_out;
    a.xs_out = xs_out; a.xs_stride = xs_stride; a.logdet_out = logdet_out;
    return launch_plan(f, a, inverse, stream);
}

gf_status launch_recompute(const gf_flow* f, int layer, int64_t B, const float* xl, float* h1_out, float* h2_out,
                           float* s_out, cudaStream_t stream) {
    if (fp32_c32_recompute_supported(f)) return launch_c32_recompute(f, layer, B, xl, h1_out, h2_out, s_out, stream);
    FlowArgs a;
    std::memset(&a, 0, sizeof(a));
    a.layer0 = layer;
    a.n_layers = 1;
    a.head_train = 1;
    a.B = B;
    a.z_in = xl;
    a.h1_out = h1_out; a.h2_out = h2_out; a.s_out = s_out;
    return launch_plan(f, a, false, stream);
}

}  // namespace gf
