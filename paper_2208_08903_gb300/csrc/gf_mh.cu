// gf_mh.cu -- Metropolis-Hastings independence chain over flow proposals
// (paper arXiv:2208.08903 Sec. 1: proposals from the flow corrected by the
// MH test with the Jacobian; acceptance min(1, w'/w), w = p/q).
//
// Proposal k is accepted iff a_k > log w_cur, a_k = log w_k - log u_g
// (w_k / w_cur > u_g, the proposal-only term formed first), u_g from Philox word
// 0 of ctr = (g, 0, 0, TAG_MH), key = (seed, stream_id).  Doubles are compared
// as order-preserving int64 keys.  Two kernels on the caller's stream (one for
// up to kFuseN proposals):
//  1. mh_prep_kernel: the keys of a_k, in parallel, into the workspace;
//  2. mh_scan_kernel: the chain, in one CTA.  After an accepted proposal j the
//     next accept is the first later k with a_k > log w_j, whatever came
//     before j: within a chunk of 32 proposals the accepts that follow from an
//     accept at j are known without the chain, as a 32-bit mask (each lane
//     compares its log w with the 32 a_k, then five rounds of pointer
//     doubling).  What is left to do in order is one step per chunk: the first
//     a_k above the current state (one ballot) names the chunk's mask and its
//     last state.  Warp 0 does that for batch i of 31 chunks while the other
//     warps write out batch i - 1 and prepare batch i + 1.
// The scan is bound by the ordered steps' latency, about 200 cycles each.
// Measured on 16,384 proposals with about half of them accepted, against one
// warp with a ballot per accept: 547 -> 55 us.
#include <algorithm>
#include <mutex>

#include "gf_common.cuh"

namespace gf {

// Order-preserving map of doubles to int64 (x < y <=> key(x) < key(y) for
// non-NaN x, y; -0 and +0 map to the same key).  `nan_key` is returned for NaN.
__device__ __forceinline__ int64_t order_key(double x, int64_t nan_key) {
    if (x != x) return nan_key;
    int64_t b = __double_as_longlong(x);
    if (b == INT64_MIN) b = 0;                              // -0 -> +0
    return b >= 0 ? b : (b ^ INT64_MAX);
}

__global__ void mh_prep_kernel(const gf_mh_state* __restrict__ st, int64_t n, const double* __restrict__ logw,
                               int64_t* __restrict__ key_a) {
    const int64_t step0 = st->step;
    const uint64_t seed = st->seed, stream_id = st->stream_id;
    for (int64_t k = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; k < n;
         k += (int64_t)gridDim.x * blockDim.x) {
        const u64x4 w = philox4x64_10(seed, stream_id, u64x4{(uint64_t)(step0 + k), 0ull, 0ull, TAG_MH});
        key_a[k] = order_key(logw[k] - log(u53(w.x)), INT64_MIN);      // NaN never accepts
    }
}

constexpr int kBatch = 31;                       // chunks of 32 proposals a batch: one per preparing warp
// Up to here the scan computes the keys itself: a launch less (about 4 us) for
// about 35 FP64 instructions per chunk on one SM (0.3 us); beyond it the
// logarithms take longer than the launch.
constexpr int64_t kFuseN = 128;

struct MhBatch {
    int64_t key[32 * kBatch];                    // a_k
    int64_t last[32 * kBatch];                   // key of the state the accept of k leads to at the chunk's end
    uint32_t mask[32 * kBatch];                  // accepts of the chunk that follow from the accept of k (k included)
    uint32_t accm[32];                           // the chain's accepts in the chunk
    int64_t idx[32];                             // the state before the chunk
};

// FUSE: key_a is not read; the keys are formed here.
template <bool FUSE>
__global__ void __launch_bounds__(1024) mh_scan_kernel(gf_mh_state* __restrict__ st, int64_t n,
                                                       const double* __restrict__ logw,
                                                       const int64_t* __restrict__ key_a,
                                                       int64_t* __restrict__ chain_idx,
                                                       uint8_t* __restrict__ acc_out) {
    extern __shared__ __align__(16) unsigned char mh_smem[];
    MhBatch* ring = reinterpret_cast<MhBatch*>(mh_smem);     // 3: being prepared, scanned, written out
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    const int64_t chunks = (n + 31) / 32, batches = (chunks + kBatch - 1) / kBatch;
    const int64_t g0 = st->step;
    int64_t cur_key = order_key(st->logw_cur, INT64_MAX);    // a NaN state accepts nothing more
    int64_t idx = st->idx_cur, nacc = 0;

    // a chunk's inputs, loaded a batch before they are used
    double lw = 0.0;
    int64_t ka_in = INT64_MIN;
    const auto load = [&](int64_t batch, int c) {
        const int64_t k = (batch * kBatch + c) * 32 + lane;
        if (k >= n) return;
        lw = __ldg(logw + k);
        if (!FUSE) ka_in = __ldg(key_a + k);
    };
    const auto prepare = [&](int64_t batch, int c) {
        MhBatch& r = ring[batch % 3];
        const int64_t k = (batch * kBatch + c) * 32 + lane;
        int64_t ka = INT64_MIN, wk = INT64_MAX;
        if (k < n) {
            wk = order_key(lw, INT64_MAX);
            if (FUSE) {
                const u64x4 w = philox4x64_10(st->seed, st->stream_id, u64x4{(uint64_t)(g0 + k), 0ull, 0ull, TAG_MH});
                ka = order_key(lw - log(u53(w.x)), INT64_MIN);
            } else {
                ka = ka_in;
            }
        }
        r.key[32 * c + lane] = ka;
        __syncwarp();
        uint32_t above = 0u;                     // proposals whose a exceeds this lane's log w
#pragma unroll
        for (int s = 0; s < 32; s += 2) {        // (broadcast reads: two keys each)
            const longlong2 a = *reinterpret_cast<const longlong2*>(r.key + 32 * c + s);
            above |= (uint32_t)(a.x > wk) << s | (uint32_t)(a.y > wk) << (s + 1);
        }
        above &= lane == 31 ? 0u : ~((2u << lane) - 1u);
        uint32_t m = 1u << lane;
        int nxt = above ? __ffs(above) - 1 : lane;           // the next accept after one at `lane` (itself: none)
#pragma unroll
        for (int i = 0; i < 5; ++i) {
            m |= __shfl_sync(0xffffffffu, m, nxt);
            nxt = __shfl_sync(0xffffffffu, nxt, nxt);
        }
        r.mask[32 * c + lane] = m;
        r.last[32 * c + lane] = __shfl_sync(0xffffffffu, wk, nxt);
    };
    const auto write_out = [&](int64_t batch, int c) {
        const MhBatch& r = ring[batch % 3];
        const int64_t base = (batch * kBatch + c) * 32, k = base + lane;
        const uint32_t accm = r.accm[c];
        // state after this lane's step: the last accept at or before it
        const uint32_t le = lane == 31 ? accm : (accm & ((2u << lane) - 1u));
        if (k < n) {
            if (chain_idx) chain_idx[k] = le ? g0 + base + (31 - __clz(le)) : r.idx[c];
            if (acc_out) acc_out[k] = (uint8_t)((accm >> lane) & 1u);
        }
    };
    const auto chunks_of = [&](int64_t batch) {
        return batch < 0 || batch >= batches ? 0 : (int)min((int64_t)kBatch, chunks - batch * kBatch);
    };

    const int c0 = warp - 1;                     // this warp's chunk of every batch (warp 0: none)
    if (warp > 0 && c0 < chunks_of(0)) {
        load(0, c0);
        prepare(0, c0);
        load(1, c0);
    }
    __syncthreads();
    for (int64_t i = 0; i <= batches; ++i) {
        if (warp == 0) {
            if (i < batches) {
                MhBatch& r = ring[i % 3];
                const int nc = chunks_of(i);
                uint32_t mine = 0u;                                          // the accepts of chunk `lane`
                int64_t ka = r.key[lane], last = r.last[lane];
                uint32_t mask = r.mask[lane];
                const auto one = [&](int c, bool first) {
                    const int nx = 32 * min(c + 1, kBatch - 1) + lane;       // the next chunk, loaded ahead
                    const int64_t ka_n = r.key[nx], last_n = r.last[nx];
                    const uint32_t mask_n = r.mask[nx];
                    uint32_t m = __ballot_sync(0xffffffffu, ka > cur_key);
                    if (first) m |= 1u;
                    const int j = __ffs(m) - 1;                              // (-1: every lane's shuffle reads lane 31)
                    const int64_t nk = __shfl_sync(0xffffffffu, last, j);
                    const uint32_t acc = __shfl_sync(0xffffffffu, mask, j);
                    cur_key = m ? nk : cur_key;
                    if (lane == c) mine = m ? acc : 0u;
                    ka = ka_n;
                    last = last_n;
                    mask = mask_n;
                };
                one(0, g0 == 0 && i == 0);                                   // (the first proposal of a chain is accepted)
#pragma unroll 4
                for (int c = 1; c < nc; ++c) one(c, false);
                // the state before chunk `lane`: the last accept of the chunks before it
                const uint32_t some = __ballot_sync(0xffffffffu, mine != 0u), prev = some & ((1u << lane) - 1u);
                const int64_t my_last = g0 + (i * kBatch + lane) * 32 + (31 - __clz(mine));
                const int64_t from = __shfl_sync(0xffffffffu, my_last, prev ? 31 - __clz(prev) : 0);
                r.accm[lane] = mine;
                r.idx[lane] = prev ? from : idx;
                if (some) idx = __shfl_sync(0xffffffffu, my_last, 31 - __clz(some));
                nacc += __reduce_add_sync(0xffffffffu, __popc(mine));
            }
        }
        if (warp > 0) {
            if (c0 < chunks_of(i + 1)) {
                prepare(i + 1, c0);
                load(i + 2, c0);
            }
            if (c0 < chunks_of(i - 1)) write_out(i - 1, c0);
        }
        __syncthreads();
    }
    if (threadIdx.x == 0) {
        // the state's log weight: that of its proposal, when one was accepted
        if (nacc > 0) st->logw_cur = logw[idx - g0];
        st->idx_cur = idx;
        st->n_acc += nacc - (g0 == 0 && n > 0 ? 1 : 0);      // step 0 is not counted
        st->step = g0 + n;
    }
}

gf_status mh_launch(gf_mh_state* d_state, int64_t n, const double* d_logw, int64_t* d_idx,
                    uint8_t* d_acc, int64_t* d_keys, cudaStream_t stream) {
    const size_t smem = 3 * sizeof(MhBatch);
    // one warp scans, the others prepare and write: as many as a batch has chunks
    const int warps = (int)std::min<int64_t>(32, (n + 31) / 32 + 1);
    const auto kern = n <= kFuseN ? mh_scan_kernel<true> : mh_scan_kernel<false>;
    if (cudaFuncSetAttribute(kern, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem) != cudaSuccess)
        return GF_ECUDA;
    if (n > kFuseN) {
        const int64_t blocks = std::min<int64_t>((n + 255) / 256, (int64_t)num_sms() * 8);
        mh_prep_kernel<<<(unsigned)blocks, 256, 0, stream>>>(d_state, n, d_logw, d_keys);
        GF_CHECK_LAUNCH();
    }
    kern<<<1, 32 * warps, smem, stream>>>(d_state, n, d_logw, d_keys, d_idx, d_acc);
    GF_CHECK_LAUNCH();
    return GF_OK;
}

// ---------------------------------------------------------------------------
// Allocation-free variant: log u goes to a fixed device array owned by the
// library instead of caller workspace.  Host code cannot use the array's
// name as a device address, so its address is looked up on every call made
// outside stream capture (a device reset or a new primary context can move
// it) and cached per device; a call being captured into a graph uses the
// cached address (looked up first if there is none).
// ---------------------------------------------------------------------------
static __device__ __align__(256) int64_t g_mh_noalloc_keys[GF_MH_NOALLOC_MAX_N];

namespace {
constexpr int kMaxDevices = 64;
std::mutex g_noalloc_mu;
int64_t* g_noalloc_ptr[kMaxDevices] = {};

gf_status noalloc_scratch(cudaStream_t stream, int64_t** out) {
    int dev = 0;
    if (cudaGetDevice(&dev) != cudaSuccess) return GF_ECUDA;
    if (dev < 0 || dev >= kMaxDevices) return GF_EUNSUPPORTED;
    cudaStreamCaptureStatus cs = cudaStreamCaptureStatusNone;
    if (cudaStreamIsCapturing(stream, &cs) != cudaSuccess) return GF_ECUDA;
    std::lock_guard<std::mutex> lock(g_noalloc_mu);
    if (g_noalloc_ptr[dev] == nullptr || cs == cudaStreamCaptureStatusNone) {
        void* p = nullptr;
        if (cudaGetSymbolAddress(&p, g_mh_noalloc_keys) != cudaSuccess || p == nullptr) return GF_ECUDA;
        g_noalloc_ptr[dev] = static_cast<int64_t*>(p);
    }
    *out = g_noalloc_ptr[dev];
    return GF_OK;
}
}  // namespace

}  // namespace gf

using namespace gf;

extern "C" {

size_t gf_mh_chain_workspace_bytes(int64_t n) { return n > 0 ? (size_t)n * sizeof(int64_t) : 0; }

gf_status gf_mh_chain(gf_mh_state* d_state, int64_t n, const double* d_logw,
                      int64_t* d_chain_idx_out, uint8_t* d_acc_out,
                      void* d_workspace, size_t workspace_bytes, cudaStream_t stream) {
    if (!d_state || n < 0) return GF_EINVAL;
    if ((reinterpret_cast<uintptr_t>(d_state) & 7) != 0) return GF_EINVAL;
    if (n == 0) return GF_OK;
    if (!d_logw || !d_workspace || workspace_bytes < gf_mh_chain_workspace_bytes(n)) return GF_EINVAL;
    if ((reinterpret_cast<uintptr_t>(d_workspace) & 7) != 0) return GF_EINVAL;
    return mh_launch(d_state, n, d_logw, d_chain_idx_out, d_acc_out,
                     static_cast<int64_t*>(d_workspace), stream);
}

gf_status gf_mh_chain_noalloc(gf_mh_state* d_state, int64_t n, const double* d_logw,
                              int64_t* d_chain_idx_out, uint8_t* d_acc_out, cudaStream_t stream) {
    if (!d_state || n < 0) return GF_EINVAL;
    if ((reinterpret_cast<uintptr_t>(d_state) & 7) != 0) return GF_EINVAL;
    if (n > GF_MH_NOALLOC_MAX_N) return GF_EINVAL;
    if (n == 0) return GF_OK;
    if (!d_logw) return GF_EINVAL;
    int64_t* scratch = nullptr;
    const gf_status st = noalloc_scratch(stream, &scratch);
    if (st != GF_OK) return st;
    return mh_launch(d_state, n, d_logw, d_chain_idx_out, d_acc_out, scratch, stream);
}

}  // extern "C"
