// Route planner: Eq. 1 of the paper evaluated on the device.
//
// For every query block j of every sequence the planner writes the ascending list
// P(j) = {j, j-1, ..., j-W, 0} u {j - 2^k}, its length, and the selected token pairs of the
// block (Proposition 1's accounting).  The problem is a few hundred to a few thousand query blocks and launch
// latency, not throughput, is what a caller sees (Section 5.1: at short context the route's bookkeeping and the launch
// cost more than the attention arithmetic).  So nothing is passed between CTAs: each of them scans the sequence lengths
// itself; the first one then does everything that is one number per query block (and the hand-out order), the others
// write the lists, a thread per entry (an entry follows from its place: list_tile in bf1_common.cuh), kListSlots query
// blocks to a CTA.  What is left is a chain of launch, one read of cu_seqlens, a few block-wide synchronisations and the
// stores.
// Measured: 10.4 -> 5.7 us for four sequences of 40K tokens, 5.0 -> 3.7 for one of 1K (one CTA that merged the candidate
// streams of a list in one thread before; one CTA with a thread per entry: 13.9, its issue slots are the bound).
//
// The attention kernels work on tiles of 64 tokens.  With the route block width b = 128 every slot of
// the route is still one 64-token tile: tile t of a sequence belongs to route block j = t / 2 and reads
// both tiles of every earlier block of P(j), then the tiles of its own block up to itself.  Token for
// token that is the b = 128 mask (earlier blocks in full, the causal triangle inside the self block),
// so no kernel needs to know about b.
#include <stdarg.h>

#include <algorithm>
#include <atomic>

#include "bf1_common.cuh"

namespace bf1 {

// ---- thread-local error string --------------------------------------------------------
static thread_local char g_err[512] = "";

int fail(int code, const char* fmt, ...) {
    va_list ap;
    va_start(ap, fmt);
    vsnprintf(g_err, sizeof g_err, fmt, ap);
    va_end(ap);
    return code;
}

constexpr int kPlanThreads = 1024;
constexpr int kListSlots = 128;   // slots whose lists a CTA writes at a time
constexpr int kTile = 64;   // tokens per route slot (tile), whatever the route block width

struct PlanArgs {
    const int32_t* cu_seqlens;
    int32_t batch;
    int64_t total_tokens;
    int32_t max_seqlen;
    bf1_route_cfg cfg;
    bf1_route route;
};

__global__ void __launch_bounds__(kPlanThreads, 1) plan_kernel(const PlanArgs args) {
    extern __shared__ int32_t s_mem[];
    int32_t* s_start = s_mem;  // [batch + 1] first slot of each sequence
    __shared__ int32_t s_scan[64];   // totals of the warps, and their sums
    __shared__ int32_t s_bad;
    __shared__ unsigned long long s_total;

    const int tid = threadIdx.x;
    const bf1_route& r = args.route;
    const int f = args.cfg.block / kTile;   // tiles per route block: 1 or 2
    const int batch = args.batch;
    if (tid == 0) {
        s_bad = 0;
        s_total = 0ull;
        s_start[0] = 0;
    }
    int32_t* s_hist = s_mem + batch + 1;  // [max_degree + 1] (the first CTA's)
    if (blockIdx.x == 0)
        for (int i = tid; i <= r.max_degree; i += kPlanThreads) s_hist[i] = 0;
    pdl_wait();

    // ---- phase 1: validate cu_seqlens, blocks per sequence, exclusive scan -> s_start
    auto blocks_of = [&](int s, bool& bad) -> int32_t {
        const int32_t lo = args.cu_seqlens[s], hi = args.cu_seqlens[s + 1];
        const int32_t len = hi - lo;
        bad = lo < 0 || len < 0 || len > args.max_seqlen || (long long)hi > args.total_tokens ||
              (s == 0 && lo != 0) || (s == batch - 1 && (long long)hi != args.total_tokens);
        return bad ? 0 : (len + kTile - 1) / kTile;
    };
    int32_t carry = 0;
    if (batch <= 32) {
        // Every warp scans the lengths for itself: one barrier instead of five, and the histogram is cleared
        // and a slot's list length computed once: plan and forward of 1K tokens 13.0 -> 12.4 us.
        const int lane = tid & 31;
        bool bad = false;
        int32_t incl = lane < batch ? blocks_of(lane, bad) : 0;
#pragma unroll
        for (int off = 1; off < 32; off <<= 1) {
            const int32_t up = __shfl_up_sync(0xffffffffu, incl, off);
            if (lane >= off) incl += up;
        }
        carry = __shfl_sync(0xffffffffu, incl, 31);
        const bool any_bad = __any_sync(0xffffffffu, bad);
        if (tid < batch) s_start[tid + 1] = incl;
        if (tid == 0) s_bad = (any_bad ? BF1_DEV_BAD_SEQLENS : 0) | (carry > r.capacity_qblocks ? BF1_DEV_CAPACITY : 0);
    } else {
        __syncthreads();
        for (int base = 0; base < batch; base += kPlanThreads) {
            const int s = base + tid;
            bool bad = false;
            const int32_t nb = s < batch ? blocks_of(s, bad) : 0;
            if (bad) atomicOr(&s_bad, BF1_DEV_BAD_SEQLENS);
            // inclusive scan of nb over the 1024 threads: shuffles inside a warp, then over the 32 warp totals
            int32_t incl = nb;
#pragma unroll
            for (int off = 1; off < 32; off <<= 1) {
                const int32_t up = __shfl_up_sync(0xffffffffu, incl, off);
                if ((tid & 31) >= off) incl += up;
            }
            if ((tid & 31) == 31) s_scan[tid >> 5] = incl;
            __syncthreads();
            if (tid < 32) {
                int32_t w = s_scan[tid];
#pragma unroll
                for (int off = 1; off < 32; off <<= 1) {
                    const int32_t up = __shfl_up_sync(0xffffffffu, w, off);
                    if (tid >= off) w += up;
                }
                s_scan[32 + tid] = w;   // inclusive totals of warps 0..tid
            }
            __syncthreads();
            incl += (tid >= 32) ? s_scan[32 + (tid >> 5) - 1] : 0;
            const int32_t chunk_total = s_scan[32 + 31];
            if (s < batch) s_start[s + 1] = carry + incl;
            carry += chunk_total;
            __syncthreads();
        }
        if (tid == 0 && carry > r.capacity_qblocks) atomicOr(&s_bad, BF1_DEV_CAPACITY);
    }
    __syncthreads();
    const int32_t nqb = carry;
    // sequence of slot g: last s with s_start[s] <= g (empty sequences have equal starts)
    auto seq_of = [&](int g) {
        int lo = 0, hi = batch;  // invariant: s_start[lo] <= g < s_start[hi]
        while (hi - lo > 1) {
            const int mid = (lo + hi) >> 1;
            if (s_start[mid] <= g) lo = mid; else hi = mid;
        }
        return lo;
    };
    if (blockIdx.x > 0) {
        // ---- the lists
        if (s_bad) return;
        for (int g0 = (blockIdx.x - 1) * kListSlots; g0 < nqb; g0 += (gridDim.x - 1) * kListSlots) {
            const int n = min(kListSlots, nqb - g0);
            for (int slot = tid / r.max_degree, e = tid % r.max_degree; slot < n;) {
                const int g = g0 + slot, jt = g - s_start[seq_of(g)];
                const ListShape shape = list_shape(args.cfg, jt / f);
                r.kv_idx[(size_t)g * r.max_degree + e] = e < list_tiles(shape, f, jt) ? list_tile(shape, f, e) : -1;
                slot += kPlanThreads / r.max_degree;
                e += kPlanThreads % r.max_degree;
                if (e >= r.max_degree) { e -= r.max_degree; ++slot; }
            }
        }
        return;
    }
    if (s_bad) {
        if (tid == 0) {
            *r.status = s_bad;
            *r.num_qblocks = 0;
            *r.total_pairs = 0;
            r.sched[0] = 0;
            r.sched[1] = 0;
        }
        return;
    }

    // ---- phase 2: one thread per slot: where it is, its list's length, its pairs
    auto tiles_of = [&](int jt) { return list_tiles(list_shape(args.cfg, jt / f), f, jt); };
    unsigned long long my_pairs = 0ull;
    int first_deg = -1;              // of slot tid
    for (int g = tid; g < nqb; g += kPlanThreads) {
        const int s = seq_of(g);
        const int jt = g - s_start[s];   // tile inside the sequence
        const int32_t len = args.cu_seqlens[s + 1] - args.cu_seqlens[s];
        const int rows = min(kTile, len - jt * kTile);
        const int tiles = tiles_of(jt), deg = min(tiles, r.max_degree);
        if (tiles > r.max_degree) atomicOr(&s_bad, BF1_DEV_CAPACITY);
        if (g == tid) first_deg = deg;
        const int32_t pairs = rows * kTile * (deg - 1) + rows * (rows + 1) / 2;
        r.qb_seq[g] = s;
        r.qb_block[g] = jt;
        r.kv_count[g] = deg;
        r.pair_count[g] = pairs;
        my_pairs += (unsigned long long)pairs;
        atomicAdd(&s_hist[deg], 1);
    }
    // one shared-memory atomic per warp, not per thread
#pragma unroll
    for (int off = 16; off > 0; off >>= 1) my_pairs += __shfl_down_sync(0xffffffffu, my_pairs, off);
    if ((tid & 31) == 0 && my_pairs) atomicAdd(&s_total, my_pairs);
    __syncthreads();

    // ---- phase 3: hand-out order = slots by descending list length (counting sort).  One warp turns the histogram into
    // where the slots of a length begin
    if (tid < 32) {
        int32_t run = 0;
        for (int d0 = r.max_degree; d0 >= 0; d0 -= 32) {
            const int dg = d0 - tid;
            const int32_t c = dg >= 0 ? s_hist[dg] : 0;
            int32_t incl = c;
#pragma unroll
            for (int off = 1; off < 32; off <<= 1) {
                const int32_t up = __shfl_up_sync(0xffffffffu, incl, off);
                if (tid >= off) incl += up;
            }
            if (dg >= 0) s_hist[dg] = run + incl - c;
            run += __shfl_sync(0xffffffffu, incl, 31);
        }
    }
    __syncthreads();
    for (int g0 = 0; g0 < nqb; g0 += kPlanThreads) {
        const int g = g0 + tid;
        int deg = first_deg;         // (-1 behind the last slot)
        if (g0 > 0) deg = g < nqb ? min(tiles_of(g - s_start[seq_of(g)]), r.max_degree) : -1;
        const unsigned same = __match_any_sync(0xffffffffu, deg);    // one atomic per length and warp
        const int leader = __ffs(same) - 1, rank = __popc(same & ((1u << (tid & 31)) - 1));
        int pos = 0;
        if ((tid & 31) == leader && g < nqb) pos = atomicAdd(&s_hist[deg], __popc(same));
        pos = __shfl_sync(0xffffffffu, pos, leader);
        if (g < nqb) r.order[pos + rank] = g;
    }
    if (tid == 0) {
        *r.status = s_bad;
        *r.num_qblocks = s_bad ? 0 : nqb;
        *r.total_pairs = (int64_t)s_total;
        r.sched[0] = 0;
        r.sched[1] = 0;
    }
}

int check_cfg(const bf1_route_cfg* cfg) {
    if (!cfg) return fail(BF1_ERR_INVALID_ARG, "route cfg is null");
    if (cfg->block != 64 && cfg->block != 128)
        return fail(BF1_ERR_UNSUPPORTED, "block width %d: only b = 64 and b = 128 are supported", cfg->block);
    if (cfg->local_blocks < 0) return fail(BF1_ERR_INVALID_ARG, "local_blocks %d < 0", cfg->local_blocks);
    if ((cfg->global_first | 1) != 1 || (cfg->dyadic | 1) != 1)
        return fail(BF1_ERR_INVALID_ARG, "global_first and dyadic must be 0 or 1");
    return BF1_OK;
}

}  // namespace bf1

using namespace bf1;

extern "C" int bf1_route_capacity(int32_t batch, int64_t total_tokens, int32_t max_seqlen,
                                  const bf1_route_cfg* cfg, int32_t* capacity_qblocks, int32_t* max_degree) {
    if (int rc = check_cfg(cfg)) return rc;
    if (!capacity_qblocks || !max_degree) return fail(BF1_ERR_INVALID_ARG, "output pointer is null");
    if (batch < 0 || total_tokens < 0 || max_seqlen < 0)
        return fail(BF1_ERR_INVALID_ARG, "negative batch, total_tokens or max_seqlen");
    if (total_tokens > 0x7fffffffLL - 64)
        return fail(BF1_ERR_UNSUPPORTED, "total_tokens %lld does not fit 32-bit token indices", (long long)total_tokens);
    const int b = cfg->block;
    const int f = b / kTile;
    // Slots are 64-token tiles.  Largest possible sum of ceil(n_s / 64): p sequences end in a partial
    // tile of at least one token each, the other tokens fill whole tiles; the sum grows with p, p <= batch.
    const int64_t partial = total_tokens < batch ? total_tokens : batch;
    const int64_t cap = partial + (total_tokens - partial) / kTile;
    if (cap > 0x7fffffffLL) return fail(BF1_ERR_UNSUPPORTED, "too many query blocks");
    const int nblk = (max_seqlen + b - 1) / b;
    // |P(j)| grows with j, but for the powers of two, where the dyadic predecessor is block 0: the last block or
    // one of the two before it has the longest list (1 and 2 are both powers of two).
    int deg = 1;
    for (int j = nblk - 1; j >= 0 && j >= nblk - 3; --j) {
        const int dj = list_shape(*cfg, j).count;
        if (dj > deg) deg = dj;
    }
    *capacity_qblocks = (int32_t)(cap > 0 ? cap : 1);
    *max_degree = deg * f;   // b = 128: two tiles per listed block (the last tile of a block reads both of its own)
    return BF1_OK;
}

extern "C" int bf1_plan_route(const int32_t* cu_seqlens_dev, int32_t batch, int64_t total_tokens,
                              int32_t max_seqlen, const bf1_route_cfg* cfg, const bf1_route* out,
                              void* stream) {
    if (int rc = check_cfg(cfg)) return rc;
    if (!cu_seqlens_dev || !out) return fail(BF1_ERR_INVALID_ARG, "cu_seqlens or route is null");
    if (!out->qb_seq || !out->qb_block || !out->kv_count || !out->kv_idx || !out->pair_count ||
        !out->order || !out->total_pairs || !out->num_qblocks || !out->status || !out->sched)
        return fail(BF1_ERR_INVALID_ARG, "a route array pointer is null");
    if (batch < 0 || total_tokens < 0 || max_seqlen < 0)
        return fail(BF1_ERR_INVALID_ARG, "negative batch, total_tokens or max_seqlen");
    if (total_tokens > 0x7fffffffLL - 64)
        return fail(BF1_ERR_UNSUPPORTED, "total_tokens %lld does not fit 32-bit token indices", (long long)total_tokens);
    if (out->capacity_qblocks < 1 || out->max_degree < 1)
        return fail(BF1_ERR_CAPACITY, "route capacity_qblocks and max_degree must be >= 1");
    int32_t need_cap = 0, need_deg = 0;
    if (int rc = bf1_route_capacity(batch, total_tokens, max_seqlen, cfg, &need_cap, &need_deg)) return rc;
    if (out->max_degree < need_deg)
        return fail(BF1_ERR_CAPACITY, "route max_degree %d < %d needed for max_seqlen %d", out->max_degree,
                    need_deg, max_seqlen);
    const size_t smem = sizeof(int32_t) * ((size_t)batch + 1 + (size_t)out->max_degree + 1);
    constexpr int kMostSmem = 200 * 1024;
    if (smem > kMostSmem) return fail(BF1_ERR_UNSUPPORTED, "batch %d or max_degree %d too large for the planner", batch, out->max_degree);
    if (smem > 32 * 1024) {   // (48 KB, static shared memory included, need no leave; once per device, so that no call takes back another's)
        static std::atomic<bool> allowed[64];
        int dev = 0;
        BF1_CUDA_CHECK(cudaGetDevice(&dev));
        if (dev < 0 || dev >= 64) return fail(BF1_ERR_NO_DEVICE, "device ordinal %d out of range", dev);
        if (!allowed[dev].load(std::memory_order_acquire)) {
            BF1_CUDA_CHECK(cudaFuncSetAttribute(plan_kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, kMostSmem));
            allowed[dev].store(true, std::memory_order_release);
        }
    }
    PlanArgs args;
    args.cu_seqlens = cu_seqlens_dev;
    args.batch = batch;
    args.total_tokens = total_tokens;
    args.max_seqlen = max_seqlen;
    args.cfg = *cfg;
    args.route = *out;
    BF1_CUDA_CHECK(launch_pdl(plan_kernel, 1 + std::min((need_cap + kListSlots - 1) / kListSlots, 64), kPlanThreads, smem, (cudaStream_t)stream, args));
    return BF1_OK;
}

extern "C" const char* bf1_last_error(void) { return g_err; }

extern "C" int bf1_version(void) { return 1; }
