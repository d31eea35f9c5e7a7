// Route planner: Eq. 1 of the paper evaluated on the device.
//
// For every query block j of every sequence the planner writes the ascending list
// P(j) = {j, j-1, ..., j-W, 0} u {j - 2^k}, its length, and the selected token pairs of the
// block (Proposition 1's accounting).  Lists are generated by merging the three already
// sorted candidate streams (block 0, dyadic predecessors, local window) and dropping
// repeats -- no sort, no search.  One CTA does the whole plan: the problem is a few
// hundred to a few thousand query blocks and launch latency, not throughput, is what a
// caller sees (Section 5.1: at short context the route's bookkeeping and the launch cost more
// than the attention arithmetic).
//
// The attention kernels work on tiles of 64 tokens.  With the route block width b = 128 every slot of
// the route is still one 64-token tile: tile t of a sequence belongs to route block j = t / 2 and reads
// both tiles of every earlier block of P(j), then the tiles of its own block up to itself.  Token for
// token that is the b = 128 mask (earlier blocks in full, the causal triangle inside the self block),
// so no kernel needs to know about b.
#include <stdarg.h>

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
constexpr int kTile = 64;   // tokens per route slot (tile), whatever the route block width

struct PlanArgs {
    const int32_t* cu_seqlens;
    int32_t batch;
    int64_t total_tokens;
    int32_t max_seqlen;
    bf1_route_cfg cfg;
    bf1_route route;
};

// Degree |P(j)| without storing the list (the capacity helper on the host uses it): the same
// merge of the three ascending candidate streams -- block 0, the dyadic predecessors
// j - 2^k (k descending), the local window j - W .. j -- that the planner kernel performs.
__host__ __device__ inline int route_degree(const bf1_route_cfg& c, int j) {
    int deg = 0;
    int last = -1;
    int kmax = -1;
    if (c.dyadic) {
        while ((1 << (kmax + 1)) <= j) ++kmax;  // largest k with 2^k <= j
    }
    int a = c.global_first ? 0 : 0x7fffffff;
    int k = kmax;
    int l = j - c.local_blocks;
    if (l < 0) l = 0;
    while (true) {
        int dcur = (k >= 0) ? j - (1 << k) : 0x7fffffff;
        int lcur = (l <= j) ? l : 0x7fffffff;
        int m = a < dcur ? a : dcur;
        m = m < lcur ? m : lcur;
        if (m == 0x7fffffff) break;
        if (m == a) a = 0x7fffffff;
        if (m == dcur) --k;
        if (m == lcur) ++l;
        if (m != last) { ++deg; last = m; }
    }
    return deg;
}

__global__ void __launch_bounds__(kPlanThreads, 1) plan_kernel(const PlanArgs args) {
    extern __shared__ int32_t s_mem[];
    int32_t* s_start = s_mem;  // [batch + 1] first slot of each sequence
    __shared__ int32_t s_scan[kPlanThreads];
    __shared__ int32_t s_bad;
    __shared__ unsigned long long s_total;
    __shared__ int32_t s_hist_base;  // offset of the histogram inside s_mem

    const int tid = threadIdx.x;
    const bf1_route& r = args.route;
    const int f = args.cfg.block / kTile;   // tiles per route block: 1 or 2
    const int batch = args.batch;
    if (tid == 0) {
        s_bad = 0;
        s_total = 0ull;
        s_start[0] = 0;
        s_hist_base = batch + 1;
    }
    pdl_wait();
    __syncthreads();

    // ---- phase 1: validate cu_seqlens, blocks per sequence, exclusive scan -> s_start
    int32_t carry = 0;
    for (int base = 0; base < batch; base += kPlanThreads) {
        const int s = base + tid;
        int32_t nb = 0;
        if (s < batch) {
            const int32_t lo = args.cu_seqlens[s], hi = args.cu_seqlens[s + 1];
            const int32_t len = hi - lo;
            if (lo < 0 || len < 0 || len > args.max_seqlen || (long long)hi > args.total_tokens ||
                (s == 0 && lo != 0) || (s == batch - 1 && (long long)hi != args.total_tokens)) {
                atomicOr(&s_bad, BF1_DEV_BAD_SEQLENS);
            } else {
                nb = (len + kTile - 1) / kTile;
            }
        }
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
    const int32_t nqb = carry;
    if (tid == 0 && nqb > r.capacity_qblocks) atomicOr(&s_bad, BF1_DEV_CAPACITY);
    __syncthreads();
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

    // ---- phase 2: one thread per slot builds its list
    int32_t* s_hist = s_mem + s_hist_base;  // [max_degree + 1]
    for (int i = tid; i <= r.max_degree; i += kPlanThreads) s_hist[i] = 0;
    __syncthreads();

    unsigned long long my_pairs = 0ull;
    for (int g = tid; g < nqb; g += kPlanThreads) {
        // sequence of slot g: last s with s_start[s] <= g (empty sequences have equal starts)
        int lo = 0, hi = batch;  // invariant: s_start[lo] <= g < s_start[hi]
        while (hi - lo > 1) {
            const int mid = (lo + hi) >> 1;
            if (s_start[mid] <= g) lo = mid; else hi = mid;
        }
        const int s = lo;
        const int jt = g - s_start[s];   // tile inside the sequence
        const int j = jt / f;            // its route block
        const int32_t len = args.cu_seqlens[s + 1] - args.cu_seqlens[s];
        const int rows = min(kTile, len - jt * kTile);

        int32_t* list = r.kv_idx + (size_t)g * r.max_degree;
        int deg = 0, last = -1;
        int kmax = -1;
        if (args.cfg.dyadic) {
            while ((1 << (kmax + 1)) <= j) ++kmax;
        }
        int a = args.cfg.global_first ? 0 : 0x7fffffff;
        int k = kmax;
        int l = max(j - args.cfg.local_blocks, 0);
        bool overflow = false;
        while (true) {
            const int dcur = (k >= 0) ? j - (1 << k) : 0x7fffffff;
            const int lcur = (l <= j) ? l : 0x7fffffff;
            const int m = min(a, min(dcur, lcur));
            if (m == 0x7fffffff) break;
            if (m == a) a = 0x7fffffff;
            if (m == dcur) --k;
            if (m == lcur) ++l;
            if (m != last) {
                // an earlier block: all of its tiles; the self block: its tiles up to this one
                const int t0 = m * f, t1 = (m < j) ? m * f + f - 1 : jt;
                for (int t = t0; t <= t1; ++t) {
                    if (deg < r.max_degree) list[deg] = t; else overflow = true;
                    ++deg;
                }
                last = m;
            }
        }
        if (overflow) {
            atomicOr(&s_bad, BF1_DEV_CAPACITY);
            deg = r.max_degree;
        }
        for (int e = deg; e < r.max_degree; ++e) list[e] = -1;
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

    // ---- phase 3: hand-out order = slots by descending list length (counting sort)
    if (tid == 0) {
        int32_t run = 0;
        for (int dg = r.max_degree; dg >= 0; --dg) {
            const int32_t c = s_hist[dg];
            s_hist[dg] = run;
            run += c;
        }
    }
    __syncthreads();
    for (int g = tid; g < nqb; g += kPlanThreads) {
        const int pos = atomicAdd(&s_hist[r.kv_count[g]], 1);
        r.order[pos] = g;
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
    int deg = 1;
    // |P(j)| is largest just below a power of two; scan the last octave
    for (int j = nblk > 1 ? (nblk - 1) / 2 : 0; j < nblk; ++j) {
        const int dj = route_degree(*cfg, j);
        if (dj > deg) deg = dj;
    }
    for (int j = 0; j < nblk && j < 64; ++j) {
        const int dj = route_degree(*cfg, j);
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
    if (smem > 200 * 1024) return fail(BF1_ERR_UNSUPPORTED, "batch %d or max_degree %d too large for the planner", batch, out->max_degree);
    if (smem > 48 * 1024)
        BF1_CUDA_CHECK(cudaFuncSetAttribute(plan_kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem));
    PlanArgs args;
    args.cu_seqlens = cu_seqlens_dev;
    args.batch = batch;
    args.total_tokens = total_tokens;
    args.max_seqlen = max_seqlen;
    args.cfg = *cfg;
    args.route = *out;
    BF1_CUDA_CHECK(launch_pdl(plan_kernel, 1, kPlanThreads, smem, (cudaStream_t)stream, args));
    return BF1_OK;
}

extern "C" const char* bf1_last_error(void) { return g_err; }

extern "C" int bf1_version(void) { return 1; }
