// BF1 attention backward (dQ, dK, dV) over the same route, for sm_100a (head dimension 64 or 128,
// 1, 2 or 4 query heads per KV head).
//
// The paper's correctness gates include a backward pass with finite Q, K and V gradients (Section
// 4.2).  With P = exp(S - LSE) recomputed from the saved LSE and D_i = <dO_i, O_i>:
//     dV_p += P^T dO,   dP = dO V_p^T,   dS = P o (dP - D) * scale,   dQ += dS K_p,   dK_p += dS^T Q.
// dQ of a query block sums over the KV blocks of its list; dK / dV of a KV block sum over the query
// blocks that read it.  Nothing is ever added in global memory (no atomics, no fp32 gradient buffers, the same
// bits on every run).  One call is three launches:
//
//   bwd_prep_kernel  D_i for every row (one pass over dO and O), and beside it, in one CTA, the INVERSE route:
//                    the readers of every KV block, derived from the lists on every call (any lists: the
//                    planner's or the caller's).
//   bwd_dkv_kernel   unit = (KV block p, KV head, a run of the query blocks that read p).  Per reader j and pair
//                    of query heads (the two heads are the 128 rows of every MMA):
//                        S  = Q  K_p^T   (128 x 64 x d)    A, B K-major from shared memory
//                        dP = dO V_p^T   (128 x 64 x d)
//                        dV^T += dO^T P  (d x 64 x 128)    A = dO MN-major, B = P MN-major ([q][kv] tile)
//                        dK^T += Q^T  dS (d x 64 x 128)    A = Q MN-major,  B = dS MN-major
//                    accumulating in tensor memory across all readers (head dimension on the lanes), and
//                    one store at the end.  A block with more readers than a run (2 to 16 of them, by the size of the problem)
//                    is cut into runs handled by different CTAs that leave fp32 partial sums.
//                    The dS tiles (bf16, 16 KB each) also go to the workspace, one per list entry.
//   bwd_dq_kernel    unit = (query block, KV head, pair of query heads): dQ += dS K_p over the list, dS as the
//                    dK/dV kernel left it; and, in warps of their own, the partial sums added up in run order.
//
// Keeping dS costs 32 KB of traffic per list entry, KV head and pair; computing it again costs two more MMA passes (S and
// dP), the exponentials and the V tiles.  Measured (recomputed -> kept,
// inverse route and D_i included): 0.135 -> 0.115 ms for forward and backward of 4K tokens (16 query heads, d = 128),
// 1.02 -> 0.944 ms at 32K.
// A route whose dS would not fit (kDsMost for one KV head) is run by bwd_dq_recompute_kernel instead.
//
// The compute kernels are persistent: one CTA of 11 or 16 warps per SM that walks through its share of the units, with
// warps for copies, for issuing MMAs, for the arithmetic on S and dP and for reading finished sums out, so that copies,
// MMAs and arithmetic of neighbouring entries and units overlap (see the comment in front of each kernel).  P is rounded
// to bf16 before the MMAs, as in the forward.  With d = 64 the transposed products still run as M = 128 MMAs:
// tensor-memory lanes 64..127 then hold nothing of value and are not read.
#include <cuda.h>

#include <algorithm>
#include <atomic>

#include "bf1_common.cuh"

namespace bf1 {

constexpr int kBlock64 = 64;     // b: tokens per block
constexpr int kLeastChunk = 2, kMostChunk = 16;   // readers per dK/dV unit (run_length() chooses)
constexpr int kSms = 148;        // (sizes of the workspace only)
constexpr int kDsTile = 128 * 64 * 2;          // bytes of one dS tile: [128 q rows][64 kv], 128-byte rows, swizzled
constexpr int64_t kDsGroup = 1LL << 30;        // dS kept at a time: as many KV heads as fit this (at least one)
// One KV head's dS larger than this is not kept but computed again.  Keeping it is faster at every size that was measured, so
// the line is drawn by what a caller may be asked for.  Kept against computed again (a backward with one KV head, two
// query heads, d = 128): 4K tokens 41 / 54 us, 32K 107 / 136, 262K (0.9 GB) 953 / 1114, 1M (4.3 GB) 4895 / 5450; 64K
// tokens with windows of 63 blocks (1.1 GB) 880 / 1041, of 500 (8.4 GB) 5240 / 5810.
constexpr int64_t kDsMost = 8LL << 30;

// The inverse route and the units of bwd_dkv_kernel, all inside the caller's workspace.
struct InvPlan {
    int32_t* count;       // [cap] readers of KV slot g (with multiplicity); behind them, of the several-launch path, whether some
                          // list entry names no slot
    int32_t* start;       // [cap + 1] first reader of slot g in `readers`
    int32_t* unit0;       // [cap + 1] first unit of slot g
    int32_t* chunks;      // [cap] runs the slot's readers are cut into
    int32_t* part0;       // [cap] first partial-sum slot of a slot with more than one run, else -1
    int32_t* readers;     // [cap * max_degree] list entries (query slot * max_degree + place), ascending per KV slot
    int4* units;          // [max_units][2] longest first: {KV slot, first reader, readers, partial-sum slot or -1 (it
                          // writes the final bf16 rows)}, {first token of the sequence, block, tokens of the sequence, -}
    int4* ranked;         // [cap][2] the query blocks in the order of the dQ units: {slot, list entries, block, first token of the
                          // sequence}, {tokens of the sequence, -, -, -}
    int32_t* tickets;     // [hkv] hand-out counters of the dK/dV launches, by first KV head
    int32_t* multi;       // [cap] the KV slots whose readers were cut into more than one run
    int32_t* scalars;     // [8] number of units, total readers, chunk, partial slots, slots in `multi`
    int32_t cap, max_units, max_parts;
};

struct BwdArgs {
    const int32_t* cu_seqlens;
    const int32_t* qb_seq;
    const int32_t* qb_block;
    const int32_t* kv_count;
    const int32_t* kv_idx;
    const int32_t* num_qblocks;
    const int32_t* order;      // may be null
    int32_t batch, max_degree, capacity, total_tokens, hq, hkv, group;
    int32_t head0, nheads; // KV heads this launch works on: head0 .. head0 + nheads - 1
    int32_t sms;           // of this GPU
    int32_t interleave;    // 1: units of all KV heads interleaved (longest first over all heads); 0: KV head by KV head
    int32_t* status;
    float scale, scale_log2;
    const __nv_bfloat16* o;
    const __nv_bfloat16* d_o;
    const float* lse;
    float* delta;          // [hq, T] D_i = <dO_i, O_i>
    __nv_bfloat16* ds;     // [nheads][pairs][cap * max_degree] dS tiles of kDsTile bytes, or null: not kept
    __nv_bfloat16* dq;
    __nv_bfloat16* dk;
    __nv_bfloat16* dv;
    float* partial;        // [partial slots][hkv][2][64][d] fp32 sums of the runs of a many-reader block
    InvPlan inv;
};

// The sequence of a slot.
__device__ __forceinline__ int slot_seq(const BwdArgs& a, int g) { return a.batch > 1 ? a.qb_seq[g] : 0; }
__device__ __forceinline__ int safe_entry(int p, int e, int cnt, int j) {
    if (p < 0 || p > j || (e == cnt - 1) != (p == j)) p = (e == cnt - 1) ? j : 0;
    return p;
}
// Entry e of a list as every kernel of this library uses it: kept inside [0, j], the last entry the
// query block itself, whatever the array holds (a caller's route may be wrong; the forward flags it).
__device__ __forceinline__ int list_entry(const int32_t* list, int e, int cnt, int j) {
    return safe_entry(list[e], e, cnt, j);
}

// ---- pieces shared by the two compute kernels ------------------------------------------------------------------

// S = Q K^T (or dP = dO V^T): D / 16 k-steps over the head dimension, 128 x 64 output, A and B K-major (one thread).
template <int D>
__device__ __forceinline__ void issue_qk(uint32_t t_out, uint32_t sA, uint32_t sB) {
    constexpr uint32_t kHi = desc_hi_sw128(1024);
    constexpr uint32_t kIdS = idesc_bf16_f32_ab(64, false, false);
#pragma unroll
    for (int kk = 0; kk < D / 16; ++kk) {
        const uint32_t a_off = ((kk / 4) * 16384 + (kk % 4) * 32) >> 4, b_off = ((kk / 4) * 8192 + (kk % 4) * 32) >> 4;
        if (kk == 0) mma_ss_lohi<false>(t_out, desc_lo_sw128(sA, 16) + a_off, desc_lo_sw128(sB, 16) + b_off, kHi, kIdS);
        else mma_ss_lohi<true>(t_out, desc_lo_sw128(sA, 16) + a_off, desc_lo_sw128(sB, 16) + b_off, kHi, kIdS);
    }
}
template <int D>
__device__ __forceinline__ void issue_s_dp(uint32_t t_s, uint32_t t_dp, uint32_t sQ, uint32_t sDO, uint32_t sK, uint32_t sV) {
    issue_qk<D>(t_s, sQ, sK);
    issue_qk<D>(t_dp, sDO, sV);
}

// P and dS of this thread's 32 columns (half = 0 / 1: columns 0..31 / 32..63) of its row, from S and dP in tensor
// memory.  Masked entries get s = -inf (self block, warp-uniform branch) and rows outside the sequence an infinite
// LSE: both give P = 0 exactly, and with it dS = 0.  Results as packed bf16 pairs.
__device__ __forceinline__ void p_and_ds(uint32_t t_s, uint32_t t_dp, int half, int tl, bool diag, float lse_row2, float drow,
                                         float scale, float scale_log2, uint32_t (&pw)[16], uint32_t (&dw)[16]) {
    const uint64_t c2p = pack2(scale_log2, scale_log2), nlp = pack2(-lse_row2, -lse_row2);
    const uint64_t scp = pack2(scale, scale), ndp = pack2(-drow * scale, -drow * scale);
    uint32_t sr[32], dr[32];
    tmem_ld32(t_s + half * 32, sr);
    tmem_ld32(t_dp + half * 32, dr);
    tmem_wait_ld();
    if (diag) {
#pragma unroll
        for (int c = 0; c < 32; ++c)
            if (half * 32 + c > tl) sr[c] = 0xff800000u;   // -inf: causal triangle
    }
#pragma unroll
    for (int c = 0; c < 16; ++c) {
        const uint64_t x = fma2(pack2(__uint_as_float(sr[2 * c]), __uint_as_float(sr[2 * c + 1])), c2p, nlp);
        float x0, x1;
        unpack2(x, x0, x1);
        const float p0 = ex2_approx(x0), p1 = ex2_approx(x1);
        // dS = P * (dP - D) * scale
        const uint64_t t = fma2(pack2(__uint_as_float(dr[2 * c]), __uint_as_float(dr[2 * c + 1])), scp, ndp);
        float d0, d1;
        unpack2(mul2(pack2(p0, p1), t), d0, d1);
        pw[c] = pack_bf16x2(p0, p1);
        dw[c] = pack_bf16x2(d0, d1);
    }
}

// The same pairs as a bf16 row piece in shared memory: 128-byte rows, 16-byte chunks XOR-swizzled with the row
// (the layout the MMAs read as an MN-major operand).
__device__ __forceinline__ void store_row_piece(uint32_t row_addr, int row, int half, const uint32_t (&w)[16]) {
#pragma unroll
    for (int c4 = 0; c4 < 4; ++c4) {                          // 16-byte chunk half * 4 + c4 of the 128-byte row
        const int ch = (half * 4 + c4) ^ (row & 7);
        st_shared_v4(row_addr + (ch << 4), w[4 * c4], w[4 * c4 + 1], w[4 * c4 + 2], w[4 * c4 + 3]);
    }
}

// One head per KV head: rows 64..127 of every column chunk of the Q and dO tiles are never written by a copy;
// the MMAs still read them, so they are cleared once (they then give P = 0 and dS = 0 like rows past a sequence).
template <int D>
__device__ __forceinline__ void clear_idle_rows(uint32_t sQ, uint32_t sDO, int tid, int threads) {
    for (int i = tid; i < 2 * (D / 64) * 512; i += threads) {
        const int which = i / ((D / 64) * 512), ch = (i / 512) % (D / 64), off = i % 512;
        st_shared_v4((which ? sDO : sQ) + ch * 16384 + 8192 + off * 16, 0u, 0u, 0u, 0u);
    }
    fence_proxy_async();
}

// One Q-shaped tile (Q, dO or O) of a query block and pair of heads (one thread; expect_tx is the caller's).
template <int D>
__device__ __forceinline__ void load_q_tile(uint32_t dst, const CUtensorMap* tm, int tok0, int head, int group, uint32_t bar) {
    if (group > 1) {
        tma_load_4d(dst, tm, 0, tok0, head, 0, bar);
    } else {
#pragma unroll
        for (int ch = 0; ch < D / 64; ++ch) tma_load_4d(dst + ch * 16384, tm, 0, tok0, head, ch, bar);
    }
}

// ---- dQ from recomputed dS ---------------------------------------------------------------------------------------
//
// For routes whose dS tiles would not fit the workspace.
//
// One persistent CTA of 16 warps per SM.  Units (query block, KV head, pair of heads) are dealt out statically, in
// the route's longest-list-first order KV head by KV head, back and forth over the CTAs so that each gets the same
// mix.  Everything a unit needs travels through rings whose next entry is under way while the current one is in
// use, across unit boundaries as well:
//     warp 0    copies Q of every unit (two buffers) and the K tile of every list entry (ring of kStages)
//     warp 1    copies dO of every unit and the V tiles
//     warp 2    issues S and dP of every entry into one of two S/dP buffers in tensor memory, as soon as the K / V
//               tiles are there and the dQ MMAs that read the buffer's last dS are done
//     warp 3    issues the dQ MMAs of every entry; dQ accumulates in one of two buffers
//     warps 4-11   the arithmetic on S and dP, two threads per tile row (32 key columns each); dS (bf16) goes back
//               into tensor memory over S, from where the dQ MMAs read it as their A operand
//     warps 12-15   per unit: D_i and the LSE of every row into shared memory one unit ahead; then the finished dQ
//               tile of the unit before, from tensor memory to global memory
// Every wait of a role is on a barrier it waits on once per phase, in phase order: a parity wait is only
// meaningful one phase ahead.
constexpr int kDqrThreads = 512;
constexpr int kStages = 3;
// Q / dO buffer (and barrier) of unit n, and the parity of its n-th use
__device__ __forceinline__ int qbuf(int n) { return n & 1; }
__device__ __forceinline__ uint32_t qpar(int n) { return (n >> 1) & 1; }

template <int D>
struct DqrSmem {
    static constexpr int kQBytes = 128 * D * 2;      // Q / dO / O tile [D / 64 chunks][128 rows][128 B]
    static constexpr int kKVBytes = 64 * D * 2;      // K / V tile      [D / 64 chunks][64 rows][128 B]
    static constexpr int kQ = 0;                     // [2]
    static constexpr int kDO = kQ + 2 * kQBytes;     // [2]
    static constexpr int kRing = kDO + 2 * kQBytes;  // [kStages] of K | V
    static constexpr int kRow = kRing + kStages * 2 * kKVBytes;   // D_i [2][128], LSE [2][128] (fp32)
    static constexpr int kBar = kRow + 2048;
    static constexpr int kUsed = kBar + 512;
    // at least this much is requested so that a second CTA never fits an SM: each allocates all of tensor memory
    static constexpr int kTotal = kUsed > 120 * 1024 ? kUsed : 120 * 1024;
};

struct DqUnit {
    int ok, slot, kvh, pair, cnt, seq0, seqlen, j, tok0, rows_valid;
};

// The query block of rank r in the hand-out order, looked up for the dQ kernel (by the preparation, beside the pass over dO and O): a
// chain of three loads that would stand in front of its first copy (backward of 1000 and 4096 tokens 0.4 and 1 us shorter for it).
__device__ __forceinline__ void rank_query_block(const BwdArgs& a, int r, int nqb) {
    const int slot = min(max(a.order ? a.order[r] : r, 0), nqb - 1), seq = min(max(slot_seq(a, slot), 0), a.batch - 1);
    const int seq0 = a.cu_seqlens[seq];
    a.inv.ranked[2 * r] = make_int4(slot, min(max(a.kv_count[slot], 1), a.max_degree), a.qb_block[slot], seq0);
    a.inv.ranked[2 * r + 1] = make_int4(a.cu_seqlens[seq + 1] - seq0, 0, 0, 0);
}
// Unit n of this CTA (see above for the order).
__device__ __forceinline__ DqUnit dq_unit(const BwdArgs& a, int n, int nqb, int pairs) {
    DqUnit u;
    const int per_head = nqb * pairs, total = per_head * a.nheads;
    const int G = gridDim.x;
    const int i = n * G + ((n & 1) ? G - 1 - (int)blockIdx.x : (int)blockIdx.x);
    u.ok = i < total;
    u.slot = u.kvh = u.pair = u.seq0 = u.seqlen = u.j = u.tok0 = 0;
    u.cnt = 1;
    u.rows_valid = 0;
    if (u.ok) {
        int rank;
        if (a.interleave) {          // rank-major: the longest lists of all heads first
            const int per_rank = pairs * a.nheads;
            rank = i / per_rank;
            const int rem = i - rank * per_rank;
            u.kvh = rem / pairs;
            u.pair = rem - u.kvh * pairs;
        } else {                     // head-major: a head's K and V stay hot in L2
            u.kvh = i / per_head;
            const int rem = i - u.kvh * per_head;
            rank = rem / pairs;
            u.pair = rem - rank * pairs;
        }
        u.kvh += a.head0;
        const int4 x = a.inv.ranked[2 * rank];
        u.slot = x.x;
        u.cnt = x.y;
        u.j = x.z;
        u.seq0 = x.w;
        u.seqlen = a.inv.ranked[2 * rank + 1].x;
        u.rows_valid = min(kBlock64, u.seqlen - u.j * kBlock64);
        u.tok0 = u.seq0 + u.j * kBlock64;
    }
    return u;
}

__device__ __forceinline__ void named_sync(int id, int threads) {
    asm volatile("bar.sync %0, %1;" ::"r"(id), "r"(threads) : "memory");
}

template <int D>
__global__ void __launch_bounds__(kDqrThreads, 1) bwd_dq_recompute_kernel(const __grid_constant__ CUtensorMap tm_q,
                                                                       const __grid_constant__ CUtensorMap tm_k,
                                                                       const __grid_constant__ CUtensorMap tm_v,
                                                                       const __grid_constant__ CUtensorMap tm_do,
                                                                       const BwdArgs a) {
    using L = DqrSmem<D>;
    extern __shared__ __align__(1024) uint8_t smem[];
    uint32_t& s_tmem = *reinterpret_cast<uint32_t*>(smem + L::kBar + 496);
    int& s_abort = *reinterpret_cast<int*>(smem + L::kBar + 500);
    float* s_drow = reinterpret_cast<float*>(smem + L::kRow);          // [2][128]
    float* s_lse = s_drow + 256;                                       // [2][128]
    const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31;
    if (a.status && (*a.status & BF1_DEV_WAIT_TIMEOUT)) return;
    const int nqb = a.inv.scalars[0] ? min(*a.num_qblocks, a.capacity) : 0;   // (no units: no gradients of this route)
    const int pairs = a.group == 4 ? 2 : 1;

    const uint32_t base = smem_u32(smem);
    const uint32_t bars = base + L::kBar;
    // barriers (8 bytes each)
    const uint32_t qdo_full = bars;                          // [2] Q and dO of a unit landed (both copy warps announce bytes)
    const uint32_t qdo_free = qdo_full + 16;                 // [2] the unit's MMAs are done
    const uint32_t row_full = qdo_free + 16;                 // [2] D_i and LSE of the unit's rows are in shared memory
    const uint32_t row_free = row_full + 16;                 // [2] ... and have been read by both arithmetic groups (8 warps)
    const uint32_t sdp_full = row_free + 16;                 // [2] S and dP of an entry computed
    const uint32_t ds_ready = sdp_full + 16;                 // [2] dS written (8 warps)
    const uint32_t dq_full = ds_ready + 16;                  // [2] the unit's dQ is complete
    const uint32_t dq_free = dq_full + 16;                   // [2] ... and has been read out of tensor memory
    const uint32_t dq_done = dq_free + 16;                   // [2] the dQ MMAs that read dS from an S / dP buffer are done
    const uint32_t kv_full = dq_done + 16;                   // [kStages] a K and a V tile landed (both copy warps announce bytes)
    const uint32_t ring_free = kv_full + 8 * kStages;        // [kStages] the stage's tiles have been used
    static_assert(144 + 16 * kStages <= 496, "barriers overlap the words behind them");
    if (tid == 0) {
        s_abort = (base & 1023u) ? 1 : 0;
        if (s_abort && a.status) atomicOr(a.status, BF1_DEV_WAIT_TIMEOUT);
        for (int b = 0; b < 2; ++b) {
            mbar_init(qdo_full + 8 * b, 2);
            mbar_init(qdo_free + 8 * b, 1);
            mbar_init(row_full + 8 * b, 1);
            mbar_init(row_free + 8 * b, 8);
            mbar_init(sdp_full + 8 * b, 1);
            mbar_init(ds_ready + 8 * b, 8);
            mbar_init(dq_full + 8 * b, 1);
            mbar_init(dq_free + 8 * b, 1);
            mbar_init(dq_done + 8 * b, 1);
        }
        for (int s = 0; s < kStages; ++s) {
            mbar_init(kv_full + 8 * s, 2);
            mbar_init(ring_free + 8 * s, 1);
        }
        fence_mbar_init();
    }
    __syncwarp();
    if (warp == 0) {
        tmem_alloc(smem_u32(&s_tmem), 512);
        tmem_relinquish();
    }
    if (a.group == 1) {   // one head per KV head: rows 64..127 of the Q / dO buffers are never written by a copy
        clear_idle_rows<D>(base + L::kQ, base + L::kDO, tid, kDqrThreads);
        clear_idle_rows<D>(base + L::kQ + L::kQBytes, base + L::kDO + L::kQBytes, tid, kDqrThreads);
    }
    tc_fence_before();
    __syncthreads();
    tc_fence_after();
    const uint32_t tmem = s_tmem;
    volatile int* abort_flag = &s_abort;
    if (s_abort) {   // (uniform over the CTA)
        __syncthreads();
        if (warp == 0) tmem_dealloc(tmem, 512);
        return;
    }
    // tensor memory: S | dP of buffer b at columns 128 b (dS takes over columns 0..15 and 32..47 of S), dQ of
    // buffer b at 256 + 128 b
    constexpr uint32_t kColDP = 64, kColDQ = 256;
    const uint32_t q_tx = a.group > 1 ? L::kQBytes : L::kQBytes / 2;   // one head per KV head: half a tile per copy set
    auto stage_k = [&](int s) { return base + L::kRing + s * 2 * L::kKVBytes; };
    auto stage_v = [&](int s) { return base + L::kRing + s * 2 * L::kKVBytes + L::kKVBytes; };

    if (warp == 0 || warp == 1) {
        // ---- copies ----
        const bool first = warp == 0;
        int r = 0;                      // ring entries so far: stage r % kStages, its phase r / kStages
        int rs = 0, rk = 0;             // the same as (stage, phase counter)
        auto ring_wait_free = [&]() {
            if (r >= kStages) mbar_wait(ring_free + 8 * rs, (rk - 1) & 1, abort_flag, a.status);
        };
        auto ring_next = [&]() {
            ++r;
            if (++rs == kStages) { rs = 0; ++rk; }
        };
        DqUnit u = dq_unit(a, 0, nqb, pairs);
        for (int n = 0; u.ok; ++n) {
            const DqUnit un = dq_unit(a, n + 1, nqb, pairs);
            const int head0 = u.kvh * a.group + u.pair * 2;
            const int32_t* list = a.kv_idx + (size_t)u.slot * a.max_degree;
            const int qb = qbuf(n);
            if (n >= 2) mbar_wait(qdo_free + 8 * qb, qpar(n - 2), abort_flag, a.status);
            if (elect_one()) {
                mbar_expect_tx(qdo_full + 8 * qb, q_tx);
                if (first) load_q_tile<D>(base + L::kQ + qb * L::kQBytes, &tm_q, u.tok0, head0, a.group, qdo_full + 8 * qb);
                else load_q_tile<D>(base + L::kDO + qb * L::kQBytes, &tm_do, u.tok0, head0, a.group, qdo_full + 8 * qb);
            }
            __syncwarp();
            for (int it = 0; it < u.cnt; ++it) {
                const int p = list_entry(list, it, u.cnt, u.j);
                ring_wait_free();
                if (elect_one()) {
                    mbar_expect_tx(kv_full + 8 * rs, L::kKVBytes);
                    if (first) tma_load_4d(stage_k(rs), &tm_k, 0, u.seq0 + p * kBlock64, u.kvh, 0, kv_full + 8 * rs);
                    else tma_load_4d(stage_v(rs), &tm_v, 0, u.seq0 + p * kBlock64, u.kvh, 0, kv_full + 8 * rs);
                }
                __syncwarp();
                ring_next();
            }
            u = un;
        }
    } else if (warp == 2 || warp == 3) {
        // ---- MMAs: warp 2 issues S and dP of every entry, warp 3 its dQ.  Two warps, because what surrounds a batch of
        // MMAs (barrier round trips through shared memory, the unit bookkeeping) costs several hundred cycles per
        // entry, during which a single issuing warp would leave the pipe empty. ----
        constexpr uint32_t kHi = desc_hi_sw128(1024);
        constexpr uint32_t kIdQ = idesc_bf16_f32(D, true);             // dQ: 128 x d, A from tensor memory, B (K tile) MN-major
        DqUnit u = dq_unit(a, 0, nqb, pairs);
        int t = 0, rs = 0;                 // entries so far; ring stage of the entry
        uint32_t kv_phase = 0;             // per stage: parity of the K / V tiles put into it so far
        for (int n = 0; u.ok; ++n) {
            const DqUnit un = dq_unit(a, n + 1, nqb, pairs);
            const int b = n & 1;
            if (warp == 2) mbar_wait(qdo_full + 8 * b, qpar(n), abort_flag, a.status);
            else if (n >= 2) mbar_wait(dq_free + 8 * b, qpar(n - 2), abort_flag, a.status);
            for (int it = 0; it < u.cnt; ++it) {
                const int sb = t & 1;
                if (warp == 2) {
                    // the buffer's last dS must have been read by its dQ MMAs before S overwrites it
                    if (t >= 2) mbar_wait(dq_done + 8 * sb, ((t >> 1) - 1) & 1, abort_flag, a.status);
                    mbar_wait(kv_full + 8 * rs, (kv_phase >> rs) & 1, abort_flag, a.status);
                    tc_fence_after();
                    if (elect_one()) {
                        issue_s_dp<D>(tmem + sb * 128, tmem + sb * 128 + kColDP, base + L::kQ + b * L::kQBytes,
                                      base + L::kDO + b * L::kQBytes, stage_k(rs), stage_v(rs));
                        mma_commit(sdp_full + 8 * sb);
                    }
                    __syncwarp();
                } else {
                    mbar_wait(ds_ready + 8 * sb, (t >> 1) & 1, abort_flag, a.status);
                    tc_fence_after();
                    if (elect_one()) {
                        // dQ += dS K: A = dS [128 q][64 kv] from tensor memory (16 kv = 8 columns per step; keys 0..31 sit in
                        // columns 0..15, keys 32..63 in columns 32..47), B = K tile MN-major (16 kv rows = 2048 bytes per step,
                        // next 64 d columns 8 KB away)
#pragma unroll
                        for (int kk = 0; kk < 4; ++kk) {   // 64 kv rows in steps of 16
                            const uint32_t blo = desc_lo_sw128(stage_k(rs), 8192) + ((kk * 2048) >> 4);
                            const uint32_t a_ds = tmem + sb * 128 + (kk >> 1) * 32 + (kk & 1) * 8;
                            if (kk == 0) {
                                if (it == 0) mma_ts_lohi<false>(tmem + kColDQ + b * 128, a_ds, blo, kHi, kIdQ);
                                else mma_ts_lohi<true>(tmem + kColDQ + b * 128, a_ds, blo, kHi, kIdQ);
                            } else {
                                mma_ts_lohi<true>(tmem + kColDQ + b * 128, a_ds, blo, kHi, kIdQ);
                            }
                        }
                        mma_commit(dq_done + 8 * sb);
                        mma_commit(ring_free + 8 * rs);
                        if (it == u.cnt - 1) {
                            mma_commit(dq_full + 8 * b);
                            mma_commit(qdo_free + 8 * b);
                        }
                    }
                    __syncwarp();
                }
                kv_phase ^= 1u << rs;
                ++t;
                if (++rs == kStages) rs = 0;
            }
            u = un;
        }
    } else if (warp >= 4 && warp < 12) {
        // ---- arithmetic on S and dP: two threads per tile row (head hl, token tl), warps 4-7 on key columns 0..31 and
        // warps 8-11 on columns 32..63 of every entry ----
        const int half = (warp - 4) >> 2;
        const uint32_t t_lane = tmem + (static_cast<uint32_t>((warp & 3) * 32) << 16);
        const int row = tid & 127, tl = row & 63;
        int t = 0;
        DqUnit u = dq_unit(a, 0, nqb, pairs);
        for (int n = 0; u.ok; ++n) {
            const DqUnit un = dq_unit(a, n + 1, nqb, pairs);
            const int b = n & 1;
            mbar_wait(row_full + 8 * b, (n >> 1) & 1, abort_flag, a.status);
            const float Drow = s_drow[b * 128 + row], lse2 = s_lse[b * 128 + row];
            for (int it = 0; it < u.cnt; ++it, ++t) {
                const int sb = t & 1;
                mbar_wait(sdp_full + 8 * sb, (t >> 1) & 1, abort_flag, a.status);
                tc_fence_after();
                uint32_t pw[16], dw[16];
                p_and_ds(t_lane + sb * 128, t_lane + sb * 128 + kColDP, half, tl, it == u.cnt - 1, lse2, Drow, a.scale, a.scale_log2, pw, dw);
                // dS as the A operand of the dQ MMAs: bf16 pairs, written over the first 16 of the 32 S columns just read
                tmem_st16(t_lane + sb * 128 + half * 32, dw);
                tmem_wait_st();
                tc_fence_before();
                __syncwarp();
                if (lane == 0) mbar_arrive(ds_ready + 8 * sb);
            }
            __syncwarp();
            if (lane == 0) mbar_arrive(row_free + 8 * b);
            u = un;
        }
    } else if (warp >= 12) {
        // ---- per unit: D_i and LSE one unit ahead; the finished dQ tile of the unit before ----
        const uint32_t t_lane = tmem + (static_cast<uint32_t>((warp & 3) * 32) << 16);
        const int row = tid & 127, hl = row >> 6, tl = row & 63;
        auto prologue = [&](const DqUnit& u, int n) {
            const int b = n & 1;
            const int h = u.kvh * a.group + u.pair * 2 + hl, tok = u.tok0 + tl;
            const bool row_ok = tl < u.rows_valid && u.pair * 2 + hl < a.group;   // G = 1: rows 64..127 belong to no head
            float lse2 = INFINITY, Drow = 0.f;
            if (row_ok) {
                lse2 = a.lse[(size_t)h * a.total_tokens + tok] * 1.4426950408889634f;
                Drow = a.delta[(size_t)h * a.total_tokens + tok];
            }
            if (n >= 2) mbar_wait(row_free + 8 * b, ((n >> 1) - 1) & 1, abort_flag, a.status);
            s_drow[b * 128 + row] = Drow;
            s_lse[b * 128 + row] = lse2;
            named_sync(1, 128);
            if ((tid & 127) == 0) mbar_arrive(row_full + 8 * b);
        };
        DqUnit u = dq_unit(a, 0, nqb, pairs);
        if (u.ok) prologue(u, 0);
        for (int n = 0; u.ok; ++n) {
            const DqUnit un = dq_unit(a, n + 1, nqb, pairs);
            if (un.ok) prologue(un, n + 1);
            const int b = n & 1;
            const int h = u.kvh * a.group + u.pair * 2 + hl, tok = u.tok0 + tl;
            const bool row_ok = tl < u.rows_valid && u.pair * 2 + hl < a.group;
            mbar_wait(dq_full + 8 * b, (n >> 1) & 1, abort_flag, a.status);
            tc_fence_after();
            __nv_bfloat16* dqrow = a.dq + ((size_t)tok * a.hq + h) * D;
#pragma unroll
            for (int c = 0; c < D / 32; ++c) {
                uint32_t v[32];
                tmem_ld32(t_lane + kColDQ + b * 128 + c * 32, v);
                tmem_wait_ld();
                if (row_ok) {
#pragma unroll
                    for (int e = 0; e < 32; e += 8) {
                        uint4 w;
                        w.x = pack_bf16x2(__uint_as_float(v[e + 0]), __uint_as_float(v[e + 1]));
                        w.y = pack_bf16x2(__uint_as_float(v[e + 2]), __uint_as_float(v[e + 3]));
                        w.z = pack_bf16x2(__uint_as_float(v[e + 4]), __uint_as_float(v[e + 5]));
                        w.w = pack_bf16x2(__uint_as_float(v[e + 6]), __uint_as_float(v[e + 7]));
                        *reinterpret_cast<uint4*>(dqrow + c * 32 + e) = w;
                    }
                }
            }
            tc_fence_before();
            named_sync(1, 128);
            if ((tid & 127) == 0) mbar_arrive(dq_free + 8 * b);
            u = un;
        }
    }
    tc_fence_before();
    __syncthreads();
    if (warp == 0) tmem_dealloc(tmem, 512);
}

// ---- the inverse route -----------------------------------------------------------------------------------------

// The readers of KV slot gp are the list entries of the same sequence that name its block (an entry is its query slot
// times max_degree plus its place in the list).  Transposing the lists is a counting sort by KV slot, linear in the
// number of list entries: count (one thread per entry), scan (inverse_units_kernel), fill in whatever order the
// atomics give, then sort every slot's readers ascending -- the order in which the dK/dV kernel adds is thereby the
// same on every run.
// The slot of an entry's block p lies as many slots in front of its query slot g as p blocks in front of j, because the
// planner numbers the query blocks of a sequence one after the other.  Nothing else needs that (the forward takes a route
// with its slots in any order, and a shard's, whose first blocks have no slots), so it is checked for every entry: the slot
// exists, and it is that block of the same sequence.  One entry for which it is not so and the route has no backward.
__device__ __forceinline__ bool names_slot(int kv, int nqb, int p, int seq, int batch, const int32_t* block, const int32_t* seqs) {
    return kv >= 0 && kv < nqb && block[kv] == p && seq >= 0 && seq < batch && (batch == 1 || seqs[kv] == seq);
}
// 1: an entry and the slot kv it names; 0: no entry; -1: an entry that names no slot (looked at if kCheck).
template <bool kCheck>
__device__ __forceinline__ int inverse_entry(const BwdArgs& a, int nqb, int f, int& kv) {
    const int g = f / a.max_degree, e = f - g * a.max_degree;
    const int cnt = min(max(a.kv_count[g], 1), a.max_degree);
    if (e >= cnt) return 0;
    const int j = a.qb_block[g], p = list_entry(a.kv_idx + (size_t)g * a.max_degree, e, cnt, j);
    kv = g - j + p;
    return !kCheck || names_slot(kv, nqb, p, slot_seq(a, g), a.batch, a.qb_block, a.qb_seq) ? 1 : -1;
}

// kFill = false: count[kv] += 1 (count, and the word behind it, are zero on entry).  kFill = true: count[kv] is counted down again and hands out
// the places behind start[kv].
template <bool kFill>
__global__ void __launch_bounds__(256) inverse_route_kernel(const BwdArgs a) {
    const int nqb = min(*a.num_qblocks, a.capacity);
    const int total = nqb * a.max_degree;
    if (kFill && a.inv.scalars[0] == 0) return;      // (some entry names no slot)
    for (int f = blockIdx.x * 256 + threadIdx.x; f < total; f += gridDim.x * 256) {
        int kv;
        const int is = inverse_entry<!kFill>(a, nqb, f, kv);
        if (!kFill && is < 0) a.inv.count[a.inv.cap] = 1;
        if (is <= 0) continue;
        if (!kFill) atomicAdd(a.inv.count + kv, 1);
        else a.inv.readers[a.inv.start[kv] + atomicSub(a.inv.count + kv, 1) - 1] = f;
    }
}

// Ascending sort of c <= 32 values, one per lane.
__device__ __forceinline__ int rank_in_warp(int v, int c, int lane) {
    int rank = 0;
    for (int j = 0; j < c; ++j) {
        const int vj = __shfl_sync(0xffffffffu, v, j);
        rank += (vj < v) || (vj == v && j < lane);
    }
    return rank;
}

// One CTA per KV slot: its readers ascending.  Up to 32 by ranking inside a warp; more by a bitonic network whose
// comparators all point the same way, so that a length that is no power of two needs no padding (elements past the end
// count as +infinity and never move); in shared memory when they fit, else in place.
constexpr int kSortSmem = 4096;
__global__ void __launch_bounds__(256) inverse_sort_kernel(const BwdArgs a) {
    __shared__ int32_t s_v[kSortSmem];
    const int gp = blockIdx.x, tid = threadIdx.x, lane = tid & 31;
    if (gp >= min(*a.num_qblocks, a.capacity) || a.inv.scalars[0] == 0) return;
    const int s0 = a.inv.start[gp], c = a.inv.start[gp + 1] - s0;
    int32_t* r = a.inv.readers + s0;
    if (c <= 1) return;
    if (c <= 32) {
        if (tid >= 32) return;
        const int v = lane < c ? r[lane] : 0x7fffffff;
        const int rank = rank_in_warp(v, c, lane);
        if (lane < c) r[rank] = v;
        return;
    }
    int32_t* v = c <= kSortSmem ? s_v : r;
    if (c <= kSortSmem) {
        for (int i = tid; i < c; i += 256) s_v[i] = r[i];
    }
    __syncthreads();
    for (int k = 2; (k >> 1) < c; k <<= 1) {
        for (int j = k >> 1; j > 0; j >>= 1) {
            for (int i = tid; i < c; i += 256) {
                const int l = (j == (k >> 1)) ? (i ^ (k - 1)) : (i ^ j);   // first step of a merge: mirrored partner
                if (l > i && l < c) {
                    const int x = v[i], y = v[l];
                    if (x > y) { v[i] = y; v[l] = x; }
                }
            }
            __syncthreads();
        }
    }
    if (c <= kSortSmem) {
        for (int i = tid; i < c; i += 256) r[i] = s_v[i];
    }
}

// Readers to a run: two more than what an SM gets on average, at most 16 (a unit's K, V and sums are moved once for them), and
// never so few that the slots with more than one run need more than `max_parts` partial-sum slots between them (such a slot
// has fewer than 2 * count / chunk runs).  With 16 everywhere the readers of block 0 were one unit of 16 steps, 1.4 us each,
// while most SMs had less.  A backward in us with runs of 2 / 4 / 6 / 8 / 12 / 16 readers: 1000 tokens, 2 query heads, d = 64 (0.5
// readers an SM) 20.0 / 22.6 / 24.6 / 27.1 / 31.9 / 37.3; 8 heads, d = 128 (2.1) 28.3 / 25.0 / 26.1 / 28.0 / 32.7 / 38.1; 4096 tokens,
// 2 heads (3.0) 35.1 / 30.5 / 29.6 / 29.6 / 33.8 / 38.4; 2000 tokens, 16 heads (10) 75 / 55 / 38.3 / 37.6 / 37.3 / 41.8; 4096
// tokens, 8 heads (12) 88 / 66 / 51.8 / 41.9 / 41.4 / 43.8; from 15 readers an SM on 10, 12 and 16 cost the same.
__device__ __forceinline__ int run_length(const BwdArgs& a, int readers_total) {
    const int even = (int)min((long long)readers_total * a.hkv / a.sms + kLeastChunk, (long long)kMostChunk);
    return max(even, (2 * readers_total + a.inv.max_parts - 1) / a.inv.max_parts);
}

// One CTA: offsets of the reader lists, the run length, and the units of the dK/dV kernel.  inverse_route_kernel has
// counted the readers in the workspace and will fill them in.
__global__ void __launch_bounds__(1024, 1) inverse_units_kernel(const BwdArgs a) {
    __shared__ unsigned long long s_warp[32];
    __shared__ int32_t s_bin[1024];
    const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
    const int nqb = min(*a.num_qblocks, a.capacity);
    const InvPlan& v = a.inv;
    int32_t *start = v.start, *unit0 = v.unit0;
    // inclusive scan of x over the CTA
    auto scan = [&](unsigned long long x, unsigned long long& total) {
#pragma unroll
        for (int off = 1; off < 32; off <<= 1) {
            const unsigned long long up = __shfl_up_sync(0xffffffffu, x, off);
            if (lane >= off) x += up;
        }
        if (lane == 31) s_warp[warp] = x;
        __syncthreads();
        unsigned long long w = s_warp[lane];
#pragma unroll
        for (int off = 1; off < 32; off <<= 1) {
            const unsigned long long up = __shfl_up_sync(0xffffffffu, w, off);
            if (lane >= off) w += up;
        }
        total = __shfl_sync(0xffffffffu, w, 31);
        const unsigned long long before = __shfl_sync(0xffffffffu, w, (warp - 1) & 31);
        __syncthreads();
        return x + (warp > 0 ? before : 0ull);
    };
    auto count_of = [&](int g) { return __ldcg(v.count + g); };   // (written by atomics: read where they were performed)
    s_bin[tid] = 0;
    for (int i = tid; i < a.hkv; i += 1024) v.tickets[i] = 0;
    // pass 1: where each slot's readers start; the total decides the run length
    int readers_total = 0;
    for (int b0 = 0; b0 < nqb; b0 += 1024) {
        const int g = b0 + tid;
        const int c = g < nqb ? count_of(g) : 0;
        unsigned long long total;
        const int incl = (int)scan((unsigned long long)c, total);
        if (g < nqb) start[g] = readers_total + incl - c;
        readers_total += (int)total;
    }
    if (tid == 0) start[nqb] = readers_total;
    const int chunk = run_length(a, readers_total);
    // pass 2: runs per slot -> unit numbers, partial-sum slots and places in `multi`: one scan, 21 bits each
    int units = 0, parts = 0, multis = 0;
    for (int b0 = 0; b0 < nqb; b0 += 1024) {
        const int g = b0 + tid;
        const int c = g < nqb ? count_of(g) : 0;
        const int runs = (c + chunk - 1) / chunk, split = runs > 1 ? runs : 0;
        const unsigned long long x = (unsigned long long)runs | (unsigned long long)split << 21 | (unsigned long long)(runs > 1) << 42;
        unsigned long long total;
        const unsigned long long excl = scan(x, total) - x;
        const int q0 = parts + (int)(excl >> 21 & 0x1fffff), m0 = multis + (int)(excl >> 42);
        if (g < nqb) {
            unit0[g] = units + (int)(excl & 0x1fffff);
            if (runs > 1) v.multi[m0] = g;
            v.chunks[g] = runs;
            v.part0[g] = runs > 1 ? q0 : -1;
        }
        units += (int)(total & 0x1fffff), parts += (int)(total >> 21 & 0x1fffff), multis += (int)(total >> 42);
    }
    const bool sound = __ldcg(v.count + v.cap) == 0, fits = sound && units <= v.max_units && parts <= v.max_parts;
    if (tid == 0) {
        unit0[nqb] = units;
        if (!fits && a.status) atomicOr(a.status, sound ? BF1_DEV_CAPACITY : BF1_DEV_BAD_ROUTE);
        v.scalars[0] = fits ? units : 0;
        v.scalars[1] = readers_total;
        v.scalars[2] = chunk;
        v.scalars[3] = parts;
        v.scalars[4] = fits ? multis : 0;
    }
    __syncthreads();
    // the units, a thread each: the slot by binary search
    auto unit_of = [&](int un, int& g, int& begin, int& end) {
        int lo = 0, hi = nqb;     // unit0[lo] <= un < unit0[hi]  (a slot without readers has no unit)
        while (hi - lo > 1) {
            const int mid = (lo + hi) >> 1;
            if (unit0[mid] <= un) lo = mid; else hi = mid;
        }
        g = lo;
        begin = start[g] + (un - unit0[g]) * chunk;
        end = min(begin + chunk, start[g + 1]);
    };
    auto bin_of = [](int len) { return 1023 - min(len, 1023); };
    if (fits) {
        for (int un = tid; un < units; un += 1024) {
            int g, begin, end;
            unit_of(un, g, begin, end);
            atomicAdd(&s_bin[bin_of(end - begin)], 1);
        }
    }
    __syncthreads();
    // units by descending length (a counting sort; which of two equally long units comes first does not matter: the
    // order only decides which CTA works on which unit)
    {
        const int c = s_bin[tid];
        unsigned long long total;
        const int incl = (int)scan((unsigned long long)c, total);
        s_bin[tid] = incl - c;       // where the units of this length start
    }
    __syncthreads();
    if (fits) {
        for (int un = tid; un < units; un += 1024) {
            int g, begin, end;
            unit_of(un, g, begin, end);
            const int at = atomicAdd(&s_bin[bin_of(end - begin)], 1), seq = slot_seq(a, g);
            const bool split = unit0[g + 1] - unit0[g] > 1;
            const int seq0 = a.cu_seqlens[seq];
            v.units[2 * at] = make_int4(g, begin, end - begin, split ? v.part0[g] + un - unit0[g] : -1);
            v.units[2 * at + 1] = make_int4(seq0, a.qb_block[g], a.cu_seqlens[seq + 1] - seq0, 0);
        }
    }
}

// The whole inverse route by one CTA of 1024 threads, in inverse_words() words of shared memory: the chain that
// bwd_prep_kernel hides behind the pass over dO and O, and at 4K tokens the longer of the two, so what counts is the number
// of dependent steps.  Every load whose address is known goes out first (nothing waits for the number of query blocks);
// the readers are counted in total beside the counts of the slots, so that one prefix sum gives everything; all full runs
// of a slot have one length, so that a thread counts and places its slot's units with two atomics each; and the units'
// places are found while the readers are filled in.
// A slot with many readers (block 0) has a warp go through all entries in order instead of every reader counting the smaller
// ones, which grows with their square: a backward of 261,000 tokens that read block 0 and their own (4079 readers) takes 236
// us (2 query heads, d = 64), 592 with the counting alone.  The line lies where the two cost the same at 12,000 entries, the
// most that fit: 256^2 / 32 steps of the CTA against 12,000 / 32 of one warp, about six times as long each.
constexpr int kManyReaders = 256;
constexpr int kInvInts = 24576;     // words of shared memory, at most
__host__ __device__ inline int64_t inverse_words(int64_t cap, int64_t max_degree) { return 2 * cap + 1 + 2 * cap * max_degree; }

__device__ __forceinline__ void inverse_route_in_cta(const BwdArgs& a, int32_t* smem, int status) {
    __shared__ int32_t s_bin[1024];     // units of a length, then where they start: longest first
    __shared__ unsigned long long s_warp[32];
    __shared__ int32_t s_total, s_bad, s_nmany, s_many[kInvInts / 2 / kManyReaders];   // (entries take half of the words at most)
    const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
    const InvPlan& v = a.inv;
    const int entries = a.capacity * a.max_degree;
    int32_t* count = smem;
    int32_t* start = count + a.capacity;            // [nqb + 1] first reader of a slot
    int32_t* kv_of = start + a.capacity + 1;        // per entry: the KV slot it names, or -1
    int32_t* readers = kv_of + entries;
    constexpr int kAtOnce = 4;      // entries a thread reads together: each is three loads
    int c[kAtOnce], j[kAtOnce], p[kAtOnce];
    auto load = [&](int f0) {
#pragma unroll
        for (int i = 0; i < kAtOnce; ++i) {
            const int f = min(f0 + i * 1024, entries - 1), g = f / a.max_degree;
            c[i] = a.kv_count[g], j[i] = a.qb_block[g], p[i] = a.kv_idx[f];
        }
    };
    load(tid);
    const int my_slot = min(tid, a.capacity - 1);
    const int my_j = a.qb_block[my_slot], my_seq = slot_seq(a, my_slot);
    // the slots' blocks and sequences, for names_slot(): in the place of the readers until those are filled in (with one
    // entry to a list there is none to check but the slot itself)
    int32_t *block = a.max_degree > 1 ? readers : count, *seqs = a.max_degree > 1 ? readers + a.capacity : count;
    const int nqb = min(*a.num_qblocks, a.capacity);
    if (status & BF1_DEV_WAIT_TIMEOUT) return;
    if (a.max_degree > 1) {
#pragma unroll 1
        for (int g = tid; g < a.capacity; g += 1024) {
            block[g] = g == tid ? my_j : a.qb_block[g];
            seqs[g] = g == tid ? my_seq : slot_seq(a, g);
        }
    }
#pragma unroll 1
    for (int g = tid; g < a.capacity; g += 1024) count[g] = 0;
    s_bin[tid] = 0;
    if (tid == 0) s_total = s_bad = s_nmany = 0;
#pragma unroll 1
    for (int i = tid; i < a.hkv; i += 1024) v.tickets[i] = 0;
    __syncthreads();
    // (a slot behind the last one may hold anything)
    int my_seq0 = 0, my_end = 0;
    if (tid < nqb && my_seq >= 0 && my_seq < a.batch) my_seq0 = a.cu_seqlens[my_seq], my_end = a.cu_seqlens[my_seq + 1];
    int mine = 0;
#pragma unroll 1
    for (int f0 = tid; f0 < nqb * a.max_degree; f0 += kAtOnce * 1024) {
        if (f0 != tid) load(f0);
#pragma unroll
        for (int i = 0; i < kAtOnce; ++i) {
            const int f = f0 + i * 1024, g = f / a.max_degree, e = f - g * a.max_degree;
            const int cnt = min(max(c[i], 1), a.max_degree);
            if (f >= nqb * a.max_degree) continue;
            int kv = -1;
            if (e < cnt) {
                const int b = safe_entry(p[i], e, cnt, j[i]);
                kv = g - j[i] + b;
                if (a.max_degree == 1 || names_slot(kv, nqb, b, seqs[g], a.batch, block, seqs)) {
                    atomicAdd(count + kv, 1);
                    ++mine;
                } else {
                    s_bad = 1;
                }
            }
            kv_of[f] = kv;
        }
    }
    mine = __reduce_add_sync(0xffffffffu, mine);
    if (lane == 0) atomicAdd(&s_total, mine);
    __syncthreads();
    if (s_bad) {                     // (uniform over the CTA)
        if (tid == 0) {
            if (a.status) atomicOr(a.status, BF1_DEV_BAD_ROUTE);
            v.scalars[0] = v.scalars[4] = 0;
        }
        return;
    }
    const int readers_total = s_total, chunk = run_length(a, readers_total);
    // prefix sums over the slots of the readers, the units, the partial-sum slots and the slots cut into runs, 16 bits each
    // (there are fewer entries than that); the number of units of every length is counted beside them
    auto bin_of = [](int len) { return 1023 - min(len, 1023); };
    unsigned long long carry = 0;
#pragma unroll 1
    for (int b0 = 0; b0 < nqb; b0 += 1024) {
        const int g = b0 + tid, n = g < nqb ? count[g] : 0;
        // a slot's units: n / chunk of `chunk` readers, and one with the rest
        const int full = n < chunk ? 0 : n / chunk, rest = n - full * chunk, runs = full + (rest > 0);
        if (full) atomicAdd(s_bin + bin_of(chunk), full);
        if (rest) atomicAdd(s_bin + bin_of(rest), 1);
        const unsigned long long x = (unsigned long long)(n | runs << 16) | (unsigned long long)(runs > 1 ? runs | 1 << 16 : 0) << 32;
        unsigned long long incl = x;
        if (b0 + warp * 32 < nqb) {
#pragma unroll
            for (int off = 1; off < 32; off <<= 1) {
                const unsigned long long up = __shfl_up_sync(0xffffffffu, incl, off);
                if (lane >= off) incl += up;
            }
        }
        if (lane == 31) s_warp[warp] = incl;
        __syncthreads();
        unsigned long long w = s_warp[lane];
#pragma unroll
        for (int off = 1; off < 32; off <<= 1) {
            const unsigned long long up = __shfl_up_sync(0xffffffffu, w, off);
            if (lane >= off) w += up;
        }
        const unsigned long long before = __shfl_sync(0xffffffffu, w, (warp - 1) & 31);
        const unsigned long long at = carry + incl - x + (warp > 0 ? before : 0ull);
        carry += __shfl_sync(0xffffffffu, w, 31);
        if (g < nqb) {
            const int part = (int)(at >> 32 & 0xffff);
            start[g] = (int)(at & 0xffff);
            v.chunks[g] = runs;
            v.part0[g] = runs > 1 ? part : -1;
            if (runs > 1) v.multi[at >> 48] = g;
            if (n > kManyReaders) s_many[atomicAdd(&s_nmany, 1)] = g;
        }
        __syncthreads();
    }
    const int units = (int)(carry >> 16 & 0xffff), parts = (int)(carry >> 32 & 0xffff);
    const bool fits = units > 0 && units <= v.max_units && parts <= v.max_parts;
    if (tid == 0) {
        start[nqb] = readers_total;
        if (units > 0 && !fits && a.status) atomicOr(a.status, BF1_DEV_CAPACITY);
        v.scalars[0] = fits ? units : 0;
        v.scalars[1] = readers_total;
        v.scalars[2] = chunk;
        v.scalars[3] = parts;
        v.scalars[4] = fits ? (int)(carry >> 48) : 0;
    }
    if (warp == 0) {        // (no unit is longer than `chunk`)
        int first = 0;
#pragma unroll 1
        for (int b = bin_of(chunk) & ~31; b < 1024; b += 32) {
            const int x = s_bin[b + lane];
            int incl = x;
#pragma unroll
            for (int off = 1; off < 32; off <<= 1) {
                const int up = __shfl_up_sync(0xffffffffu, incl, off);
                if (lane >= off) incl += up;
            }
            s_bin[b + lane] = first + incl - x;
            first += __shfl_sync(0xffffffffu, incl, 31);
        }
    } else {
#pragma unroll 1
        for (int f = tid - 32; f < nqb * a.max_degree; f += 1024 - 32) {
            const int kv = kv_of[f];
            if (kv >= 0) readers[start[kv] + atomicSub(count + kv, 1) - 1] = f;
        }
    }
    __syncthreads();
    if (fits) {
#pragma unroll 1
        for (int g = tid; g < nqb; g += 1024) {
            int seq0 = my_seq0, seqlen = my_end - my_seq0, jg = my_j;
            if (g != tid) {
                const int seq = slot_seq(a, g);
                seq0 = a.cu_seqlens[seq], seqlen = a.cu_seqlens[seq + 1] - seq0, jg = a.qb_block[g];
            }
            const int s0 = start[g], n = start[g + 1] - s0, full = n < chunk ? 0 : n / chunk, rest = n - full * chunk;
            const int part = full + (rest > 0) > 1 ? v.part0[g] : -1;
            const int at_full = full ? atomicAdd(s_bin + bin_of(chunk), full) : 0;
            const int at_rest = rest ? atomicAdd(s_bin + bin_of(rest), 1) : 0;
#pragma unroll 1
            for (int i = 0; i < full + (rest > 0); ++i) {
                const int at = i < full ? at_full + i : at_rest;
                v.units[2 * at] = make_int4(g, s0 + i * chunk, i < full ? chunk : rest, part >= 0 ? part + i : -1);
                v.units[2 * at + 1] = make_int4(seq0, jg, seqlen, 0);
            }
        }
    }
    // an entry's place among its slot's readers is the number of smaller ones (they are distinct)
#pragma unroll 1
    for (int b = warp; b < s_nmany; b += 32) {
        const int g = s_many[b];
        int at = start[g];
#pragma unroll 4
        for (int f0 = g * a.max_degree; f0 < nqb * a.max_degree; f0 += 32) {
            const bool is = f0 + lane < nqb * a.max_degree && kv_of[f0 + lane] == g;
            const unsigned all = __ballot_sync(0xffffffffu, is);
            if (is) v.readers[at + __popc(all & ((1u << lane) - 1))] = f0 + lane;
            at += __popc(all);
        }
    }
#pragma unroll 1
    for (int i = tid; i < readers_total; i += 1024) {
        const int f = readers[i], kv = kv_of[f], s0 = start[kv], s1 = start[kv + 1];
        if (s1 - s0 > kManyReaders) continue;
        int rank = 0;
#pragma unroll 4
        for (int k = s0; k < s1; ++k) rank += readers[k] < f;
        v.readers[s0 + rank] = f;
    }
}

// D_i = <dO_i, O_i> of every row, and (kInverse) in the first CTA the whole inverse route: a chain of a few
// microseconds on one SM that is hidden behind the pass over dO and O on the others.  kInverse is chosen while the
// entries fit shared memory beside the counters (kInvInts words): up to 945 query blocks of one sequence with
// the paper's route, 60,480 tokens; beyond, several launches share the work.  Where the two meet they cost the same: a backward of
// 60,480 tokens 197.7 us, of 60,500 196.9 (2 query heads, d = 64).
// Measured: 8 us at 4K tokens (16 query heads, d = 128), of which the pass over dO and O alone takes 5.1 and the inverse
// route alone 7.8 (7.5 without looking at the slot that an entry names; looking at four entries' slots without a branch, all
// at once: 9.7), and 48 us at 32K, where the inverse route alone takes 22.  (With more dependent steps in the
// inverse route, a scan for each of its sums, a search for every unit and everything behind the number of query blocks: 8.2
// and 28 us of its own, a forward and backward of 4K tokens 97.6 us, 95.4 as it is; 16K tokens in 12 sequences 163.7 and
// 162.8.  As launches of their own: 12 and 28 us, with D_i in the dQ kernel.)
template <int D, bool kInverse>
__global__ void __launch_bounds__(1024, 1) bwd_prep_kernel(const BwdArgs a) {
    extern __shared__ int32_t s_inv[];
    pdl_wait();
    const int status = a.status ? *a.status : 0;
    int cta = blockIdx.x, ctas = gridDim.x;
    if (kInverse) {
        if (cta == 0) {
            inverse_route_in_cta(a, s_inv, status);
            return;
        }
        --cta, --ctas;
    }
    if (status & BF1_DEV_WAIT_TIMEOUT) return;
    // a warp takes 16 tokens of one head; a row is read by D / 8 lanes, 16 bytes each
    constexpr int kLanes = D / 8, kRowsAtOnce = 32 / kLanes, kTokens = 16;
    const int lane = threadIdx.x & 31, sub = lane % kLanes, r0 = lane / kLanes;
    const int items = ((a.total_tokens + kTokens - 1) / kTokens) * a.hq;
    for (int item = cta * 32 + (threadIdx.x >> 5); item < items; item += ctas * 32) {
        const int h = item % a.hq, t0 = (item / a.hq) * kTokens;
        float mine = 0.f;
#pragma unroll
        for (int it0 = 0; it0 < kTokens / kRowsAtOnce; it0 += 4) {   // 4 rows' loads in flight at once
            uint4 x[4], g[4];
#pragma unroll
            for (int i = 0; i < 4; ++i) {
                const int tok = min(t0 + (it0 + i) * kRowsAtOnce + r0, a.total_tokens - 1);
                const size_t at = ((size_t)tok * a.hq + h) * D + sub * 8;
                x[i] = *reinterpret_cast<const uint4*>(a.o + at);
                g[i] = *reinterpret_cast<const uint4*>(a.d_o + at);
            }
#pragma unroll
            for (int i = 0; i < 4; ++i) {
                const uint32_t xw[4] = {x[i].x, x[i].y, x[i].z, x[i].w}, gw[4] = {g[i].x, g[i].y, g[i].z, g[i].w};
                float sum = 0.f;
#pragma unroll
                for (int e = 0; e < 4; ++e) {
                    sum = fmaf(__uint_as_float(xw[e] << 16), __uint_as_float(gw[e] << 16), sum);
                    sum = fmaf(__uint_as_float(xw[e] & 0xffff0000u), __uint_as_float(gw[e] & 0xffff0000u), sum);
                }
#pragma unroll
                for (int off = kLanes / 2; off > 0; off >>= 1) sum += __shfl_xor_sync(0xffffffffu, sum, off);
                if (sub == it0 + i) mine = sum;
            }
        }
        const int tok = t0 + sub * kRowsAtOnce + r0;
        if (sub < kTokens / kRowsAtOnce && tok < a.total_tokens) a.delta[(size_t)h * a.total_tokens + tok] = mine;
    }
    const int nqb = min(*a.num_qblocks, a.capacity);
    for (int r = (ctas - 1 - cta) * 1024 + threadIdx.x; r < nqb; r += ctas * 1024) rank_query_block(a, r, nqb);
}

// ---- dK, dV ----------------------------------------------------------------------------------------------------
//
// One persistent CTA of 16 warps per SM.  A unit is (KV block, KV head, run of the block's readers); units are
// handed out through a counter, longest first (KV head by KV head, or all heads together: BwdArgs::interleave).  K and V
// of a unit stay in shared memory (two buffers: the next unit's arrive early), Q and dO of every step (a reader and a
// pair of its heads) travel through a ring of two stages:
//     warp 0    takes the units and describes them to the other roles; copies K of every unit and Q of every step;
//               brings every step's LSE into shared memory
//     warp 1    copies V and dO; brings D_i into shared memory
//     warp 2    issues S = Q K^T and dP = dO V^T of every step into one of two S/dP buffers in tensor memory
//     warp 3    issues dV^T += dO^T P and dK^T += Q^T dS of every step; the sums stay in one of two accumulator
//               buffers in tensor memory across all steps of the unit.  It also starts the copy of every dS tile to
//               the workspace, as it lies in shared memory: its own MMAs read the tile at the same time
//     warps 4-11   the arithmetic on S and dP (two threads per tile row), P and dS as bf16 tiles to shared memory
//     warps 12-15  the finished sums of the unit before, from tensor memory to global memory
// A step moves 304 KiB through shared memory (192 of MMA operands, 64 in, P and dS written, dS read again): 2432 cycles
// at 128 bytes per cycle, which is the bound.
// Units described through shared memory, LSE and D_i brought there a step ahead and dynamic hand-out: 55 -> 46 us at 4K
// tokens, 96 -> 76 us for 16K tokens in 12 sequences (four heads per KV head), 544 -> 483 us at 32K.  (Every role read the
// unit and the rows' LSE from global memory itself before: 940 of 2900 cycles of a step in the arithmetic warps; and
// the static deal left the busiest CTA 23 %, 35 % and 9 % above the mean.)
constexpr int kDkvThreads = 512;

// What warp 0 tells the other roles about a unit.
struct DkvUnit {
    int steps;                      // 0: no more units
    int kvh, part, gp, p, seq0, seqlen, r_begin;
    int first[32];                  // its first 32 readers (list entries)
};
struct DkvStep {
    int entry, diag;                // the reader, and whether it is the unit's own block
};

template <int D>
struct DkvSmem {
    static constexpr int kQBytes = 128 * D * 2;      // Q / dO tile [D / 64 chunks][128 rows][128 B]
    static constexpr int kKVBytes = 64 * D * 2;      // K / V tile  [D / 64 chunks][64 rows][128 B]
    static constexpr int kQ = 0;                     // [2]
    static constexpr int kDO = kQ + 2 * kQBytes;     // [2]
    static constexpr int kK = kDO + 2 * kQBytes;     // [2]
    static constexpr int kV = kK + 2 * kKVBytes;     // [2]
    static constexpr int kP = kV + 2 * kKVBytes;     // P  [128 q rows][64 kv] bf16, 128-byte rows, swizzled
    static constexpr int kDS = kP + 16384;           // dS likewise
    static constexpr int kRow = kDS + 16384;         // LSE (log2 domain) [2][128], D_i [2][128]
    static constexpr int kUnit = kRow + 4 * 512;     // DkvUnit [2]
    static constexpr int kStep = kUnit + 2 * (int)sizeof(DkvUnit);   // DkvStep [2]
    static constexpr int kBar = kStep + 2 * (int)sizeof(DkvStep);
    static constexpr int kUsed = kBar + 8 * 25 + 8;
    // at least this much is requested so that a second CTA never fits an SM: each allocates all of tensor memory
    static constexpr int kTotal = kUsed > 120 * 1024 ? kUsed : 120 * 1024;
};
static_assert(DkvSmem<128>::kTotal <= 227 * 1024, "shared memory of an SM");

template <int D>
__global__ void __launch_bounds__(kDkvThreads, 1) bwd_dkv_kernel(const __grid_constant__ CUtensorMap tm_q,
                                                              const __grid_constant__ CUtensorMap tm_k,
                                                              const __grid_constant__ CUtensorMap tm_v,
                                                              const __grid_constant__ CUtensorMap tm_do,
                                                              const BwdArgs a) {
    using L = DkvSmem<D>;
    extern __shared__ __align__(1024) uint8_t smem[];
    uint32_t& s_tmem = *reinterpret_cast<uint32_t*>(smem + L::kBar + 8 * 25);
    int& s_abort = *reinterpret_cast<int*>(smem + L::kBar + 8 * 25 + 4);
    volatile DkvUnit* s_unit = reinterpret_cast<volatile DkvUnit*>(smem + L::kUnit);
    volatile DkvStep* s_step = reinterpret_cast<volatile DkvStep*>(smem + L::kStep);
    volatile float* s_lse = reinterpret_cast<volatile float*>(smem + L::kRow);
    volatile float* s_delta = s_lse + 256;
    const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31;
    const int pairs = a.group == 4 ? 2 : 1;

    const uint32_t base = smem_u32(smem);
    const uint32_t bars = base + L::kBar;
    const uint32_t kv_full = bars;                 // [2] K and V of a unit landed (both copy warps announce bytes)
    const uint32_t kv_free = kv_full + 16;         // [2] the unit's S / dP MMAs are done
    const uint32_t q_full = kv_free + 16;          // [2] Q of a step landed; its LSE and DkvStep are written
    const uint32_t do_full = q_full + 16;          // [2] dO of a step landed; its D_i are written
    const uint32_t q_free = do_full + 16;          // [2] the step's dK^T MMAs are done (they come first: S of the step after
    const uint32_t do_free = q_free + 16;          //     next can then start while its dO is still travelling); [2] its dV^T MMAs
    const uint32_t sdp_full = do_free + 16;        // [2] S and dP of a step computed
    const uint32_t pds_ready = sdp_full + 16;      // [2] P and dS of a step are in shared memory (8 warps); S / dP have been read
    const uint32_t acc_full = pds_ready + 16;      // [2] the unit's sums are complete
    const uint32_t acc_free = acc_full + 16;       // [2] ... and have been read out of tensor memory
    const uint32_t unit_full = acc_free + 16;      // [2] the unit is described
    const uint32_t unit_free = unit_full + 16;     // [2] ... and every other warp has read the description
    const uint32_t pds_free = unit_free + 16;      // [1] the MMAs that read P and dS, and the copy of dS, are done
    if (tid == 0) {
        s_abort = (base & 1023u) ? 1 : 0;
        for (int b = 0; b < 2; ++b) {
            mbar_init(kv_full + 8 * b, 2);
            mbar_init(kv_free + 8 * b, 1);
            mbar_init(q_full + 8 * b, 2);
            mbar_init(do_full + 8 * b, 2);
            mbar_init(q_free + 8 * b, 1);
            mbar_init(do_free + 8 * b, 1);
            mbar_init(sdp_full + 8 * b, 1);
            mbar_init(pds_ready + 8 * b, 8);
            mbar_init(acc_full + 8 * b, 1);
            mbar_init(acc_free + 8 * b, 1);
            mbar_init(unit_full + 8 * b, 1);
            mbar_init(unit_free + 8 * b, 15);
        }
        mbar_init(pds_free, 2);
        fence_mbar_init();
    }
    __syncwarp();
    if (warp == 0) {
        tmem_alloc(smem_u32(&s_tmem), 512);
        tmem_relinquish();
    }
    if (a.group == 1) {   // one head per KV head: rows 64..127 of the Q / dO buffers are never written by a copy
        clear_idle_rows<D>(base + L::kQ, base + L::kDO, tid, kDkvThreads);
        clear_idle_rows<D>(base + L::kQ + L::kQBytes, base + L::kDO + L::kQBytes, tid, kDkvThreads);
    }
    // warp 0's next unit, taken and read a few steps before it is needed: ticket, then description, then readers
    int n_units = 0;
    int next_i = blockIdx.x, next_kvh = 0, next_f = 0;
    int4 next_a = make_int4(0, 0, 0, -1), next_b = make_int4(0, 0, 0, 0);
    auto take = [&]() { if (lane == 0) next_i = (int)gridDim.x + atomicAdd(a.inv.tickets + a.head0, 1); };
    auto look_up = [&]() {          // (interleaved heads: no need of the number of units)
        int ui;
        if (a.interleave) {
            ui = next_i / a.nheads;
            next_kvh = next_i - ui * a.nheads;
        } else {
            next_kvh = next_i / max(n_units, 1);
            ui = next_i - next_kvh * n_units;
        }
        next_kvh += a.head0;
        ui = min(ui, a.inv.max_units - 1);
        next_a = a.inv.units[2 * ui];
        next_b = a.inv.units[2 * ui + 1];
    };
    auto describe = [&]() {
        next_i = __shfl_sync(0xffffffffu, next_i, 0);
        next_a.z = 0;
        if (next_i < n_units * a.nheads) look_up();
    };
    auto read_readers = [&]() { next_f = lane < next_a.z ? a.inv.readers[next_a.y + lane] : 0; };
    pdl_wait();
    // The first unit is read beside the status word (interleaved heads: where it stands does not depend on the number of
    // units).  After an earlier launch gave up it may be anything and is not used: its index is in range all the same.
    // (With the dQ kernel's first units likewise: forward and backward of 4K tokens 96.3 us behind the status word, 95.7 so.)
    if (warp == 0) {
        n_units = a.inv.scalars[0];
        if (a.interleave) look_up();
    }
    if (tid == 0 && a.status) {
        if (s_abort) atomicOr(a.status, BF1_DEV_WAIT_TIMEOUT);
        if (*a.status & BF1_DEV_WAIT_TIMEOUT) s_abort = 1;
    }
    tc_fence_before();
    __syncthreads();
    tc_fence_after();
    const uint32_t tmem = s_tmem;
    volatile int* abort_flag = &s_abort;
    if (s_abort) {   // (uniform over the CTA)
        __syncthreads();
        if (warp == 0) tmem_dealloc(tmem, 512);
        return;
    }
    // tensor memory: S | dP of buffer b at columns 128 b; dV^T | dK^T (64 columns each: head dimension on the lanes,
    // the block's 64 key rows along the columns) of buffer b at 256 + 128 b
    constexpr uint32_t kColDP = 64, kColAcc = 256, kColDKt = 64;
    const uint32_t q_tx = a.group > 1 ? L::kQBytes : L::kQBytes / 2;   // one head per KV head: half a tile per copy set
    const uint32_t sP = base + L::kP, sDS = base + L::kDS;
    // the description of unit n; a warp that is done with it says so
    auto wait_unit = [&](int n) -> volatile DkvUnit& {
        mbar_wait(unit_full + 8 * (n & 1), (n >> 1) & 1, abort_flag, a.status);
        return s_unit[n & 1];
    };
    auto free_unit = [&](int n) {
        __syncwarp();
        if (lane == 0) mbar_arrive(unit_free + 8 * (n & 1));
    };
    auto unit_steps = [&](volatile DkvUnit& u) { return *abort_flag ? 0 : u.steps; };

    if (warp == 0 || warp == 1) {
        // ---- copies (and, in warp 0, the units) ----
        const bool first = warp == 0;
        const uint32_t full = first ? q_full : do_full, free_ = first ? q_free : do_free;
        const float* rows = first ? a.lse : a.delta;
        volatile float* s_row = first ? s_lse : s_delta;
        if (first) {
            if (!a.interleave) look_up();
            if (next_i >= n_units * a.nheads) next_a.z = 0;
            read_readers();
        }
        int s = 0;   // steps so far
        for (int n = 0;; ++n) {
            const int b = n & 1;
            if (first) {
                if (n >= 2) mbar_wait(unit_free + 8 * b, ((n >> 1) - 1) & 1, abort_flag, a.status);
                volatile DkvUnit& d = s_unit[b];
                d.first[lane] = next_f;
                if (lane == 0) {
                    d.steps = next_a.z * pairs;
                    d.kvh = next_kvh;
                    d.part = next_a.w;
                    d.gp = next_a.x;
                    d.p = next_b.y;
                    d.seq0 = next_b.x;
                    d.seqlen = next_b.z;
                    d.r_begin = next_a.y;
                }
                __syncwarp();
                if (lane == 0) mbar_arrive(unit_full + 8 * b);
            }
            volatile DkvUnit& u = wait_unit(n);
            const int steps = unit_steps(u), kvh = u.kvh, gp = u.gp, p = u.p, seq0 = u.seq0, seqlen = u.seqlen, r_begin = u.r_begin;
            int my_f = u.first[lane];
            if (!first) free_unit(n);
            if (steps == 0) break;
            if (n >= 2) mbar_wait(kv_free + 8 * b, ((n >> 1) - 1) & 1, abort_flag, a.status);
            if (elect_one()) {
                mbar_expect_tx(kv_full + 8 * b, L::kKVBytes);
                if (first) tma_load_4d(base + L::kK + b * L::kKVBytes, &tm_k, 0, seq0 + p * kBlock64, kvh, 0, kv_full + 8 * b);
                else tma_load_4d(base + L::kV + b * L::kKVBytes, &tm_v, 0, seq0 + p * kBlock64, kvh, 0, kv_full + 8 * b);
            }
            __syncwarp();
            for (int step = 0; step < steps; ++step, ++s) {
                const int sb = s & 1, idx = step / pairs, pr = step % pairs;
                if (idx >= 32 && (idx & 31) == 0 && pr == 0)        // runs longer than a warp: the next 32 readers
                    my_f = r_begin + idx + lane < r_begin + steps / pairs ? a.inv.readers[r_begin + idx + lane] : 0;
                const int f = __shfl_sync(0xffffffffu, my_f, idx & 31), g = f / a.max_degree;
                const int jq = g - gp + p;                          // slots of a sequence are consecutive
                const int head0 = kvh * a.group + pr * 2, rows_valid = min(kBlock64, seqlen - jq * kBlock64);
                // this step's LSE / D_i, four rows a lane: asked for now, put into shared memory behind the copy
                float v[4];
#pragma unroll
                for (int i = 0; i < 4; ++i) {
                    const int row = i * 32 + lane, hl = row >> 6, tl = row & 63;
                    v[i] = first ? INFINITY : 0.f;                  // rows outside: P = 0
                    if (tl < rows_valid && pr * 2 + hl < a.group)
                        v[i] = rows[(size_t)(head0 + hl) * a.total_tokens + seq0 + jq * kBlock64 + tl];
                }
                if (s >= 2) mbar_wait(free_ + 8 * sb, ((s >> 1) - 1) & 1, abort_flag, a.status);
                if (elect_one()) {
                    mbar_expect_tx(full + 8 * sb, q_tx);
                    if (first) load_q_tile<D>(base + L::kQ + sb * L::kQBytes, &tm_q, seq0 + jq * kBlock64, head0, a.group, full + 8 * sb);
                    else load_q_tile<D>(base + L::kDO + sb * L::kQBytes, &tm_do, seq0 + jq * kBlock64, head0, a.group, full + 8 * sb);
                }
                __syncwarp();
#pragma unroll
                for (int i = 0; i < 4; ++i) s_row[sb * 128 + i * 32 + lane] = first ? v[i] * 1.4426950408889634f : v[i];
                if (first && lane == 0) {
                    s_step[sb].entry = f;
                    s_step[sb].diag = g == gp;
                }
                __syncwarp();
                if (lane == 0) mbar_arrive(full + 8 * sb);
                if (first) {
                    if (step == max(steps - 3, 0)) take();
                    if (step == max(steps - 2, 0)) describe();
                    if (step == steps - 1) read_readers();
                }
            }
        }
    } else if (warp == 2 || warp == 3) {
        // ---- MMAs: warp 2 issues S and dP of every step, warp 3 the two transposed products ----
        constexpr uint32_t kHi = desc_hi_sw128(1024);
        constexpr uint32_t kIdT = idesc_bf16_f32_ab(64, true, true);   // dV^T, dK^T: A and B MN-major
        const size_t tiles = (size_t)a.capacity * a.max_degree;
        int s = 0;
        for (int n = 0;; ++n) {
            volatile DkvUnit& u = wait_unit(n);
            const int steps = unit_steps(u), kvh = u.kvh;
            free_unit(n);
            if (steps == 0) break;
            const int b = n & 1;
            char* ds_head = reinterpret_cast<char*>(a.ds) + (size_t)(kvh - a.head0) * pairs * tiles * kDsTile;
            if (warp == 2) mbar_wait(kv_full + 8 * b, (n >> 1) & 1, abort_flag, a.status);
            else if (n >= 2) mbar_wait(acc_free + 8 * b, ((n >> 1) - 1) & 1, abort_flag, a.status);
            for (int step = 0; step < steps; ++step, ++s) {
                const int sb = s & 1;
                const uint32_t sQ = base + L::kQ + sb * L::kQBytes, sDO = base + L::kDO + sb * L::kQBytes;
                if (warp == 2) {
                    // the buffer's last S and dP must have been read
                    if (s >= 2) mbar_wait(pds_ready + 8 * sb, ((s >> 1) - 1) & 1, abort_flag, a.status);
                    mbar_wait(q_full + 8 * sb, (s >> 1) & 1, abort_flag, a.status);
                    tc_fence_after();
                    if (elect_one()) issue_qk<D>(tmem + sb * 128, sQ, base + L::kK + b * L::kKVBytes);
                    __syncwarp();
                    mbar_wait(do_full + 8 * sb, (s >> 1) & 1, abort_flag, a.status);
                    if (elect_one()) {
                        issue_qk<D>(tmem + sb * 128 + kColDP, sDO, base + L::kV + b * L::kKVBytes);
                        mma_commit(sdp_full + 8 * sb);
                        if (step == steps - 1) mma_commit(kv_free + 8 * b);
                    }
                    __syncwarp();
                } else {
                    mbar_wait(q_full + 8 * sb, (s >> 1) & 1, abort_flag, a.status);   // (DkvStep)
                    const int entry = s_step[sb].entry;
                    mbar_wait(pds_ready + 8 * sb, (s >> 1) & 1, abort_flag, a.status);
                    tc_fence_after();
                    if (elect_one()) {
                        if (a.ds) {
                            bulk_store(ds_head + ((step % pairs) * tiles + entry) * kDsTile, sDS, kDsTile);
                            bulk_commit_group();
                        }
                        // dK^T += Q^T dS, then dV^T += dO^T P: A = Q / dO MN-major (M = d: 64 per 128-byte row, next 64 at
                        // +16 KB; K = q rows, 16 per step = 2048 bytes), B = P / dS MN-major (N = 64 kv per row)
                        const uint32_t t_acc = tmem + kColAcc + b * 128;
#pragma unroll
                        for (int kk = 0; kk < 8; ++kk) {
                            const uint32_t ko = (kk * 2048) >> 4;
                            if (kk == 0) {
                                if (step == 0) mma_ss_lohi<false>(t_acc + kColDKt, desc_lo_sw128(sQ, 16384) + ko, desc_lo_sw128(sDS, 16) + ko, kHi, kIdT);
                                else mma_ss_lohi<true>(t_acc + kColDKt, desc_lo_sw128(sQ, 16384) + ko, desc_lo_sw128(sDS, 16) + ko, kHi, kIdT);
                            } else {
                                mma_ss_lohi<true>(t_acc + kColDKt, desc_lo_sw128(sQ, 16384) + ko, desc_lo_sw128(sDS, 16) + ko, kHi, kIdT);
                            }
                        }
                        mma_commit(q_free + 8 * sb);
#pragma unroll
                        for (int kk = 0; kk < 8; ++kk) {
                            const uint32_t ko = (kk * 2048) >> 4;
                            if (kk == 0) {
                                if (step == 0) mma_ss_lohi<false>(t_acc, desc_lo_sw128(sDO, 16384) + ko, desc_lo_sw128(sP, 16) + ko, kHi, kIdT);
                                else mma_ss_lohi<true>(t_acc, desc_lo_sw128(sDO, 16384) + ko, desc_lo_sw128(sP, 16) + ko, kHi, kIdT);
                            } else {
                                mma_ss_lohi<true>(t_acc, desc_lo_sw128(sDO, 16384) + ko, desc_lo_sw128(sP, 16) + ko, kHi, kIdT);
                            }
                        }
                        mma_commit(do_free + 8 * sb);
                        mma_commit(pds_free);
                        if (step == steps - 1) mma_commit(acc_full + 8 * b);
                        bulk_wait_read0();               // the copy has read the dS tile
                        mbar_arrive(pds_free);
                    }
                    __syncwarp();
                }
            }
        }
    } else if (warp < 12) {
        // ---- arithmetic on S and dP: two threads per tile row (head hl, token tl of the reader), warps 4-7 on key
        // columns 0..31 and warps 8-11 on columns 32..63 ----
        const int half = (warp - 4) >> 2;
        const uint32_t t_lane = tmem + (static_cast<uint32_t>((warp & 3) * 32) << 16);
        const int row = tid & 127, tl = row & 63;
        int s = 0;
        for (int n = 0;; ++n) {
            volatile DkvUnit& u = wait_unit(n);
            const int steps = unit_steps(u);
            free_unit(n);
            if (steps == 0) break;
            for (int step = 0; step < steps; ++step, ++s) {
                const int sb = s & 1;
                mbar_wait(q_full + 8 * sb, (s >> 1) & 1, abort_flag, a.status);
                mbar_wait(do_full + 8 * sb, (s >> 1) & 1, abort_flag, a.status);
                const float lse2 = s_lse[sb * 128 + row], drow = s_delta[sb * 128 + row];
                const bool diag = s_step[sb].diag;
                mbar_wait(sdp_full + 8 * sb, (s >> 1) & 1, abort_flag, a.status);
                tc_fence_after();
                uint32_t pw[16], dw[16];
                p_and_ds(t_lane + sb * 128, t_lane + sb * 128 + kColDP, half, tl, diag, lse2, drow, a.scale, a.scale_log2, pw, dw);
                if (s >= 1) mbar_wait(pds_free, (s - 1) & 1, abort_flag, a.status);   // the MMAs of the step before have read P and dS
                store_row_piece(sP + row * 128, row, half, pw);
                store_row_piece(sDS + row * 128, row, half, dw);
                fence_proxy_async();
                tc_fence_before();
                __syncwarp();
                if (lane == 0) mbar_arrive(pds_ready + 8 * sb);
            }
        }
    } else {
        // ---- the finished dV^T / dK^T of a unit: lane = head-dimension index, 64 key rows along the columns ----
        const uint32_t t_lane = tmem + (static_cast<uint32_t>((warp & 3) * 32) << 16);
        const int row = tid & 127;
        for (int n = 0;; ++n) {
            volatile DkvUnit& u = wait_unit(n);
            const int steps = unit_steps(u), kvh = u.kvh, part = u.part, tok0 = u.seq0 + u.p * kBlock64;
            const int kv_valid = min(kBlock64, u.seqlen - u.p * kBlock64);      // key rows of this block inside the sequence
            free_unit(n);
            if (steps == 0) break;
            const int b = n & 1;
            mbar_wait(acc_full + 8 * b, (n >> 1) & 1, abort_flag, a.status);
            tc_fence_after();
            if (row < D) {   // d = 64: lanes 64..127 hold nothing (warp-uniform)
                float* pk = part >= 0 ? a.partial + (((size_t)part * a.hkv + kvh) * 2) * (kBlock64 * D) + row : nullptr;
#pragma unroll 1
                for (int hh = 0; hh < 4; ++hh) {                     // dV / dK, key rows 0..31 / 32..63
                    const int which = hh >> 1, r0 = (hh & 1) * 32;
                    uint32_t v[32];
                    tmem_ld32(t_lane + kColAcc + b * 128 + which * kColDKt + r0, v);
                    tmem_wait_ld();
                    if (part < 0) {
                        // four lanes hold four neighbouring head-dimension elements of every key row: after exchanging with
                        // lane ^ 1 and lane ^ 2 a lane has all four of one row in four, 8 bytes to store at once
                        __nv_bfloat16* out = (which ? a.dk : a.dv) + ((size_t)tok0 * a.hkv + kvh) * D + (row & ~3);
#pragma unroll
                        for (int c = 0; c < 32; c += 4) {
                            const uint32_t w0 = pack_bf16x2(__uint_as_float(v[c]), __uint_as_float(v[c + 1]));
                            const uint32_t w1 = pack_bf16x2(__uint_as_float(v[c + 2]), __uint_as_float(v[c + 3]));
                            const uint32_t x0 = __shfl_xor_sync(0xffffffffu, w0, 1), x1 = __shfl_xor_sync(0xffffffffu, w1, 1);
                            // even lanes: row c (c + 2), elements lane, lane + 1; odd lanes: row c + 1 (c + 3), lane - 1, lane
                            const uint32_t sel = (lane & 1) ? 0x3276u : 0x5410u;
                            const uint32_t y0 = __byte_perm(w0, x0, sel), y1 = __byte_perm(w1, x1, sel);
                            const uint32_t z = __shfl_xor_sync(0xffffffffu, (lane & 2) ? y0 : y1, 2);
                            const int kvr = r0 + c + (lane & 3);
                            if (kvr < kv_valid)
                                *reinterpret_cast<uint2*>(out + (size_t)kvr * a.hkv * D) = (lane & 2) ? make_uint2(z, y1) : make_uint2(y0, z);
                        }
                    } else {
#pragma unroll
                        for (int c = 0; c < 32; ++c)
                            if (r0 + c < kv_valid) pk[(which ? 0 : kBlock64 * D) + (r0 + c) * D] = __uint_as_float(v[c]);
                    }
                }
            }
            tc_fence_before();
            named_sync(1, 128);
            if ((tid & 127) == 0) mbar_arrive(acc_free + 8 * b);
        }
    }
    tc_fence_before();
    __syncthreads();
    if (warp == 0) tmem_dealloc(tmem, 512);
}

// KV blocks whose readers were cut into several runs: add the runs' partial sums in run order.  A work item is (such a block,
// KV head, kCombineRows of its key rows, dK or dV), one warp each: what is looked up for it is a chain of four loads, so
// several rows share it and are read together.  (A row to an item, and only in the CTAs that had dQ units: 47 us for the 2048
// rows of 1000 tokens cut into runs of 2, under 4 as it is.)
constexpr int kCombineRows = 4;
template <int D>
__device__ __forceinline__ void combine_runs(const BwdArgs& a, int worker, int workers) {
    constexpr int kVec = D / 32, kGroups = kBlock64 / kCombineRows;
    const int lane = threadIdx.x & 31;
    const int items = a.inv.scalars[4] * a.nheads * kGroups * 2;
    for (int item = worker; item < items; item += workers) {
        const int which = item & 1, row0 = (item >> 1) % kGroups * kCombineRows;   // which = 0: dK, 1: dV
        const int hm = item / (2 * kGroups), kvh = a.head0 + hm % a.nheads;
        const int gp = a.inv.multi[hm / a.nheads];
        const int runs = a.inv.chunks[gp], q0 = a.inv.part0[gp];
        const int seq = slot_seq(a, gp), p = a.qb_block[gp];
        const int seq0 = a.cu_seqlens[seq];
        const int rows = a.cu_seqlens[seq + 1] - seq0 - p * kBlock64 - row0;       // rows behind these lie outside the sequence
        const float* pk = a.partial + (((size_t)q0 * a.hkv + kvh) * 2 + which) * (kBlock64 * D) + row0 * D + lane * kVec;
        const size_t run_stride = (size_t)a.hkv * 2 * kBlock64 * D;
        if (rows <= 0) continue;
        float sum[kCombineRows][kVec] = {};
#pragma unroll 4
        for (int r = 0; r < runs; ++r) {
#pragma unroll
            for (int i = 0; i < kCombineRows; ++i) {
#pragma unroll
                for (int e = 0; e < kVec; ++e) sum[i][e] += pk[r * run_stride + min(i, rows - 1) * D + e];
            }
        }
        uint32_t* out = reinterpret_cast<uint32_t*>((which ? a.dv : a.dk) + ((size_t)(seq0 + p * kBlock64 + row0) * a.hkv + kvh) * D + lane * kVec);
#pragma unroll
        for (int i = 0; i < kCombineRows; ++i) {
            if (i >= rows) break;
#pragma unroll
            for (int e = 0; e < kVec; e += 2) out[i * (a.hkv * D / 2) + e / 2] = pack_bf16x2(sum[i][e], sum[i][e + 1]);
        }
    }
}
template <int D>
__global__ void __launch_bounds__(256) bwd_combine_kernel(const BwdArgs a) {
    combine_runs<D>(a, blockIdx.x * 8 + (threadIdx.x >> 5), gridDim.x * 8);
}

// ---- dQ --------------------------------------------------------------------------------------------------------
//
// dQ += dS K_p over the list of a query block: 4 MMAs of 128 x d x 16 per entry.  Per entry the SM takes in 16 KB of dS
// and 16 KB of K (d = 128) and the MMAs read as much, 512 cycles of shared-memory bandwidth; the dS tiles come from HBM once
// they outgrow L2, which is then the bound (0.67 GB at 32K tokens, 16 query heads).
// Measured: 18 us at 4K tokens and 153 us at 32K (recomputing S and dP: 35 and 303): dS and K arrive at 8.7 TB/s in
// both cases, whether dS lies in L2 or comes from HBM, which is what bounds it now.
// One persistent CTA of 11 warps per SM; units are dealt out statically, longest list first (KV head by KV head, or all
// heads together: BwdArgs::interleave), back and forth over the CTAs:
//     warp 10   describes the units to the other roles: what the preparation wrote down of the query block, then its list, two
//               dependent loads, for 32 units at a time, one per lane.  (With every role looking its units up itself, in what was
//               a chain of four loads before the preparation made it, 4K tokens took 0.6 us more.)
//     warp 0    copies: the dS tile (as the dK/dV kernel left it: the K-major layout of an A operand) and the K tile of
//               every list entry, through a ring of kDqStages
//     warp 1    issues the MMAs; dQ accumulates in one of two buffers in tensor memory
//     warps 2-5  the finished dQ tile of a unit, through shared memory and TMA stores
//     warps 6-9  KV blocks whose readers were cut into several runs: the runs' partial sums of dK and dV, in run order
constexpr int kDqThreads = 352;
constexpr int kDqStages = 6;
constexpr int kDqUnits = 4;      // descriptions of units in shared memory

// What warp 10 tells the other roles about a unit.
struct DqDesc {
    int cnt;                     // list entries; 0: no more units
    int slot, j, seq0;           // query slot, its block, first token of the sequence
    int kvh, pair, seqlen;       // KV head, pair of query heads, tokens of the sequence
    int first[32];               // the first 32 list entries, as the route holds them
};

template <int D>
struct DqSmem {
    static constexpr int kKBytes = 64 * D * 2;
    static constexpr int kStage = kDsTile + kKBytes;
    static constexpr int kOut = kDqStages * kStage;          // 4 warps x 2 buffers x 32 rows x 64 B
    static constexpr int kUnit = kOut + 4 * 2 * 2048;        // DqDesc [kDqUnits]
    static constexpr int kBar = kUnit + (kDqUnits * (int)sizeof(DqDesc) + 15) / 16 * 16;
    static constexpr int kTotal = kBar + 256;
};

template <int D>
__global__ void __launch_bounds__(kDqThreads, 1) bwd_dq_kernel(const __grid_constant__ CUtensorMap tm_k,
                                                            const __grid_constant__ CUtensorMap tm_dq, const BwdArgs a) {
    using L = DqSmem<D>;
    extern __shared__ __align__(1024) uint8_t smem[];
    uint32_t& s_tmem = *reinterpret_cast<uint32_t*>(smem + L::kBar + 240);
    int& s_abort = *reinterpret_cast<int*>(smem + L::kBar + 244);
    const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31;
    const int pairs = a.group == 4 ? 2 : 1;
    const uint32_t base = smem_u32(smem), bars = base + L::kBar;
    volatile DqDesc* s_unit = reinterpret_cast<volatile DqDesc*>(smem + L::kUnit);
    const uint32_t full = bars;                              // [kDqStages] the entry's tiles landed
    const uint32_t free_ = full + 8 * kDqStages;             // [kDqStages] ... and have been used
    const uint32_t acc_full = free_ + 8 * kDqStages;         // [2] the unit's dQ is complete
    const uint32_t acc_free = acc_full + 16;                 // [2] ... and has been read out of tensor memory (4 warps)
    const uint32_t unit_full = acc_free + 16;                // [kDqUnits] the unit is described
    const uint32_t unit_free = unit_full + 8 * kDqUnits;     // [kDqUnits] ... and has been read (6 warps)
    static_assert(16 * kDqStages + 32 + 16 * kDqUnits <= 240, "barriers overlap the words behind them");
    if (tid == 0) {
        s_abort = (base & 1023u) ? 1 : 0;
        for (int s = 0; s < kDqStages; ++s) {
            mbar_init(full + 8 * s, 1);
            mbar_init(free_ + 8 * s, 1);
        }
        for (int b = 0; b < 2; ++b) {
            mbar_init(acc_full + 8 * b, 1);
            mbar_init(acc_free + 8 * b, 4);
        }
        for (int u = 0; u < kDqUnits; ++u) {
            mbar_init(unit_full + 8 * u, 1);
            mbar_init(unit_free + 8 * u, 6);
        }
        fence_mbar_init();
    }
    __syncwarp();
    if (warp == 0) {
        tmem_alloc(smem_u32(&s_tmem), 256);
        tmem_relinquish();
    }
    pdl_wait();
    int nqb = 0;
    DqUnit u;
    if (warp == 10) {       // its first units, beside the status word
        nqb = min(*a.num_qblocks, a.capacity);
        if (a.inv.scalars[0] == 0) nqb = 0;     // the dK/dV kernel had no units: there is no dS
        u = dq_unit(a, lane, nqb, pairs);
    }
    if (tid == 0 && a.status) {
        if (s_abort) atomicOr(a.status, BF1_DEV_WAIT_TIMEOUT);
        if (*a.status & BF1_DEV_WAIT_TIMEOUT) s_abort = 1;
    }
    tc_fence_before();
    __syncthreads();
    tc_fence_after();
    const uint32_t tmem = s_tmem;
    volatile int* abort_flag = &s_abort;
    if (s_abort) {   // (uniform over the CTA)
        __syncthreads();
        if (warp == 0) tmem_dealloc(tmem, 256);
        return;
    }
    auto wait_unit = [&](int n) -> volatile DqDesc& {
        mbar_wait(unit_full + 8 * (n % kDqUnits), (n / kDqUnits) & 1, abort_flag, a.status);
        return s_unit[n % kDqUnits];
    };
    auto free_unit = [&](int n) {
        __syncwarp();
        if (lane == 0) mbar_arrive(unit_free + 8 * (n % kDqUnits));
    };
    if (warp == 0) {
        // ---- copies ----
        const size_t tiles = (size_t)a.capacity * a.max_degree;
        int r = 0, rs = 0, rk = 0;      // entries so far, as (stage, turn of the ring)
        for (int n = 0;; ++n) {
            volatile DqDesc& u = wait_unit(n);
            const int cnt = u.cnt, slot = u.slot, j = u.j, seq0 = u.seq0, kvh = u.kvh, pair = u.pair;
            int p = u.first[lane];
            free_unit(n);
            if (cnt == 0 || *abort_flag) break;
            const char* ds = reinterpret_cast<const char*>(a.ds) +
                             (((size_t)(kvh - a.head0) * pairs + pair) * tiles + (size_t)slot * a.max_degree) * kDsTile;
            for (int it = 0; it < cnt; ++it) {
                if (it > 0 && (it & 31) == 0)   // lists longer than a warp: the next 32 entries
                    p = it + lane < cnt ? a.kv_idx[(size_t)slot * a.max_degree + it + lane] : 0;
                const int kb = safe_entry(__shfl_sync(0xffffffffu, p, it & 31), it, cnt, j);
                if (r >= kDqStages) mbar_wait(free_ + 8 * rs, (rk - 1) & 1, abort_flag, a.status);
                if (elect_one()) {
                    const uint32_t dst = base + rs * L::kStage;
                    mbar_expect_tx(full + 8 * rs, L::kStage);
                    bulk_load(dst, ds + (size_t)it * kDsTile, kDsTile, full + 8 * rs);
                    tma_load_4d(dst + kDsTile, &tm_k, 0, seq0 + kb * kBlock64, kvh, 0, full + 8 * rs);
                }
                __syncwarp();
                ++r;
                if (++rs == kDqStages) { rs = 0; ++rk; }
            }
        }
    } else if (warp == 10) {
        // ---- units, 32 at a time ----
        bool more = true;
        for (int n0 = 0; more; n0 += 32) {
            if (n0 > 0) u = dq_unit(a, n0 + lane, nqb, pairs);
            int p_next = 0;
            auto list_of = [&](int k) {
                const int slot = __shfl_sync(0xffffffffu, u.slot, k);
                p_next = lane < a.max_degree ? a.kv_idx[(size_t)slot * a.max_degree + lane] : 0;
            };
            list_of(0);
            for (int k = 0; k < 32 && more; ++k) {
                const int n = n0 + k, ub = n % kDqUnits, p = p_next;
                more = __shfl_sync(0xffffffffu, u.ok, k) && !*abort_flag;
                if (k < 31) list_of(k + 1);            // (on its way while this unit's place is waited for)
                if (n >= kDqUnits) mbar_wait(unit_free + 8 * ub, (n / kDqUnits - 1) & 1, abort_flag, a.status);
                volatile DqDesc& d = s_unit[ub];
                d.first[lane] = p;
                if (lane == k) {
                    d.cnt = more ? u.cnt : 0;
                    d.slot = u.slot;
                    d.j = u.j;
                    d.seq0 = u.seq0;
                    d.kvh = u.kvh;
                    d.pair = u.pair;
                    d.seqlen = u.seqlen;
                }
                __syncwarp();
                if (lane == 0) mbar_arrive(unit_full + 8 * ub);
            }
        }
    } else if (warp == 1) {
        // ---- MMAs: A = dS [128 q][64 kv] K-major (16 kv = 32 bytes per step), B = K tile MN-major (16 kv rows = 2048
        // bytes per step, next 64 d columns 8 KB away) ----
        constexpr uint32_t kHi = desc_hi_sw128(1024);
        constexpr uint32_t kIdQ = idesc_bf16_f32(D, true);
        int rs = 0;
        uint32_t phase = 0;
        for (int n = 0;; ++n) {
            const int cnt = wait_unit(n).cnt;
            free_unit(n);
            if (cnt == 0 || *abort_flag) break;
            const int b = n & 1;
            if (n >= 2) mbar_wait(acc_free + 8 * b, ((n >> 1) - 1) & 1, abort_flag, a.status);
            for (int it = 0; it < cnt; ++it) {
                mbar_wait(full + 8 * rs, phase, abort_flag, a.status);
                tc_fence_after();
                if (elect_one()) {
                    const uint32_t alo = desc_lo_sw128(base + rs * L::kStage, 16);
                    const uint32_t blo = desc_lo_sw128(base + rs * L::kStage + kDsTile, 8192);
#pragma unroll
                    for (int kk = 0; kk < 4; ++kk) {
                        if (kk == 0 && it == 0) mma_ss_lohi<false>(tmem + b * 128, alo, blo, kHi, kIdQ);
                        else mma_ss_lohi<true>(tmem + b * 128, alo + ((kk * 32) >> 4), blo + ((kk * 2048) >> 4), kHi, kIdQ);
                    }
                    mma_commit(free_ + 8 * rs);
                    if (it == cnt - 1) mma_commit(acc_full + 8 * b);
                }
                __syncwarp();
                if (++rs == kDqStages) { rs = 0; phase ^= 1; }
            }
        }
    } else if (warp < 6) {
        // ---- finished dQ tiles: one thread per row ----
        const int quarter = warp & 3, row = quarter * 32 + lane, hl = row >> 6, tl = row & 63;
        const uint32_t t_lane = tmem + (static_cast<uint32_t>(quarter * 32) << 16);
        const uint32_t stage_w = base + L::kOut + quarter * 4096;
        for (int n = 0;; ++n) {
            volatile DqDesc& u = wait_unit(n);
            const int cnt = u.cnt, h = u.kvh * a.group + u.pair * 2 + hl, tok0 = u.seq0 + u.j * kBlock64;
            const int rows_valid = min(kBlock64, u.seqlen - u.j * kBlock64);
            const bool head_ok = u.pair * 2 + hl < a.group;   // G = 1: rows 64..127 belong to no head (warp-uniform)
            free_unit(n);
            if (cnt == 0 || *abort_flag) break;
            const int b = n & 1;
            mbar_wait(acc_full + 8 * b, (n >> 1) & 1, abort_flag, a.status);
            tc_fence_after();
            uint32_t pk[D / 2];
#pragma unroll
            for (int c = 0; c < D / 32; ++c) {
                uint32_t v[32];
                tmem_ld32(t_lane + b * 128 + c * 32, v);
                tmem_wait_ld();
#pragma unroll
                for (int e = 0; e < 16; ++e) pk[c * 16 + e] = pack_bf16x2(__uint_as_float(v[2 * e]), __uint_as_float(v[2 * e + 1]));
            }
            tc_fence_before();
            __syncwarp();
            if (lane == 0) mbar_arrive(acc_free + 8 * b);
            if (head_ok && (tl | 31) < rows_valid) {        // all 32 rows of the warp lie in the sequence (warp-uniform)
                const uint32_t sw = (lane >> 1) & 3;          // 64-byte swizzle: chunk ^= (row / 2) % 4
#pragma unroll
                for (int c = 0; c < D / 32; ++c) {            // 32 columns at a time, two staging tiles in turn
                    const uint32_t tile = stage_w + (c & 1) * 2048;
                    if (lane == 0) bulk_wait_read1();         // the store before the last has read its tile
                    __syncwarp();
#pragma unroll
                    for (int ch = 0; ch < 4; ++ch)
                        st_shared_v4(tile + lane * 64 + ((ch ^ sw) << 4), pk[c * 16 + ch * 4], pk[c * 16 + ch * 4 + 1],
                                     pk[c * 16 + ch * 4 + 2], pk[c * 16 + ch * 4 + 3]);
                    fence_proxy_async();
                    __syncwarp();
                    if (lane == 0) {
                        tma_store_3d(&tm_dq, c * 32, h, tok0 + (tl & 32), tile);
                        bulk_commit_group();
                    }
                }
            } else if (head_ok && tl < rows_valid) {        // the rows after these belong to someone else
                __nv_bfloat16* dqrow = a.dq + ((size_t)(tok0 + tl) * a.hq + h) * D;
#pragma unroll
                for (int c = 0; c < D / 8; ++c)
                    *reinterpret_cast<uint4*>(dqrow + c * 8) = make_uint4(pk[c * 4], pk[c * 4 + 1], pk[c * 4 + 2], pk[c * 4 + 3]);
            }
        }
        if (lane == 0) bulk_wait_read0();     // (that the stores land is waited for by the end of the grid)
        __syncwarp();
    } else {
        combine_runs<D>(a, blockIdx.x * 4 + (warp - 6), gridDim.x * 4);
    }
    tc_fence_before();
    __syncthreads();
    if (warp == 0) tmem_dealloc(tmem, 256);
}

int make_map_4d(CUtensorMap* m, const void* ptr, int64_t T, int H, int d, int heads_per_box, int chunks_per_box);   // bf1_attn.cu
int make_store_map(CUtensorMap* m, void* ptr, int64_t T, int H, int d);                                             // bf1_attn.cu

// Where everything lives in the caller's workspace (256-byte aligned sections).
struct BwdLayout {
    size_t delta, ints, partial, ds, total;
    int ds_heads;   // KV heads whose dS is kept at a time; 0: dS is computed again
    size_t n_count, n_start, n_chunks, n_part0, n_readers, n_units, n_parts, n_multi, n_ranked;
    BwdLayout(int64_t T, int hq, int hkv, int d, int cap, int max_degree) {
        auto up = [](size_t x) { return (x + 255) / 256 * 256; };
        n_count = (size_t)cap + 1;
        n_start = (size_t)cap + 1;
        n_chunks = (size_t)cap;
        n_part0 = (size_t)cap;
        n_readers = (size_t)cap * max_degree;
        // (what run_length() can make of as many readers; a slot whose readers are not cut has one unit)
        n_parts = std::max<size_t>(cap, std::min<size_t>(2 * (size_t)cap * max_degree / kLeastChunk, 2 * kSms / hkv + 1));
        n_units = cap + n_parts;
        n_multi = (size_t)cap;
        n_ranked = 2 * (size_t)cap;
        delta = 0;
        ints = up((size_t)T * hq * sizeof(float));
        const size_t n_ints = n_count + 2 * n_start + n_chunks + n_part0 + n_readers + 8 * n_units + 4 * n_ranked + (size_t)hkv + n_multi + 8;
        partial = ints + up(n_ints * sizeof(int32_t));
        ds = partial + up(n_parts * hkv * 2 * kBlock64 * d * sizeof(float));
        const int64_t per_head = (int64_t)cap * max_degree * (hq / hkv == 4 ? 2 : 1) * kDsTile;
        ds_heads = per_head > kDsMost ? 0 : (int)std::max<int64_t>(1, std::min<int64_t>(hkv, kDsGroup / per_head));
        total = ds + up((size_t)ds_heads * per_head);
    }
};

}  // namespace bf1

using namespace bf1;

extern "C" int64_t bf1_attn_bwd_workspace_bytes(const bf1_route* route, int64_t total_tokens, int32_t hq, int32_t hkv,
                                                int32_t d) {
    if (!route || total_tokens < 0 || hq <= 0 || hkv <= 0 || d <= 0 || route->capacity_qblocks < 1 || route->max_degree < 1)
        return -1;
    return (int64_t)BwdLayout(total_tokens, hq, hkv, d, route->capacity_qblocks, route->max_degree).total;
}

extern "C" int bf1_attn_bwd(const void* q, const void* k, const void* v, const void* o, const float* lse,
                            const void* d_o, const int32_t* cu_seqlens_dev, int32_t batch, int64_t total_tokens,
                            int32_t max_seqlen, int32_t hq, int32_t hkv, int32_t d, float softmax_scale,
                            const bf1_route* route, void* workspace, void* dq, void* dk, void* dv, void* stream) {
    if (!q || !k || !v || !o || !lse || !d_o || !cu_seqlens_dev || !route || !workspace || !dq || !dk || !dv)
        return fail(BF1_ERR_INVALID_ARG, "a pointer is null");
    if (batch < 0 || total_tokens < 0 || max_seqlen < 0 || hq <= 0 || hkv <= 0)
        return fail(BF1_ERR_INVALID_ARG, "negative or zero size argument");
    if (total_tokens > 0x7fffffffLL - 64) return fail(BF1_ERR_UNSUPPORTED, "total_tokens does not fit 32-bit token indices");
    if (hq % hkv != 0) return fail(BF1_ERR_INVALID_ARG, "hq %d is not a multiple of hkv %d", hq, hkv);
    const int group = hq / hkv;
    if (group != 1 && group != 2 && group != 4)
        return fail(BF1_ERR_UNSUPPORTED, "GQA group size %d: only G = 1, 2 and 4 are supported", group);
    if (d != 64 && d != 128) return fail(BF1_ERR_UNSUPPORTED, "head dimension %d: only 64 and 128 are supported", d);
    if (((uintptr_t)q | (uintptr_t)k | (uintptr_t)v | (uintptr_t)o | (uintptr_t)d_o | (uintptr_t)dq | (uintptr_t)dk |
         (uintptr_t)dv) & 15)
        return fail(BF1_ERR_INVALID_ARG, "tensors must be 16-byte aligned");
    if ((uintptr_t)workspace & 255) return fail(BF1_ERR_INVALID_ARG, "workspace must be 256-byte aligned");
    if (!route->qb_seq || !route->qb_block || !route->kv_count || !route->kv_idx || !route->num_qblocks || !route->status)
        return fail(BF1_ERR_INVALID_ARG, "a route array pointer is null");
    if (route->capacity_qblocks < 1 || route->max_degree < 1 || hkv > 65535)
        return fail(BF1_ERR_CAPACITY, "bad route capacities or hkv");
    if (total_tokens == 0 || batch == 0) return BF1_OK;
    int dev = 0, major = 0;
    BF1_CUDA_CHECK(cudaGetDevice(&dev));
    BF1_CUDA_CHECK(cudaDeviceGetAttribute(&major, cudaDevAttrComputeCapabilityMajor, dev));
    if (major != 10) return fail(BF1_ERR_NO_DEVICE, "device compute capability %d.x is not sm_100", major);
    static std::atomic<bool> configured[64];
    if (dev < 0 || dev >= 64) return fail(BF1_ERR_NO_DEVICE, "device ordinal %d out of range", dev);
    if (!configured[dev].load(std::memory_order_acquire)) {
        const int kInvBytes = kInvInts * (int)sizeof(int32_t);
        BF1_CUDA_CHECK(cudaFuncSetAttribute(bwd_prep_kernel<128, true>, cudaFuncAttributeMaxDynamicSharedMemorySize, kInvBytes));
        BF1_CUDA_CHECK(cudaFuncSetAttribute(bwd_prep_kernel<64, true>, cudaFuncAttributeMaxDynamicSharedMemorySize, kInvBytes));
        BF1_CUDA_CHECK(cudaFuncSetAttribute(bwd_dq_kernel<128>, cudaFuncAttributeMaxDynamicSharedMemorySize, DqSmem<128>::kTotal));
        BF1_CUDA_CHECK(cudaFuncSetAttribute(bwd_dq_kernel<64>, cudaFuncAttributeMaxDynamicSharedMemorySize, DqSmem<64>::kTotal));
        BF1_CUDA_CHECK(cudaFuncSetAttribute(bwd_dq_recompute_kernel<128>, cudaFuncAttributeMaxDynamicSharedMemorySize, DqrSmem<128>::kTotal));
        BF1_CUDA_CHECK(cudaFuncSetAttribute(bwd_dq_recompute_kernel<64>, cudaFuncAttributeMaxDynamicSharedMemorySize, DqrSmem<64>::kTotal));
        BF1_CUDA_CHECK(cudaFuncSetAttribute(bwd_dkv_kernel<128>, cudaFuncAttributeMaxDynamicSharedMemorySize, DkvSmem<128>::kTotal));
        BF1_CUDA_CHECK(cudaFuncSetAttribute(bwd_dkv_kernel<64>, cudaFuncAttributeMaxDynamicSharedMemorySize, DkvSmem<64>::kTotal));
        configured[dev].store(true, std::memory_order_release);
    }
    CUtensorMap tq, tk, tv, tg, tdq;
    // Q and dO: two heads and all column chunks per copy; with one head per KV head, one head and one chunk
    const int q_heads = group == 1 ? 1 : 2, q_chunks = group == 1 ? 1 : d / 64;
    if (int rc = make_map_4d(&tq, q, total_tokens, hq, d, q_heads, q_chunks)) return rc;
    if (int rc = make_map_4d(&tg, d_o, total_tokens, hq, d, q_heads, q_chunks)) return rc;
    if (int rc = make_store_map(&tdq, dq, total_tokens, hq, d)) return rc;
    if (int rc = make_map_4d(&tk, k, total_tokens, hkv, d, 1, d / 64)) return rc;
    if (int rc = make_map_4d(&tv, v, total_tokens, hkv, d, 1, d / 64)) return rc;
    const int cap = route->capacity_qblocks;
    const BwdLayout lay(total_tokens, hq, hkv, d, cap, route->max_degree);
    char* ws = (char*)workspace;
    BwdArgs a;
    a.cu_seqlens = cu_seqlens_dev;
    a.qb_seq = route->qb_seq;
    a.qb_block = route->qb_block;
    a.kv_count = route->kv_count;
    a.kv_idx = route->kv_idx;
    a.num_qblocks = route->num_qblocks;
    a.order = route->order;
    a.batch = batch;
    a.max_degree = route->max_degree;
    a.capacity = cap;
    a.total_tokens = (int32_t)total_tokens;
    a.hq = hq;
    a.hkv = hkv;
    a.group = group;
    a.status = route->status;
    a.scale = softmax_scale > 0.f ? softmax_scale : 1.0f / sqrtf((float)d);
    a.scale_log2 = a.scale * 1.4426950408889634f;
    // The same rule as the forward's hand-out order: while K and V of all heads fit L2 together there is nothing
    // to gain from working head by head, and the longest units of all heads first balance the CTAs better.
    a.interleave = (total_tokens * (int64_t)hkv * d * 4 <= (48LL << 20)) ? 1 : 0;
    a.o = (const __nv_bfloat16*)o;
    a.d_o = (const __nv_bfloat16*)d_o;
    a.lse = lse;
    a.delta = (float*)(ws + lay.delta);
    a.dq = (__nv_bfloat16*)dq;
    a.dk = (__nv_bfloat16*)dk;
    a.dv = (__nv_bfloat16*)dv;
    a.partial = (float*)(ws + lay.partial);
    a.inv.units = (int4*)(ws + lay.ints);   // (16-byte entries first)
    a.inv.ranked = a.inv.units + 2 * lay.n_units;
    int32_t* ip = (int32_t*)(a.inv.ranked + lay.n_ranked);
    a.inv.count = ip;            ip += lay.n_count;
    a.inv.start = ip;            ip += lay.n_start;
    a.inv.unit0 = ip;            ip += lay.n_start;
    a.inv.chunks = ip;           ip += lay.n_chunks;
    a.inv.part0 = ip;            ip += lay.n_part0;
    a.inv.readers = ip;          ip += lay.n_readers;
    a.inv.tickets = ip;          ip += hkv;
    a.inv.multi = ip;            ip += lay.n_multi;
    a.inv.scalars = ip;
    a.inv.cap = cap;
    a.inv.max_units = (int32_t)lay.n_units;
    a.inv.max_parts = (int32_t)lay.n_parts;
    cudaStream_t st = (cudaStream_t)stream;
    int sms = 0;
    BF1_CUDA_CHECK(cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev));
    a.sms = sms;
    // D_i of every row, and the inverse route (readers of every KV block, cut into units)
    const bool one_cta = inverse_words(cap, route->max_degree) <= kInvInts;
    // (one CTA fits an SM: with the inverse route's there must not be more than SMs, or the last one runs all by itself)
    const int prep_ctas = (int)std::max<int64_t>(1, std::min<int64_t>(sms - (one_cta ? 1 : 0), ((total_tokens + 15) / 16 * hq + 31) / 32));
    if (!one_cta) {
        BF1_CUDA_CHECK(cudaMemsetAsync(a.inv.count, 0, lay.n_count * sizeof(int32_t), st));
        const int grid_inv = (int)std::min<int64_t>(((int64_t)cap * route->max_degree + 255) / 256, 4 * (int64_t)sms);
        inverse_route_kernel<false><<<grid_inv, 256, 0, st>>>(a);
        inverse_units_kernel<<<1, 1024, 0, st>>>(a);
        inverse_route_kernel<true><<<grid_inv, 256, 0, st>>>(a);
        inverse_sort_kernel<<<cap, 256, 0, st>>>(a);
        BF1_CUDA_CHECK(launch_pdl(d == 128 ? bwd_prep_kernel<128, false> : bwd_prep_kernel<64, false>, prep_ctas, 1024, 0, st, a));
    } else {
        const int inv_bytes = (int)inverse_words(cap, route->max_degree) * (int)sizeof(int32_t);
        BF1_CUDA_CHECK(launch_pdl(d == 128 ? bwd_prep_kernel<128, true> : bwd_prep_kernel<64, true>, prep_ctas + 1, 1024,
                                  inv_bytes, st, a));
    }
    BF1_CUDA_CHECK(cudaGetLastError());
    // dK / dV along the inverse route, then dQ along the route, for as many KV heads at a time as the dS buffer holds
    const int step = lay.ds_heads ? lay.ds_heads : hkv;
    a.ds = lay.ds_heads ? (__nv_bfloat16*)(ws + lay.ds) : nullptr;
    for (int h0 = 0; h0 < hkv; h0 += step) {
        a.head0 = h0;
        a.nheads = std::min(step, hkv - h0);
        const int busy_q = (int)std::min<int64_t>(sms, (int64_t)cap * a.nheads * (group == 4 ? 2 : 1));   // persistent: one CTA per SM
        const int grid_q = a.ds ? sms : busy_q;          // (CTAs without a unit add up partial sums all the same)
        const int grid_kv = (int)std::min<int64_t>(sms, (int64_t)lay.n_units * a.nheads);
        if (d == 128) {
            BF1_CUDA_CHECK(launch_pdl(bwd_dkv_kernel<128>, grid_kv, kDkvThreads, DkvSmem<128>::kTotal, st, tq, tk, tv, tg, a));
            if (a.ds) {
                BF1_CUDA_CHECK(launch_pdl(bwd_dq_kernel<128>, grid_q, kDqThreads, DqSmem<128>::kTotal, st, tk, tdq, a));
            } else {
                bwd_dq_recompute_kernel<128><<<grid_q, kDqrThreads, DqrSmem<128>::kTotal, st>>>(tq, tk, tv, tg, a);
                bwd_combine_kernel<128><<<4 * sms, 256, 0, st>>>(a);
            }
        } else {
            BF1_CUDA_CHECK(launch_pdl(bwd_dkv_kernel<64>, grid_kv, kDkvThreads, DkvSmem<64>::kTotal, st, tq, tk, tv, tg, a));
            if (a.ds) {
                BF1_CUDA_CHECK(launch_pdl(bwd_dq_kernel<64>, grid_q, kDqThreads, DqSmem<64>::kTotal, st, tk, tdq, a));
            } else {
                bwd_dq_recompute_kernel<64><<<grid_q, kDqrThreads, DqrSmem<64>::kTotal, st>>>(tq, tk, tv, tg, a);
                bwd_combine_kernel<64><<<4 * sms, 256, 0, st>>>(a);
            }
        }
    }
    BF1_CUDA_CHECK(cudaGetLastError());
    return BF1_OK;
}
