// BF1 cached one-token decode over selected KV pages (paper Section 3.2 and 5.4).
//
// The newest token of a sequence of n cached tokens (position n-1, block j = (n-1) / 64) reads
// the pages of P(j) -- O(log B) pages, O(b d log B) key/value elements per head -- out of a paged
// KV cache: page = 64 tokens, [page, 64, Hkv, d] bf16, logical block -> physical page through a
// page table.  The page list only changes when n crosses a block boundary, so the plan
// (bf1_plan_decode) is made once per 64-token "route epoch" and reused by every decode step in
// it; the attention call reads the current lengths itself to find how many tokens of the self
// page are valid.  The paper measures planning at 100-121 us against 12-23 us of execution and
// names plan reuse across the epoch as the open problem; here the plan is a ~3 us kernel and is
// off the per-token path.
//
// The work is memory-bound (every selected K/V byte is read once, 2*G MACs per element): one kernel,
// decode_fused_kernel, in which a CTA serves one KV head with all its query heads and walks a page list, or a part of
// it, with an online softmax over a ring of cp.async page pairs.  With enough lists to fill the GPU a CTA takes a whole
// list; with fewer, every list is cut into even parts, and the CTAs of a list form a thread-block cluster: they send a
// partial (max, sum, O) into the shared memory of the CTA that adds the parts up, in list order (each CTA of the cluster some
// of the columns).  Partial results in global memory behind an atomic ticket were a chain of store, fence, atomic and reload
// at the end of every call, and partial results that the first CTA fetched from the others' shared memory needed a second cluster
// barrier: 6.6, 4.6 and 4.3 us for one sequence of 32K tokens (16 query / 8 KV heads, d = 128).
// Rounding P to bf16 costs more precision the longer a part is (a key that is the part's maximum has P = 1 and is not rounded
// at all).  Where a list is cut, what the rounding takes away is therefore multiplied with V as well: it stands in rows of the
// mma's operand that were zero, so that it costs no mma.  The relative error against 64 bits is then 1.6e-3 (the rounding of
// the result) whatever the parts are, 1.95e-3 page by page without it and 1.99e-3 in parts of two pages, and
// the parts are free to be what is fastest: eight sequences of 65 to 32768 tokens 7.2 -> 6.1 us against runs that were
// kept short for their precision and dealt to the CTAs.  Where there are lists for every SM (four
// heads, d = 128: for half of them), P is rounded.
// Four query heads share a CTA and with it one reading of K and V (a CTA for each pair of heads before): 192 lists of 11
// pages 23.6 -> 13.9 us, 40 lists 9.5 -> 6.0.
#include <algorithm>
#include <atomic>
#include <cfloat>

#include "bf1_common.cuh"

namespace bf1 {

constexpr int kPage = 64;             // tokens per page = block width b
constexpr int kDecThreads = 128;
constexpr int kDecStages = 3;          // page-pair buffers per CTA
// CTAs asked for, at most, while there are few lists (how many fit decides): over 645 shapes 0.3 % faster than two, on average.
constexpr int kDecCtasPerSm = 4;
// CTAs of a cluster at most.  Above 8 a cluster may find fewer places (bf1_decode_fwd asks), but a CTA with one page instead
// of two or more wins whatever it costs: one list of 11 / 41 / 64 pages takes 5.1 / 9.4 / 11.6 us with eight CTAs, 4.0 /
// 6.7 / 8.1 with up to sixteen.
constexpr int kMaxCtas = 16;

struct DecodeArgs {
    const __nv_bfloat16* q;           // [batch, hq, d]
    const __nv_bfloat16* k_pages;     // [pages, 64, hkv, d]
    const __nv_bfloat16* v_pages;
    const int32_t* seqlens;           // [batch] current cached lengths (>= 0)
    const int32_t* count;             // plan: [batch] pages to read
    const int32_t* page;              // plan: [batch, max_degree] physical pages, self page last
    const int32_t* block;             // plan: [batch] block index the plan was made for
    int32_t* status;
    int32_t max_degree, hq, hkv, num_pages;
    int32_t group;                    // G = hq / hkv (1, 2 or 4)
    float scale_log2;
    __nv_bfloat16* o;                 // [batch, hq, d]
    float* lse;                       // [hq, batch]
    int32_t batch;
    int32_t nctas;                    // CTAs (a cluster) that a page list is dealt to
    int32_t share;                    // columns (of the heads' G d) a CTA of the cluster adds up, a multiple of 32
    int32_t sums, gather, ring;       // shared memory: the CTA's RunState, then from these bytes on (max, sum) [CTA][heads] and
                                      // columns [CTA][share] of the list's parts, and the page ring
};

__device__ __forceinline__ void cp_async_commit() { asm volatile("cp.async.commit_group;" ::: "memory"); }
template <int N>
__device__ __forceinline__ void cp_async_wait() {
    asm volatile("cp.async.wait_group %0;" ::"n"(N) : "memory");
}

// cp.async that writes zeros when src_bytes is 0 (rows behind the newest token: unwritten cache memory
// that may hold anything, NaN included, and must not reach a multiply)
__device__ __forceinline__ void cp_async16_zfill(uint32_t dst, const void* src, uint32_t src_bytes) {
    asm volatile("cp.async.cg.shared.global [%0], [%1], 16, %2;" ::"r"(dst), "l"(src), "r"(src_bytes) : "memory");
}
__device__ __forceinline__ void mma_16816(float (&c)[4], uint32_t a0, uint32_t a1, uint32_t a2, uint32_t a3, uint32_t b0,
                                          uint32_t b1) {
    asm volatile("mma.sync.aligned.m16n8k16.row.col.f32.bf16.bf16.f32 {%0, %1, %2, %3}, {%4, %5, %6, %7}, {%8, %9}, {%0, %1, %2, %3};"
                 : "+f"(c[0]), "+f"(c[1]), "+f"(c[2]), "+f"(c[3])
                 : "r"(a0), "r"(a1), "r"(a2), "r"(a3), "r"(b0), "r"(b1));
}
__device__ __forceinline__ void ldmatrix_x4_trans(uint32_t addr, uint32_t& r0, uint32_t& r1, uint32_t& r2, uint32_t& r3) {
    asm volatile("ldmatrix.sync.aligned.m8n8.x4.trans.shared.b16 {%0, %1, %2, %3}, [%4];"
                 : "=r"(r0), "=r"(r1), "=r"(r2), "=r"(r3)
                 : "r"(addr));
}

__device__ __forceinline__ void cluster_arrive_relaxed() { asm volatile("barrier.cluster.arrive.relaxed.aligned;" ::: "memory"); }
__device__ __forceinline__ void cluster_arrive() { asm volatile("barrier.cluster.arrive.release.aligned;" ::: "memory"); }
__device__ __forceinline__ void cluster_wait() { asm volatile("barrier.cluster.wait.acquire.aligned;" ::: "memory"); }
// This shared-memory address in the cluster's CTA `rank`.
__device__ __forceinline__ uint32_t map_cluster(uint32_t addr, uint32_t rank) {
    uint32_t r;
    asm volatile("mapa.shared::cluster.u32 %0, %1, %2;" : "=r"(r) : "r"(addr), "r"(rank));
    return r;
}
template <int N>
__device__ __forceinline__ void st_cluster(uint32_t addr, const float (&v)[N]) {      // 4 N bytes, aligned to as many
    if constexpr (N == 4) asm volatile("st.shared::cluster.v4.f32 [%0], {%1, %2, %3, %4};" ::"r"(addr), "f"(v[0]), "f"(v[1]), "f"(v[2]), "f"(v[3]) : "memory");
    else if constexpr (N == 2) asm volatile("st.shared::cluster.v2.f32 [%0], {%1, %2};" ::"r"(addr), "f"(v[0]), "f"(v[1]) : "memory");
    else asm volatile("st.shared::cluster.f32 [%0], %1;" ::"r"(addr), "f"(v[0]) : "memory");
}
// x / y for small whole numbers (below 2^20: half a step from a whole quotient is more than the division's error)
__device__ __forceinline__ int small_div(int x, int y) { return (int)__fdividef((float)x + 0.5f, (float)y); }

// A sum over the rounded weights and the one over what rounding left of them.  Where V is not finite the first says it all, as in a
// whole list: the rest of a weight is zero or has the other sign half of the time, and would make NaN of an infinity.
__device__ __forceinline__ float with_rest(float sum, float rest) { return fabsf(sum) <= FLT_MAX ? sum + rest : sum; }

// One CTA per (sequence, KV head[, part of the list]).  Pages stream in through a kDecStages-deep cp.async ring with ONE
// block-wide synchronisation per page; inside a page each of the four warps owns 16 keys and keeps its own online-softmax
// state (max, sum, O) for all grouped heads, merged at the end.  The arithmetic uses warp-level mma (m16n8k16): the work
// is memory-bound, but as scalar FMAs it was a chain of 1500 dependent instructions and five synchronisations per page,
// which is what bounded the kernel.  The grouped heads are rows 0 .. G - 1 of the 16-row operand; in P V their weights
// rounded to bf16 are rows 0 .. G - 1 and what the rounding left over is rows 8 .. 8 + G - 1.
template <int D, int kHeads>
struct RunState {                                       // the four warps' states at the end of the CTA's part
    float o[4][kHeads][D + 8], m[4][kHeads], l[4][kHeads];   // (rows 8 banks apart)
};
// kSplit: the list is cut, and the CTAs of a cluster add the parts up.  kRest: what rounding takes from P is multiplied with V too (always
// where the list is cut).
template <int D, int kHeads, bool kSplit, bool kRest>
__global__ void __launch_bounds__(kDecThreads, D == 64 ? 4 : 2) decode_fused_kernel(const DecodeArgs a) {
    constexpr int kRowBytes = D * 2;
    constexpr int kVecPerRow = D / 8;                   // 16-byte chunks per row
    constexpr int kVecPerThread = kPage * kVecPerRow / kDecThreads;
    constexpr int kPageBytes = kPage * D * 2;
    // [stage][K | V][64 rows][D bf16]; the 16-byte chunks of every row are XOR-swizzled with (row & 7), which
    // keeps both the B-fragment loads of K (8 rows, same chunk) and the ldmatrix rows of V conflict-free
    extern __shared__ __align__(128) uint8_t dsmem[];
    RunState<D, kHeads>& st = *reinterpret_cast<RunState<D, kHeads>*>(dsmem);   // in front of the ring
    __shared__ int sPages[64];                          // the sequence's page list (max_degree <= 64)

    const int kvh = blockIdx.x, s = blockIdx.y, tid = threadIdx.x;
    const int hbase = kvh * a.group;                    // first query head of this CTA (kHeads of them, one if G = 1)
    const int warp = tid >> 5, lane = tid & 31, gid = lane >> 2, tig = lane & 3;
    // The page list is fetched together with the plan's count and the length (independent loads in flight at
    // once), not after them: at small batch the kernel is one chain of dependent memory round trips.
    pdl_wait();
    if (tid < a.max_degree) sPages[tid] = a.page[(size_t)s * a.max_degree + tid];
    int cnt = max(min(a.count[s], a.max_degree), 0);
    const int n = a.seqlens[s];
    const int j = (n - 1) / kPage;
    if (cnt > 0 && j != a.block[s]) {    // the plan belongs to another route epoch
        if (tid == 0 && kvh == 0) atomicOr(a.status, BF1_DEV_BAD_ROUTE);
        cnt = 0;
    }
    // Nothing to do.  A CTA of a cluster stays all the same: whatever it reads here, the others may store to its shared memory.
    if (!kSplit && cnt == 0) return;
    const int tail = n - j * kPage;   // valid tokens of the self page (the last list entry)
    __syncthreads();                  // sPages is complete
    const int* pages = sPages;
    // the part of the list this CTA walks (may be empty)
    const int e_lo = kSplit ? small_div(blockIdx.z * cnt, a.nctas) : 0;
    const int e_hi = kSplit ? small_div((blockIdx.z + 1) * cnt, a.nctas) : cnt;
    const uint32_t ring = smem_u32(dsmem) + a.ring;
    auto issue_page = [&](int e, int stage) {
        int pg = pages[e];
        if (pg < 0 || pg >= a.num_pages) {
            if (tid == 0) atomicOr(a.status, BF1_DEV_BAD_ROUTE);
            pg = 0;
        }
        const int valid = (e == cnt - 1) ? tail : kPage;
        const size_t row_stride = (size_t)a.hkv * D;
        const __nv_bfloat16* kp = a.k_pages + ((size_t)pg * kPage * a.hkv + kvh) * D;
        const __nv_bfloat16* vp = a.v_pages + ((size_t)pg * kPage * a.hkv + kvh) * D;
        const uint32_t kb = ring + stage * 2 * kPageBytes, vb = kb + kPageBytes;
#pragma unroll
        for (int q = 0; q < kVecPerThread; ++q) {
            const int i = tid + q * kDecThreads, rr = i / kVecPerRow, c = i % kVecPerRow;
            const uint32_t off = rr * kRowBytes + ((c ^ (rr & 7)) << 4);
            const uint32_t nbytes = rr < valid ? 16u : 0u;
            cp_async16_zfill(kb + off, kp + rr * row_stride + c * 8, nbytes);
            cp_async16_zfill(vb + off, vp + rr * row_stride + c * 8, nbytes);
        }
    };
    // Two pages are asked for at the start and the third when the first has landed.  With three at once the first lands later: 64
    // lists of 11 / 26 pages that no cache holds 8.7 / 12.9 us in parts, 8.1 / 12.0 as it is (16 query / 8 KV heads, d = 128); 256 whole
    // lists of 11 and 12 pages, with their plan, 20.0 and 19.4.
#pragma unroll
    for (int i = 0; i < kDecStages - 1; ++i) {
        if (e_lo + i < e_hi) issue_page(e_lo + i, i);
        cp_async_commit();                               // possibly empty: keeps the group count uniform
    }
    if (kSplit) cluster_arrive_relaxed();                        // (waited for in front of the first store to another CTA)
    // A fragments of Q: the grouped heads are the first rows of the 16-row operand, the rest zero
    uint32_t qa[D / 16][2];
    {
        const uint32_t* qrow = reinterpret_cast<const uint32_t*>(a.q + ((size_t)s * a.hq + hbase + (gid < a.group ? gid : 0)) * D);
#pragma unroll
        for (int kk = 0; kk < D / 16; ++kk) {
            qa[kk][0] = gid < a.group ? qrow[kk * 8 + tig] : 0u;          // columns kk*16 + 2*tig, +1
            qa[kk][1] = gid < a.group ? qrow[kk * 8 + tig + 4] : 0u;      // columns kk*16 + 8 + 2*tig, +1
        }
    }
    float m_run = -INFINITY, l_run = 0.f;                // per lane: head gid (lanes with gid >= kHeads carry dummies)
    float acc[D / 8][4];
#pragma unroll
    for (int dn = 0; dn < D / 8; ++dn) acc[dn][0] = acc[dn][1] = acc[dn][2] = acc[dn][3] = 0.f;
    const int key0 = warp * 16;                          // this warp's 16 keys of every page

    for (int e = e_lo, stage = 0; e < e_hi; ++e) {
        cp_async_wait<kDecStages - 2>();                 // page e has landed (for this thread's copies)
        __syncthreads();                                 // ... for everybody's; and page e-1 is no longer read
        if (e + kDecStages - 1 < e_hi) issue_page(e + kDecStages - 1, stage == 0 ? kDecStages - 1 : stage - 1);
        cp_async_commit();
        const int valid = (e == cnt - 1) ? tail : kPage;
        const uint32_t kb = ring + stage * 2 * kPageBytes, vb = kb + kPageBytes;
        if (++stage == kDecStages) stage = 0;
        if (key0 >= valid) continue;                     // (warp-uniform) none of this warp's keys exist
        // ---- scores of 16 keys: two n-tiles of 8 keys, D / 16 k-steps ----------------------------
        float sc[2][4] = {{0.f, 0.f, 0.f, 0.f}, {0.f, 0.f, 0.f, 0.f}};
#pragma unroll
        for (int kk = 0; kk < D / 16; ++kk) {
#pragma unroll
            for (int nt = 0; nt < 2; ++nt) {
                const int key = key0 + nt * 8 + gid;     // B fragment: n = gid, k = 2*tig (+8)
                const uint32_t row = kb + key * kRowBytes + tig * 4;
                uint32_t b0, b1;
                asm volatile("ld.shared.b32 %0, [%1];" : "=r"(b0) : "r"(row + (((2 * kk) ^ (key & 7)) << 4)));
                asm volatile("ld.shared.b32 %0, [%1];" : "=r"(b1) : "r"(row + (((2 * kk + 1) ^ (key & 7)) << 4)));
                mma_16816(sc[nt], qa[kk][0], 0u, qa[kk][1], 0u, b0, b1);
            }
        }
        // lane (gid < kHeads, tig) holds head gid's scores of keys key0 + nt*8 + 2*tig, +1
        float sv[4];
        float mx = -INFINITY;
#pragma unroll
        for (int i = 0; i < 4; ++i) {
            const int key = key0 + (i >> 1) * 8 + 2 * tig + (i & 1);
            sv[i] = (gid < kHeads) ? ((key < valid) ? sc[i >> 1][i & 1] * a.scale_log2 : -INFINITY) : 0.f;
            mx = fmaxf(mx, sv[i]);
        }
        mx = fmaxf(mx, __shfl_xor_sync(0xffffffffu, mx, 1));
        mx = fmaxf(mx, __shfl_xor_sync(0xffffffffu, mx, 2));       // finite: key0 < valid
        const float m_new = fmaxf(m_run, mx);
        const float alpha = exp2f(m_run - m_new);           // 0 on the warp's first page
        float pv[4], psum = 0.f;
#pragma unroll
        for (int i = 0; i < 4; ++i) {
            pv[i] = exp2f(sv[i] - m_new);
            psum += pv[i];
        }
        psum += __shfl_xor_sync(0xffffffffu, psum, 1);
        psum += __shfl_xor_sync(0xffffffffu, psum, 2);
        l_run = l_run * alpha + psum;
        m_run = m_new;
        const bool rescale = __any_sync(0xffffffffu, alpha != 1.f);      // some head's maximum has moved
        // P as the A operand of the second mma: the C layout of the scores is the A layout of the next k-step.  Rows
        // 8 .. 15 hold what rounding to bf16 took from rows 0 .. 7
        uint32_t hi[2], lo[2];
#pragma unroll
        for (int i = 0; i < 2; ++i) {                    // keys 2*tig, +1 and 8 + 2*tig, +1
            hi[i] = pack_bf16x2(pv[2 * i], pv[2 * i + 1]);
            lo[i] = !kRest ? 0u : pack_bf16x2(pv[2 * i] - __uint_as_float(hi[i] << 16), pv[2 * i + 1] - __uint_as_float(hi[i] & 0xffff0000u));
            if (gid >= kHeads) hi[i] = lo[i] = 0u;
        }
        // ---- O = alpha * O + P V: D / 8 n-tiles of 8 columns, V fragments by ldmatrix.trans ---------
        const int lrow = key0 + (lane & 7) + ((lane >> 3) & 1) * 8;      // ldmatrix: lane supplies row (lane % 8) of matrix lane / 8
        const uint32_t vrow = vb + lrow * kRowBytes;
#pragma unroll
        for (int dn = 0; dn < D / 8; dn += 2) {
            if (rescale) {
#pragma unroll
                for (int i = 0; i < (kRest ? 4 : 2); ++i) acc[dn][i] *= alpha, acc[dn + 1][i] *= alpha;
            }
            uint32_t r0, r1, r2, r3;   // matrices: (keys 0-7, dn), (keys 8-15, dn), (keys 0-7, dn+1), (keys 8-15, dn+1)
            ldmatrix_x4_trans(vrow + (((dn + (lane >> 4)) ^ (lrow & 7)) << 4), r0, r1, r2, r3);
            mma_16816(acc[dn], hi[0], lo[0], hi[1], lo[1], r0, r1);
            mma_16816(acc[dn + 1], hi[0], lo[0], hi[1], lo[1], r2, r3);
        }
    }
    cp_async_wait<0>();
    if (gid < kHeads) {
        if (tig == 0) { st.m[warp][gid] = m_run; st.l[warp][gid] = l_run; }
#pragma unroll
        for (int dn = 0; dn < D / 8; ++dn)
            *reinterpret_cast<float2*>(&st.o[warp][gid][dn * 8 + 2 * tig]) = kRest ? make_float2(with_rest(acc[dn][0], acc[dn][2]), with_rest(acc[dn][1], acc[dn][3])) : make_float2(acc[dn][0], acc[dn][1]);
    }
    __syncthreads();
    // ---- merge the four warps' states -------------------------------------------------------------------
    constexpr int kColsPerThread = kHeads * D / kDecThreads, kThreadsPerHead = kDecThreads / kHeads;
    const int h = tid / kThreadsPerHead, c0 = (tid % kThreadsPerHead) * kColsPerThread;
    float m_all = -INFINITY, l_all = 0.f, out[kColsPerThread] = {};
    if (e_lo < e_hi) {
        m_all = fmaxf(fmaxf(st.m[0][h], st.m[1][h]), fmaxf(st.m[2][h], st.m[3][h]));   // warp 0 has key 0 of every page
#pragma unroll
        for (int w = 0; w < 4; ++w) {
            const float wgt = exp2f(st.m[w][h] - m_all);          // 0 for a warp that never saw a valid key
            l_all = fmaf(wgt, st.l[w][h], l_all);
#pragma unroll
            for (int c = 0; c < kColsPerThread; ++c) out[c] = fmaf(wgt, st.o[w][h][c0 + c], out[c]);
        }
    }
    if (!kSplit) {
        if (h >= a.group) return;                        // G = 1: the second head does not exist
        const float inv = 1.f / l_all;
        __nv_bfloat16* orow = a.o + ((size_t)s * a.hq + hbase + h) * D + c0;
#pragma unroll
        for (int c = 0; c < kColsPerThread; ++c) orow[c] = __float2bfloat16_rn(out[c] * inv);
        if (c0 == 0) a.lse[(size_t)(hbase + h) * a.batch + s] = (m_all + log2f(l_all)) * 0.6931471805599453f;
        return;
    }
    // ---- add the parts up in list order (fixed and data-independent): every CTA of the cluster its share of the columns, 32
    //      to a warp, and every warp the maxima and sums of its head, a part to a lane
    cluster_wait();                                      // the other CTAs of the cluster have started
    {                                                    // (a part without entries: zeros, under a weight of zero)
        const int v = h * D + c0, rank = small_div(v, a.share);
        const uint32_t to = map_cluster(smem_u32(dsmem) + a.gather + (blockIdx.z * a.share + v - rank * a.share) * 4, rank);
        st_cluster(to, out);
    }
    if (tid % kThreadsPerHead < a.nctas) {
        const float ml[2] = {m_all, l_all};
        st_cluster(map_cluster(smem_u32(dsmem) + a.sums + (blockIdx.z * kHeads + h) * 8, tid % kThreadsPerHead), ml);
    }
    cluster_arrive();
    cluster_wait();                                      // everything for this CTA is in its shared memory
    const int v0 = blockIdx.z * a.share, v_end = cnt > 0 ? min(v0 + a.share, kHeads * D) : 0;
    for (int v = v0 + tid; v < v_end; v += kDecThreads) {
        const int hv = v / D, col = v % D;               // (v - lane is a multiple of 32: the same head in a warp)
        const float2* sums = reinterpret_cast<const float2*>(dsmem + a.sums) + hv;        // [CTA][kHeads]
        const float* part = reinterpret_cast<const float*>(dsmem + a.gather) + (v - v0);  // [CTA][share]
        const float2 ml = lane < a.nctas ? sums[lane * kHeads] : make_float2(-INFINITY, 0.f);
        float m = ml.x;
#pragma unroll
        for (int off = 16; off > 0; off >>= 1) m = fmaxf(m, __shfl_xor_sync(0xffffffffu, m, off));
        const float w = exp2f(ml.x - m);                 // 0 for a part without entries
        float l = w * ml.y;
#pragma unroll
        for (int off = 16; off > 0; off >>= 1) l += __shfl_xor_sync(0xffffffffu, l, off);
        float o = 0.f;
#pragma unroll
        for (int i0 = 0; i0 < kMaxCtas; i0 += 4) {       // four at a time, asked for together
            if (i0 >= a.nctas) break;
            float wi[4], p[4];
#pragma unroll
            for (int i = 0; i < 4; ++i) {
                wi[i] = __shfl_sync(0xffffffffu, w, i0 + i);
                p[i] = part[min(i0 + i, a.nctas - 1) * a.share];
            }
#pragma unroll
            for (int i = 0; i < 4; ++i)
                if (i0 + i < a.nctas) o = fmaf(wi[i], p[i], o);  // (a weight of zero counts too: times an infinity it is NaN)
        }
        if (hv < a.group) {                              // (G = 1: the second head does not exist)
            a.o[((size_t)s * a.hq + hbase + hv) * D + col] = __float2bfloat16_rn(o * (1.f / l));
            if (col == 0) a.lse[(size_t)(hbase + hv) * a.batch + s] = (m + log2f(l)) * 0.6931471805599453f;
        }
    }
}

// Eq. 1 for the block of the newest token of every sequence, mapped through the page table: a warp per sequence, a lane
// per entry (each is written down from its place in the list).  A chain of launch, length, page-table entry and store:
// 3.1 us for 32 sequences of up to 64K tokens (a thread per sequence that merged three candidate streams: 10.4 us).
constexpr int kPlanDecodeWarps = 8;
__global__ void __launch_bounds__(kPlanDecodeWarps * 32) plan_decode_kernel(const int32_t* seqlens, const int32_t* page_table,
                                                                           int max_pages_per_seq, int batch, bf1_route_cfg cfg,
                                                                           bf1_decode_plan plan) {
    const int lane = threadIdx.x & 31;
    const int f = cfg.block / kPage;   // pages are 64 tokens whatever the route block width: with b = 128 a listed block
                                       // is two pages, and the newest token's own its pages up to the one that holds the token
    auto last_page = [](int n) { return n > 0 ? (n - 1) / kPage : -1; };   // logical page of the newest token
    auto bad_length = [&](int n) { return n < 0 || last_page(n) >= max_pages_per_seq; };
    pdl_wait();
    const int s = blockIdx.x * kPlanDecodeWarps + (threadIdx.x >> 5);
    if (s < batch) {
        const int n = seqlens[s], jt = last_page(n);
        int deg = 0;
        ListShape shape = {};
        if (n > 0 && !bad_length(n)) {
            shape = list_shape(cfg, jt / f);
            deg = min(list_tiles(shape, f, jt), plan.max_degree);   // (the host has checked max_degree)
        }
        for (int e = lane; e < plan.max_degree; e += 32)
            plan.page[(size_t)s * plan.max_degree + e] =
                e < deg ? page_table[(size_t)s * max_pages_per_seq + list_tile(shape, f, e)] : -1;
        if (lane == 0) {
            plan.count[s] = deg;
            plan.block[s] = jt;
        }
    }
    // The status word is WRITTEN, once: the first CTA looks at every length.
    if (blockIdx.x == 0) {
        int bad = 0;
        for (int i = threadIdx.x; i < batch; i += blockDim.x) bad |= bad_length(seqlens[i]);
        bad = __syncthreads_or(bad);
        if (threadIdx.x == 0) *plan.status = bad ? BF1_DEV_BAD_SEQLENS : 0;
    }
}

// Clusters of `ctas` CTAs of the split kernel that the GPU runs at once; asked for once per device and shape.
static int clusters_that_fit(void (*kernel)(DecodeArgs), int dev, int which, int ctas, int stages, size_t smem, int* fit) {
    static std::atomic<int> known[64][4][kMaxCtas + 1][kDecStages + 1];   // 0: not asked yet, else one more
    std::atomic<int>& k = known[dev][which][ctas][stages];
    int n = k.load(std::memory_order_relaxed) - 1;
    if (n < 0) {
        cudaLaunchConfig_t cfg = {};
        cfg.gridDim = dim3(1, 1, ctas);
        cfg.blockDim = dim3(kDecThreads);
        cfg.dynamicSmemBytes = smem;
        cudaLaunchAttribute attr = {};
        attr.id = cudaLaunchAttributeClusterDimension;
        attr.val.clusterDim.x = attr.val.clusterDim.y = 1;
        attr.val.clusterDim.z = ctas;
        cfg.attrs = &attr;
        cfg.numAttrs = 1;
        BF1_CUDA_CHECK(cudaOccupancyMaxActiveClusters(&n, kernel, &cfg));
        k.store(n + 1, std::memory_order_relaxed);
    }
    *fit = n;
    return BF1_OK;
}

// The kernels by (four heads, d = 128): which = 2 * (four heads) + (d = 128).
typedef void (*DecodeKernel)(DecodeArgs);
struct DecodeVariant {
    DecodeKernel whole, split;
    DecodeKernel brief;               // a whole list with unrounded P (four heads only)
    int page_bytes, state_bytes;      // of a page pair, of a RunState
};
template <int D, int kHeads>
static DecodeVariant decode_variant() {
    DecodeKernel brief = nullptr;
    if constexpr (kHeads == 4) brief = decode_fused_kernel<D, kHeads, false, true>;
    return {decode_fused_kernel<D, kHeads, false, false>, decode_fused_kernel<D, kHeads, true, true>, brief, 2 * kPage * D * 2,
            (int)sizeof(RunState<D, kHeads>)};
}

int check_cfg(const bf1_route_cfg* cfg);   // bf1_plan.cu

}  // namespace bf1

using namespace bf1;

extern "C" int64_t bf1_decode_workspace_bytes(int32_t batch, int32_t hq, int32_t hkv, int32_t max_degree, int32_t d) {
    if (batch < 0 || hq <= 0 || hkv <= 0 || hq % hkv != 0 || max_degree <= 0 || d <= 0) return -1;
    return 16;   // partial results stay on the chip
}

extern "C" int bf1_plan_decode(const int32_t* seqlens_dev, const int32_t* page_table_dev, int32_t max_pages_per_seq,
                               int32_t batch, const bf1_route_cfg* cfg, const bf1_decode_plan* out, void* stream) {
    if (int rc = check_cfg(cfg)) return rc;
    if (!seqlens_dev || !page_table_dev || !out || !out->count || !out->page || !out->block || !out->status)
        return fail(BF1_ERR_INVALID_ARG, "a decode-plan pointer is null");
    if (batch < 0 || max_pages_per_seq < 1 || out->max_degree < 1)
        return fail(BF1_ERR_INVALID_ARG, "bad batch, max_pages_per_seq or max_degree");
    int32_t cap = 0, need = 0;
    if (int rc = bf1_route_capacity(1, (int64_t)max_pages_per_seq * kPage, max_pages_per_seq * kPage, cfg, &cap, &need))
        return rc;
    if (out->max_degree < need)
        return fail(BF1_ERR_CAPACITY, "decode plan max_degree %d < %d needed for %d pages per sequence", out->max_degree,
                    need, max_pages_per_seq);
    if (batch == 0) return BF1_OK;
    const int ctas = (batch + kPlanDecodeWarps - 1) / kPlanDecodeWarps;
    BF1_CUDA_CHECK(launch_pdl(plan_decode_kernel, ctas, kPlanDecodeWarps * 32, 0, (cudaStream_t)stream, seqlens_dev, page_table_dev,
                              max_pages_per_seq, batch, *cfg, *out));
    return BF1_OK;
}

extern "C" int bf1_decode_fwd(const void* q, const void* k_pages, const void* v_pages, int32_t num_pages,
                              const int32_t* seqlens_dev, int32_t batch, int32_t hq, int32_t hkv, int32_t d,
                              float softmax_scale, const bf1_decode_plan* plan, void* workspace, void* o, float* lse,
                              void* stream) {
    if (!q || !k_pages || !v_pages || !seqlens_dev || !plan || !workspace || !o || !lse)
        return fail(BF1_ERR_INVALID_ARG, "a pointer is null");
    if (!plan->count || !plan->page || !plan->block || !plan->status)
        return fail(BF1_ERR_INVALID_ARG, "a decode-plan pointer is null");
    if (batch < 0 || num_pages < 0 || hq <= 0 || hkv <= 0) return fail(BF1_ERR_INVALID_ARG, "negative or zero size argument");
    if (hq % hkv != 0) return fail(BF1_ERR_INVALID_ARG, "hq %d is not a multiple of hkv %d", hq, hkv);
    const int group = hq / hkv;
    if (group != 1 && group != 2 && group != 4)
        return fail(BF1_ERR_UNSUPPORTED, "GQA group size %d: only G = 1, 2 and 4 are supported", group);
    if (d != 64 && d != 128) return fail(BF1_ERR_UNSUPPORTED, "head dimension %d: only 64 and 128 are supported", d);
    if (((uintptr_t)q | (uintptr_t)k_pages | (uintptr_t)v_pages | (uintptr_t)o | (uintptr_t)workspace) & 15)
        return fail(BF1_ERR_INVALID_ARG, "q, k_pages, v_pages, o and workspace must be 16-byte aligned");
    if (plan->max_degree < 1 || plan->max_degree > 64 || hkv * ((group + 1) / 2) > 65535 || batch > 65535)
        return fail(BF1_ERR_UNSUPPORTED, "max_degree must be <= 64; pairs of query heads and batch <= 65535");
    if (batch == 0) return BF1_OK;
    DecodeArgs a;
    a.q = (const __nv_bfloat16*)q;
    a.k_pages = (const __nv_bfloat16*)k_pages;
    a.v_pages = (const __nv_bfloat16*)v_pages;
    a.seqlens = seqlens_dev;
    a.count = plan->count;
    a.page = plan->page;
    a.block = plan->block;
    a.status = plan->status;
    a.max_degree = plan->max_degree;
    a.hq = hq;
    a.hkv = hkv;
    a.num_pages = num_pages;
    a.group = group;
    const float scale = softmax_scale > 0.f ? softmax_scale : 1.0f / sqrtf((float)d);
    a.scale_log2 = scale * 1.4426950408889634f;
    a.o = (__nv_bfloat16*)o;
    a.lse = lse;
    a.batch = batch;
    int dev = 0;
    BF1_CUDA_CHECK(cudaGetDevice(&dev));
    if (dev < 0 || dev >= 64) return fail(BF1_ERR_NO_DEVICE, "device ordinal %d out of range", dev);
    static const DecodeVariant variants[4] = {decode_variant<64, 2>(), decode_variant<128, 2>(), decode_variant<64, 4>(), decode_variant<128, 4>()};
    auto up = [](int x) { return (x + 127) / 128 * 128; };
    // shared memory of a CTA of a cluster of `ctas` whose ring has `stages` page pairs
    auto place = [&](const DecodeVariant& v, int heads, int dim, int ctas, int stages) {
        a.nctas = ctas;
        a.share = ctas == 1 ? heads * dim : (heads * dim / 32 + ctas - 1) / ctas * 32;
        a.sums = up(v.state_bytes);
        a.gather = a.sums + up(ctas * heads * 8);
        a.ring = up(a.gather + ctas * a.share * 4);
        return (size_t)a.ring + (size_t)v.page_bytes * stages;
    };
    static std::atomic<int> sm_count[64];      // 0: this device has not been set up
    int sms = sm_count[dev].load(std::memory_order_acquire);
    if (!sms) {
        for (int i = 0; i < 4; ++i) {
            const DecodeVariant& v = variants[i];
            const int most = v.state_bytes + v.page_bytes * kDecStages + 16 * 1024;    // (exchange: kMaxCtas * (32 + 128) * 4 and less)
            BF1_CUDA_CHECK(cudaFuncSetAttribute(v.whole, cudaFuncAttributeMaxDynamicSharedMemorySize, most));
            if (v.brief) BF1_CUDA_CHECK(cudaFuncSetAttribute(v.brief, cudaFuncAttributeMaxDynamicSharedMemorySize, most));
            BF1_CUDA_CHECK(cudaFuncSetAttribute(v.split, cudaFuncAttributeMaxDynamicSharedMemorySize, most));
            BF1_CUDA_CHECK(cudaFuncSetAttribute(v.split, cudaFuncAttributeNonPortableClusterSizeAllowed, 1));
        }
        BF1_CUDA_CHECK(cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev));
        sm_count[dev].store(sms, std::memory_order_release);
    }
    const int64_t lists = (int64_t)batch * hkv;
    const int heads = group == 4 ? 4 : 2, which = (group == 4 ? 2 : 0) + (d == 128);
    const DecodeVariant& variant = variants[which];
    // Enough lists to fill the GPU: one CTA walks a whole list.  With four heads, where a part costs the most to exchange, there are
    // two more cases of it (us on pages that no cache holds):
    //   d = 128, lists for half of the SMs: 96 / 128 / 144 lists of 11 pages 9.6 / 10.4 / 11.1 whole, 10.7 / 11.6 / 12.3 in parts, of
    //     4 pages 5.4 / 5.8 / 6.0 and 7.2 / 7.8 / 8.1.  Long lists lose by it while some SMs have none: 74 / 112 / 144 lists of 26
    //     pages 18.1 / 19.4 / 21.9 whole, 14.2 / 18.8 / 22.3 in parts.
    //   brief lists, walked with what rounding takes from P, as their parts would be.  A page is 0.47 us of one CTA's time; cut, a list
    //     pays for the exchange and, with many lists, for the wait for an SM.  d = 64, whole / in parts: 48 lists of 4 pages 4.2 /
    //     4.3, 80 of 4 / 6 / 8 4.4 / 4.9, 5.4 / 5.4, 6.3 / 6.1, 112 of 4 / 8 / 11 4.6 / 5.3, 6.5 / 6.7, 8.0 / 7.9, 144 of 4 / 8 / 11
    //     4.8 / 5.8, 6.8 / 7.5, 8.2 / 8.5.  Up to three pages never pay for a cluster: 8 lists of 1 / 2 / 3 2.1 / 2.5 / 2.9 whole, 3.2 /
    //     3.3 / 3.3 in parts, with d = 128 2.5 / 3.0 / 3.5 and 4.4 / 4.0 / 4.0; of 4 (d = 64, 16 lists) 3.4 and 3.3.
    const bool half = group == 4 && d == 128 && 2 * lists >= sms;
    const bool brief = group == 4 && !half && lists < sms && (plan->max_degree <= 3 || (d == 64 && plan->max_degree * (int64_t)sms <= 12 * lists));
    if (lists >= sms || half || brief) {
        a.nctas = 1;
        a.ring = up(variant.state_bytes);
        BF1_CUDA_CHECK(launch_pdl(brief ? variant.brief : variant.whole, dim3(hkv, batch), kDecThreads,
                                  (size_t)a.ring + (size_t)variant.page_bytes * kDecStages, (cudaStream_t)stream, a));
        return BF1_OK;
    }
    // A list goes to as many CTAs as still let all clusters run at once (a cluster's CTAs share a GPC, so this is less than
    // what the SMs hold: 48 lists of 11 pages over six CTAs each took 12.0 us, a second wave of clusters; with four 8.8).  Against the
    // best of eleven numbers, over 645 shapes (8 to 144 lists of 2 to 64 pages, cold and cached) this one takes 0.6 % longer on
    // average with two heads and d = 128, 6.7 % at most; with d = 64 1.1 and 7.4 %, with four heads 1.3 and 9 %.
    auto ceil_div = [](int x, int y) { return (x + y - 1) / y; };
    const int most = plan->max_degree;
    size_t smem = 0;
    for (int ctas = (int)std::min<int64_t>({kMaxCtas, most, (kDecCtasPerSm * (int64_t)sms + lists - 1) / lists}); ctas >= 1; --ctas) {
        const int pages = ceil_div(most, ctas);          // of a CTA, at most
        ctas = ceil_div(most, pages);                    // (no more than that takes)
        const int stages = std::min(pages, kDecStages);  // (a CTA with fewer pages needs that much less shared memory)
        smem = place(variant, heads, d, ctas, stages);
        if (ctas == 1) break;
        int fit = 0;
        if (int rc = clusters_that_fit(variant.split, dev, which, ctas, stages, smem, &fit)) return rc;
        if (lists <= fit) break;
    }
    BF1_CUDA_CHECK(launch_pdl_cluster(variant.split, dim3(hkv, batch, a.nctas), dim3(1, 1, a.nctas), kDecThreads, smem,
                                      (cudaStream_t)stream, a));
    return BF1_OK;
}
