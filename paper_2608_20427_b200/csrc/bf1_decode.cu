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
// decode_fused_kernel, in which a CTA serves one KV head and one pair of query heads and walks a page
// list, or several runs of it, with an online softmax over a ring of cp.async page pairs.  With enough lists
// to fill the GPU a CTA takes a whole list; with fewer, every list is cut into runs, and the CTAs of a list form a
// thread-block cluster: they send a partial (max, sum, O) of every run into the shared memory of the CTA that adds the runs
// up, in run order (each CTA of the cluster some of the columns).  Partial results in global memory behind an atomic ticket were a
// chain of store, fence, atomic and reload at the end of every call, and partial results that the first CTA fetched from the
// others' shared memory needed a second cluster barrier: 6.6, 4.6 and 4.3 us for one sequence of 32K tokens (16 query /
// 8 KV heads, d = 128).
// What a run is and which CTA walks it are two choices.  P is rounded to bf16 against the maximum of its run, and a
// key that is that maximum (P = 1) is not rounded at all: longer runs are less precise (11 pages as runs of two: relative
// error 1.99e-3 against 64 bits, page by page: 1.95e-3).  So the runs depend on the number of lists alone, as short as two
// CTAs per SM would make them, and a CTA takes as many runs as the clusters that fit the GPU leave it.  Eight sequences of
// 65 to 32768 tokens take 7.3 us for it, 6.4 with the longer runs of four CTAs each (8.0 with the ticket).
#include <algorithm>
#include <atomic>

#include "bf1_common.cuh"

namespace bf1 {

constexpr int kPage = 64;             // tokens per page = block width b
constexpr int kDecThreads = 128;
constexpr int kDecStages = 3;          // page-pair buffers per CTA
constexpr int kDecCtasPerSm = 2;       // runs a list is cut into: what this many CTAs per SM would take, one each
constexpr int kMaxRuns = 64;           // at least 1, at most a run per page
// CTAs of a cluster at most.  Above 8 a cluster may find fewer places (bf1_decode_fwd asks), but a CTA with one run instead
// of two or more wins whatever it costs: one list of 11 / 41 / 64 pages takes 5.1 / 9.4 / 11.6 us with eight CTAs, 4.0 /
// 6.7 / 8.1 with up to sixteen.
constexpr int kMaxCtas = 16;
constexpr int kMaxRunsPerCta = 8;

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
    int32_t group, pairs;             // G = hq / hkv (1, 2 or 4) and ceil(G / 2): a CTA serves one pair of query heads
    float scale_log2;
    __nv_bfloat16* o;                 // [batch, hq, d]
    float* lse;                       // [hq, batch]
    int32_t batch;
    int32_t nsplit;                   // runs a page list is cut into, at most
    int32_t nctas;                    // CTAs (a cluster) they are dealt to
    int32_t share;                    // columns (of the pair's 2 d) a CTA of the cluster adds up, a multiple of 32
    int32_t sums, gather, ring;       // shared memory: the CTA's RunStates, then from these bytes on (max, sum) [run][2] and
                                      // columns [run][share] of the list's runs, and the page ring
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
__device__ __forceinline__ void st_cluster(uint32_t addr, float v) {
    asm volatile("st.shared::cluster.f32 [%0], %1;" ::"r"(addr), "f"(v) : "memory");
}
__device__ __forceinline__ void st_cluster_v2(uint32_t addr, float x, float y) {
    asm volatile("st.shared::cluster.v2.f32 [%0], {%1, %2};" ::"r"(addr), "f"(x), "f"(y) : "memory");
}
// x / y for small whole numbers (below 2^20: half a step from a whole quotient is more than the division's error)
__device__ __forceinline__ int small_div(int x, int y) { return (int)__fdividef((float)x + 0.5f, (float)y); }

// One CTA per (sequence, KV head, pair of query heads[, share of the list's runs]).  Pages stream in through a
// kDecStages-deep cp.async ring with ONE block-wide synchronisation per page; inside a page each of the
// four warps owns 16 keys and keeps its own online-softmax state (max, sum, O) for both grouped heads,
// merged at the end of the run.  The arithmetic uses warp-level mma (m16n8k16: the two heads are rows 0 and 1
// of the 16-row operand, the rest is zero): the work is memory-bound, but as scalar FMAs it was a chain
// of 1500 dependent instructions and five synchronisations per page, which is what bounded the kernel.
template <int D>
struct RunState {                                       // the four warps' states at the end of a run
    float o[4][2][D + 8], m[4][2], l[4][2];              // (rows 8 banks apart)
};
template <int D, bool kSplit>
__global__ void __launch_bounds__(kDecThreads, D == 64 ? 4 : 2) decode_fused_kernel(const DecodeArgs a) {
    constexpr int kRowBytes = D * 2;
    constexpr int kVecPerRow = D / 8;                   // 16-byte chunks per row
    constexpr int kVecPerThread = kPage * kVecPerRow / kDecThreads;
    constexpr int kPageBytes = kPage * D * 2;
    // [stage][K | V][64 rows][D bf16]; the 16-byte chunks of every row are XOR-swizzled with (row & 7), which
    // keeps both the B-fragment loads of K (8 rows, same chunk) and the ldmatrix rows of V conflict-free
    extern __shared__ __align__(128) uint8_t dsmem[];
    RunState<D>* sRun = reinterpret_cast<RunState<D>*>(dsmem);   // of this CTA's runs, in front of the ring
    __shared__ int sPages[64];                          // the sequence's page list (max_degree <= 64)

    const int kvp = blockIdx.x, s = blockIdx.y, tid = threadIdx.x;
    const int kvh = kvp / a.pairs, hbase = kvh * a.group + (kvp % a.pairs) * 2;   // first query head of this CTA's pair
    const int nheads = min(2, a.group - (kvp % a.pairs) * 2);                      // 1 when G = 1
    const int warp = tid >> 5, lane = tid & 31, gid = lane >> 2, tig = lane & 3;
    // The page list is fetched together with the plan's count and the length (independent loads in flight at
    // once), not after them: at small batch the kernel is one chain of dependent memory round trips.
    pdl_wait();
    if (tid < a.max_degree) sPages[tid] = a.page[(size_t)s * a.max_degree + tid];
    int cnt = max(min(a.count[s], a.max_degree), 0);
    const int n = a.seqlens[s];
    const int j = (n - 1) / kPage;
    if (cnt > 0 && j != a.block[s]) {    // the plan belongs to another route epoch
        if (tid == 0 && kvp == 0) atomicOr(a.status, BF1_DEV_BAD_ROUTE);
        cnt = 0;
    }
    // Nothing to do.  A CTA of a cluster stays all the same: whatever it reads here, the others may store to its shared memory.
    if (!kSplit && cnt == 0) return;
    const int tail = n - j * kPage;   // valid tokens of the self page (the last list entry)
    __syncthreads();                  // sPages is complete
    const int* pages = sPages;
    // the part of the list this CTA walks: all of it as one run, or its share of the list's runs of `per` entries (the later CTAs
    // get one more where they do not come out even: the last run may be shorter)
    const int per = kSplit ? max(small_div(cnt + a.nsplit - 1, a.nsplit), 1) : cnt;
    const int runs = kSplit ? small_div(cnt + per - 1, per) : 1;
    const int run0 = kSplit ? small_div(blockIdx.z * runs, a.nctas) : 0;
    const int e_lo = run0 * per, e_hi = kSplit ? min(cnt, small_div((blockIdx.z + 1) * runs, a.nctas) * per) : cnt;   // (may be empty)
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
#pragma unroll
    for (int i = 0; i < kDecStages - 1; ++i) {
        if (e_lo + i < e_hi) issue_page(e_lo + i, i);
        cp_async_commit();                               // possibly empty: keeps the group count uniform
    }
    if (kSplit) cluster_arrive_relaxed();                        // (waited for in front of the first store to another CTA)
    // A fragments of Q: rows 0 and 1 of the 16-row operand are the two grouped heads, the rest zero
    uint32_t qa[D / 16][2];
    {
        const uint32_t* qrow = reinterpret_cast<const uint32_t*>(a.q + ((size_t)s * a.hq + hbase + (gid < nheads ? gid : 0)) * D);
#pragma unroll
        for (int kk = 0; kk < D / 16; ++kk) {
            qa[kk][0] = gid < nheads ? qrow[kk * 8 + tig] : 0u;          // columns kk*16 + 2*tig, +1
            qa[kk][1] = gid < nheads ? qrow[kk * 8 + tig + 4] : 0u;      // columns kk*16 + 8 + 2*tig, +1
        }
    }
    float m_run = -INFINITY, l_run = 0.f;                // per lane: head gid (lanes with gid >= 2 carry dummies)
    float acc[D / 8][4];
#pragma unroll
    for (int dn = 0; dn < D / 8; ++dn) acc[dn][0] = acc[dn][1] = acc[dn][2] = acc[dn][3] = 0.f;
    const int key0 = warp * 16;                          // this warp's 16 keys of every page
    auto leave_sums = [&](RunState<D>& st) {             // this warp's state of a run: what is ready first ...
        if (gid < 2 && tig == 0) { st.m[warp][gid] = m_run; st.l[warp][gid] = l_run; }
    };
    auto leave_o = [&](RunState<D>& st) {                // ... and what the MMAs add up
        if (gid >= 2) return;
#pragma unroll
        for (int dn = 0; dn < D / 8; ++dn)
            *reinterpret_cast<float2*>(&st.o[warp][gid][dn * 8 + 2 * tig]) = make_float2(acc[dn][0], acc[dn][1]);
    };
    int run = 0, run_end = e_lo + per;                   // the run at hand (of this CTA's), and the entry behind it
    // Where this thread's columns of a run go: to the CTA of the cluster that adds them up.
    constexpr int kColsPerThread = D / 64;
    const int c0 = (tid & 63) * kColsPerThread;
    uint32_t to_gather = 0, to_sums = 0;
    if (kSplit) {
        const int v = (tid >> 6) * D + c0, rank = small_div(v, a.share);
        to_gather = map_cluster(smem_u32(dsmem) + a.gather + (run0 * a.share + v - rank * a.share) * 4, rank);
        to_sums = map_cluster(smem_u32(dsmem) + a.sums + (run0 * 2 + (tid >> 6)) * 8, min(tid & 63, a.nctas - 1));
    }

    for (int e = e_lo; e < e_hi; ++e) {
        cp_async_wait<kDecStages - 2>();                 // page e has landed (for this thread's copies)
        __syncthreads();                                 // ... for everybody's; and page e-1 is no longer read
        if (e + kDecStages - 1 < e_hi) issue_page(e + kDecStages - 1, (e - e_lo + kDecStages - 1) % kDecStages);
        cp_async_commit();
        const int valid = (e == cnt - 1) ? tail : kPage;
        const uint32_t kb = ring + ((e - e_lo) % kDecStages) * 2 * kPageBytes, vb = kb + kPageBytes;
        const bool keys = key0 < valid;                  // warp-uniform: some of this warp's keys exist
        uint32_t pa0 = 0, pa2 = 0;
        float alpha = 1.f;
        if (keys) {
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
            // lane (gid < 2, tig) holds head gid's scores of keys key0 + nt*8 + 2*tig, +1
            float sv[4];
            float mx = -INFINITY;
#pragma unroll
            for (int i = 0; i < 4; ++i) {
                const int key = key0 + (i >> 1) * 8 + 2 * tig + (i & 1);
                sv[i] = (gid < 2) ? ((key < valid) ? sc[i >> 1][i & 1] * a.scale_log2 : -INFINITY) : 0.f;
                mx = fmaxf(mx, sv[i]);
            }
            mx = fmaxf(mx, __shfl_xor_sync(0xffffffffu, mx, 1));
            mx = fmaxf(mx, __shfl_xor_sync(0xffffffffu, mx, 2));       // finite: key0 < valid
            const float m_new = fmaxf(m_run, mx);
            alpha = exp2f(m_run - m_new);                   // 0 on the warp's first page
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
            // P as the A operand of the second mma: the C layout of the scores is the A layout of the next k-step
            pa0 = gid < 2 ? pack_bf16x2(pv[0], pv[1]) : 0u;   // keys 2*tig, +1
            pa2 = gid < 2 ? pack_bf16x2(pv[2], pv[3]) : 0u;   // keys 8 + 2*tig, +1
        }
        if (kSplit && e == run_end) {                    // a new run: the MMAs of the one before have had the time of these scores
            leave_o(sRun[run++]);
            run_end += per;
#pragma unroll
            for (int dn = 0; dn < D / 8; ++dn) acc[dn][0] = acc[dn][1] = 0.f;      // (the other rows of the operand stay zero)
        }
        if (keys) {
            // ---- O = alpha * O + P V: D / 8 n-tiles of 8 columns, V fragments by ldmatrix.trans ---------
            const int lrow = key0 + (lane & 7) + ((lane >> 3) & 1) * 8;      // ldmatrix: lane supplies row (lane % 8) of matrix lane / 8
            const uint32_t vrow = vb + lrow * kRowBytes;
#pragma unroll
            for (int dn = 0; dn < D / 8; dn += 2) {
                acc[dn][0] *= alpha;
                acc[dn][1] *= alpha;
                acc[dn + 1][0] *= alpha;
                acc[dn + 1][1] *= alpha;
                uint32_t r0, r1, r2, r3;   // matrices: (keys 0-7, dn), (keys 8-15, dn), (keys 0-7, dn+1), (keys 8-15, dn+1)
                ldmatrix_x4_trans(vrow + (((dn + (lane >> 4)) ^ (lrow & 7)) << 4), r0, r1, r2, r3);
                mma_16816(acc[dn], pa0, 0u, pa2, 0u, r0, r1);
                mma_16816(acc[dn + 1], pa0, 0u, pa2, 0u, r2, r3);
            }
        }
        if (kSplit && e + 1 == run_end) {                // the run ends
            leave_sums(sRun[run]);
            m_run = -INFINITY;
            l_run = 0.f;
        }
    }
    cp_async_wait<0>();
    if (e_lo < e_hi) {
        if (!kSplit || e_hi != run_end) leave_sums(sRun[run]);   // (a shorter last run)
        leave_o(sRun[run++]);
    }
    __syncthreads();
    // ---- merge the four warps' states of every run ------------------------------------------------------
    if (kSplit) cluster_wait();                          // the other CTAs of the cluster have started
    float m_all = -INFINITY, l_all = 0.f, out[kColsPerThread];
#pragma unroll 2
    for (int i = 0; i < run; ++i) {
        const RunState<D>& st = sRun[i];
        const int h = tid >> 6;
        m_all = fmaxf(fmaxf(st.m[0][h], st.m[1][h]), fmaxf(st.m[2][h], st.m[3][h]));   // warp 0 has key 0 of every page
        float wgt[4];
        l_all = 0.f;
#pragma unroll
        for (int w = 0; w < 4; ++w) {
            wgt[w] = exp2f(st.m[w][h] - m_all);          // 0 for a warp that never saw a valid key
            l_all = fmaf(wgt[w], st.l[w][h], l_all);
        }
#pragma unroll
        for (int c = 0; c < kColsPerThread; ++c) {
            out[c] = 0.f;
#pragma unroll
            for (int w = 0; w < 4; ++w) out[c] = fmaf(wgt[w], st.o[w][h][c0 + c], out[c]);
            if (kSplit) st_cluster(to_gather + (i * a.share + c) * 4, out[c]);
        }
        if (kSplit && (tid & 63) < a.nctas) st_cluster_v2(to_sums + i * 16, m_all, l_all);
    }
    if (!kSplit) {
        const int h = tid >> 6;
        if (h >= nheads) return;                         // G = 1: the second head of the pair does not exist
        const float inv = 1.f / l_all;
        __nv_bfloat16* orow = a.o + ((size_t)s * a.hq + hbase + h) * D + c0;
#pragma unroll
        for (int c = 0; c < kColsPerThread; ++c) orow[c] = __float2bfloat16_rn(out[c] * inv);
        if ((tid & 63) == 0) a.lse[(size_t)(hbase + h) * a.batch + s] = (m_all + log2f(l_all)) * 0.6931471805599453f;
        return;
    }
    // ---- add the runs up in run order (fixed and data-independent): every CTA of the cluster its share of the columns, 32 to
    //      a warp, and every warp the maxima and sums of its head, a run (and the run 32 further) to a lane
    cluster_arrive();
    cluster_wait();                                      // everything for this CTA is in its shared memory
    const int v0 = blockIdx.z * a.share, v_end = runs > 0 ? min(v0 + a.share, 2 * D) : 0;
    for (int v = v0 + tid; v < v_end; v += kDecThreads) {
        const int h = v / D, col = v % D;                // (v - lane is a multiple of 32: the same head in a warp)
        const float2* sums = reinterpret_cast<const float2*>(dsmem + a.sums) + h;         // [run][2]
        const float* part = reinterpret_cast<const float*>(dsmem + a.gather) + (v - v0);  // [run][share]
        float2 ml[2];
#pragma unroll
        for (int k = 0; k < 2; ++k) ml[k] = lane + 32 * k < runs ? sums[(lane + 32 * k) * 2] : make_float2(-INFINITY, 0.f);
        float m = fmaxf(ml[0].x, ml[1].x);
#pragma unroll
        for (int off = 16; off > 0; off >>= 1) m = fmaxf(m, __shfl_xor_sync(0xffffffffu, m, off));
        float w[2] = {0.f, 0.f}, sum[2] = {0.f, 0.f};
#pragma unroll
        for (int k = 0; k < 2; ++k) {
            if (32 * k >= runs) break;
            if (lane + 32 * k < runs) w[k] = exp2f(ml[k].x - m);
            sum[k] = __fmul_rn(w[k], ml[k].y);
#pragma unroll
            for (int off = 16; off > 0; off >>= 1) sum[k] += __shfl_xor_sync(0xffffffffu, sum[k], off);
        }
        const float l = sum[0] + sum[1];
        float o = 0.f;
        for (int i0 = 0; i0 < runs; i0 += 8) {           // eight at a time, asked for together
            float wi[8], p[8];
#pragma unroll
            for (int i = 0; i < 8; ++i) {
                wi[i] = __shfl_sync(0xffffffffu, i0 & 32 ? w[1] : w[0], (i0 + i) & 31);
                p[i] = part[min(i0 + i, runs - 1) * a.share];
            }
#pragma unroll
            for (int i = 0; i < 8; ++i)
                if (i0 + i < runs) o = fmaf(wi[i], p[i], o);
        }
        if (h < nheads) {                                // (G = 1: the second head of the pair does not exist)
            a.o[((size_t)s * a.hq + hbase + h) * D + col] = __float2bfloat16_rn(o * (1.f / l));
            if (col == 0) a.lse[(size_t)(hbase + h) * a.batch + s] = (m + log2f(l)) * 0.6931471805599453f;
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
static int clusters_that_fit(void (*kernel)(DecodeArgs), int dev, int wide, int ctas, int stages, int slots, size_t smem, int* fit) {
    static std::atomic<int> known[64][2][kMaxCtas + 1][kDecStages + 1][kMaxRunsPerCta + 1];   // 0: not asked yet, else one more
    std::atomic<int>& k = known[dev][wide][ctas][stages][slots];
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
    const int group = hq / hkv, pairs = (group + 1) / 2;
    if (group != 1 && group != 2 && group != 4)
        return fail(BF1_ERR_UNSUPPORTED, "GQA group size %d: only G = 1, 2 and 4 are supported", group);
    if (d != 64 && d != 128) return fail(BF1_ERR_UNSUPPORTED, "head dimension %d: only 64 and 128 are supported", d);
    if (((uintptr_t)q | (uintptr_t)k_pages | (uintptr_t)v_pages | (uintptr_t)o | (uintptr_t)workspace) & 15)
        return fail(BF1_ERR_INVALID_ARG, "q, k_pages, v_pages, o and workspace must be 16-byte aligned");
    if (plan->max_degree < 1 || plan->max_degree > 64 || hkv * pairs > 65535 || batch > 65535)
        return fail(BF1_ERR_UNSUPPORTED, "max_degree must be <= 64; hkv and batch must fit the grid (<= 65535)");
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
    a.pairs = pairs;
    const float scale = softmax_scale > 0.f ? softmax_scale : 1.0f / sqrtf((float)d);
    a.scale_log2 = scale * 1.4426950408889634f;
    a.o = (__nv_bfloat16*)o;
    a.lse = lse;
    a.batch = batch;
    int dev = 0;
    BF1_CUDA_CHECK(cudaGetDevice(&dev));
    if (dev < 0 || dev >= 64) return fail(BF1_ERR_NO_DEVICE, "device ordinal %d out of range", dev);
    constexpr int kSmem128 = kDecStages * 2 * 64 * 128 * 2, kSmem64 = kDecStages * 2 * 64 * 64 * 2;
    constexpr int kState128 = sizeof(RunState<128>), kState64 = sizeof(RunState<64>);
    auto up = [](int x) { return (x + 127) / 128 * 128; };
    static std::atomic<int> sm_count[64];      // 0: this device has not been set up
    int sms = sm_count[dev].load(std::memory_order_acquire);
    if (!sms) {
        BF1_CUDA_CHECK(cudaFuncSetAttribute(decode_fused_kernel<128, false>, cudaFuncAttributeMaxDynamicSharedMemorySize, up(kState128) + kSmem128));
        BF1_CUDA_CHECK(cudaFuncSetAttribute(decode_fused_kernel<128, true>, cudaFuncAttributeMaxDynamicSharedMemorySize, 100 * 1024 + kSmem128));
        BF1_CUDA_CHECK(cudaFuncSetAttribute(decode_fused_kernel<64, false>, cudaFuncAttributeMaxDynamicSharedMemorySize, up(kState64) + kSmem64));
        BF1_CUDA_CHECK(cudaFuncSetAttribute(decode_fused_kernel<64, true>, cudaFuncAttributeMaxDynamicSharedMemorySize, 100 * 1024 + kSmem64));
        BF1_CUDA_CHECK(cudaFuncSetAttribute(decode_fused_kernel<128, true>, cudaFuncAttributeNonPortableClusterSizeAllowed, 1));
        BF1_CUDA_CHECK(cudaFuncSetAttribute(decode_fused_kernel<64, true>, cudaFuncAttributeNonPortableClusterSizeAllowed, 1));
        BF1_CUDA_CHECK(cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev));
        sm_count[dev].store(sms, std::memory_order_release);
    }
    const int64_t lists = (int64_t)batch * hkv * pairs;
    const int page_smem = d == 128 ? kSmem128 / kDecStages : kSmem64 / kDecStages, state = d == 128 ? kState128 : kState64;
    if (lists >= sms) {
        // enough lists to fill the GPU: one CTA walks a whole list
        a.nsplit = a.nctas = 1;
        a.ring = up(state);
        BF1_CUDA_CHECK(launch_pdl(d == 128 ? decode_fused_kernel<128, false> : decode_fused_kernel<64, false>,
                                  dim3(hkv * pairs, batch), kDecThreads, (size_t)a.ring + (size_t)page_smem * kDecStages,
                                  (cudaStream_t)stream, a));
        return BF1_OK;
    }
    a.nsplit = (int)std::min<int64_t>({(kDecCtasPerSm * (int64_t)sms + lists - 1) / lists, plan->max_degree, kMaxRuns});
    // The runs of a list go to as many CTAs as still let all clusters run at once (a cluster's CTAs share a GPC, so this is
    // less than what the SMs hold: 48 lists of 11 pages over six CTAs each took 12.0 us, a second wave of clusters; with four
    // 8.8).  Over 270 pairs of lists (1 to 147) and lengths (5 to 64 pages) this is the fastest number of CTAs or
    // within 4.3 % of it, 0.05 % on average.
    // A list has at most nsplit runs; one of max_degree entries has `most` of `per` pages, shorter ones have shorter runs.
    const int per = (plan->max_degree + a.nsplit - 1) / a.nsplit, most = (plan->max_degree + per - 1) / per;
    auto ceil_div = [](int x, int y) { return (x + y - 1) / y; };
    auto kernel = d == 128 ? decode_fused_kernel<128, true> : decode_fused_kernel<64, true>;
    size_t smem = 0;
    for (int ctas = std::min(kMaxCtas, most); ctas >= 1; --ctas) {
        ctas = ceil_div(most, ceil_div(most, ctas));     // (none of them idle)
        const int slots = ceil_div(a.nsplit, ctas);      // runs of a CTA, at most (the first choice always has few enough)
        if (slots > kMaxRunsPerCta) break;
        // a CTA with fewer pages than the ring has stages needs that much less shared memory
        const int stages = std::min(std::max(slots * (per - 1), ceil_div(most, ctas) * per), kDecStages);
        a.nctas = ctas;
        a.share = ceil_div(2 * d / 32, ctas) * 32;
        a.sums = up(slots * state);
        a.gather = a.sums + up(slots * ctas * 2 * 8);
        a.ring = a.gather + slots * ctas * a.share * 4;
        smem = (size_t)a.ring + (size_t)page_smem * stages;
        if (ctas == 1) break;
        int fit = 0;
        if (int rc = clusters_that_fit(kernel, dev, d == 128, ctas, stages, slots, smem, &fit)) return rc;
        if (lists <= fit) break;
    }
    BF1_CUDA_CHECK(launch_pdl_cluster(kernel, dim3(hkv * pairs, batch, a.nctas), dim3(1, 1, a.nctas), kDecThreads, smem,
                                      (cudaStream_t)stream, a));
    return BF1_OK;
}
