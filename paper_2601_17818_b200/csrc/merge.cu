// Cluster merge (Eq. 6 / second half of Algorithm 3): the tokens of a cluster that were not kept as elites are
// averaged into one representative row.
//
// Two kernels on one stream:
//   merge_plan_kernel   one CTA per sample: lays every cluster's non-elite tokens out contiguously in ascending token order,
//                       clusters in ascending label order.  Up to 256 to 1024 clusters, by the sample's length, by one stable
//                       counting pass over dense cluster numbers; more by a stable radix sort of the labels in shared memory.
//   merge_rows_kernel   one CTA per (merged row, sample, 1024-byte slice of the hidden row): its four warps stream
//                       the members' row slices with 128-bit loads (member r goes to warp r mod 4) and the four
//                       fp32 partial sums are added in warp order, a fixed order (bit-reproducible).  Only rows
//                       that are averaged are read.
#include <cuda_bf16.h>

#include "gram.cuh"
#include "internal.cuh"

namespace vitcop {
namespace {

constexpr int kPlanThreads = 1024;
constexpr int kPlanWarps = kPlanThreads / 32;
constexpr int kRowsThreads = 128;
constexpr int kPlanItems = VITCOP_MAX_VISUAL_TOKENS / kPlanThreads;   // rows of 32 entries a warp walks at most
constexpr int kDigitBits = 7, kDigits = 1 << kDigitBits;
static_assert(kDigits * kPlanWarps == 4 * kPlanThreads, "four counters per thread in the scan");
// The counter of (digit d, warp w) sits at w * kCntStride + d: the leaders of a row (one warp, distinct digits) and
// the four counters a thread scans (one digit, consecutive warps) both spread over the banks.
constexpr int kCntStride = kDigits + 2;
constexpr int kCntEntries = kPlanWarps * kCntStride;

// What merge_rows_kernel needs to know of a merged row; count 0 past the last one.  The headers come in the order in which the
// rows are to be worked on: those with many members first, as one of them takes several times as long as the others.
struct __align__(16) MergeHeader {
    int32_t count, start;                                 // its run in the member list
    int32_t row, pad;                                     // the merged row
    uint16_t first[4][4];                                 // member r < 16 at [r % 4][r / 4]
};
constexpr int kManyMembers = 32;
__host__ __device__ constexpr int member_stride(int Nv_cap) { return (Nv_cap + 7) & ~7; }     // a sample's member list
static_assert(sizeof(MergeHeader) == 48, "three 16-byte words");

// Every array of the planner is walked the same way: warp w owns the entries [w * 32 E, (w + 1) * 32 E), E =
// ceil(count / 1024), and takes them 32 at a time, lane by lane (coalesced, no bank conflicts, and entry order is
// (warp, row, lane) order, so that ballots and one scan over the 32 warp totals give stable positions).  The walks are
// rolled loops on purpose: the kernel runs once per call on a handful of SMs, so every instruction it executes is
// fetched cold, and a loop body fetched once beats sixteen unrolled copies.

// One walk of a warp over its items with a cursor per (digit, warp) in `cnt`: every item receives the cursor of its
// digit plus the number of items of the same digit in front of it in its row, and the cursor moves past the row's
// items.  With the cursors at zero the walk counts (dst null); with the cursors at their scanned values it writes the
// items to their sorted positions in dst.
__device__ __forceinline__ void digit_walk(const uint32_t* src, uint32_t* dst, int E, int m, int shift, uint16_t* cnt) {
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
#pragma unroll 1
    for (int e = 0; e < E; ++e) {
        const int p = (warp * E + e) * 32 + lane;
        const bool valid = p < m;
        const uint32_t item = valid ? src[p] : 0u;
        const uint32_t d = (item >> shift) & (kDigits - 1);
        // the lanes of the row that hold the same digit: one ballot per bit
        const uint32_t vb = __ballot_sync(0xffffffffu, valid);
        uint32_t peers = valid ? vb : ~vb;
#pragma unroll
        for (int k = 0; k < kDigitBits; ++k) {
            const uint32_t bk = __ballot_sync(0xffffffffu, d >> k & 1u);
            peers &= (d >> k & 1u) ? bk : ~bk;
        }
        const int leader = __ffs(peers) - 1;
        uint32_t cur = 0;
        if (valid && lane == leader) {
            cur = cnt[warp * kCntStride + d];
            cnt[warp * kCntStride + d] = (uint16_t)(cur + __popc(peers));
        }
        cur = __shfl_sync(0xffffffffu, cur, leader);
        if (dst && valid) dst[cur + __popc(peers & ((1u << lane) - 1u))] = item;
        __syncwarp();                                      // the next row's leaders may be other lanes
    }
}

// Stable sort of m items (label << 16 | token index, in ascending token order on entry) by label: least significant
// digit first, seven bits at a time, from one buffer to the other and back.  Returns the buffer that holds the result.
// `cnt`: shared uint16_t [kCntEntries]; label_bits: bits of the largest label.
__device__ uint32_t* sort_by_label(uint32_t* a, uint32_t* b, int m, int label_bits, uint16_t* cnt, uint32_t* warp_sums) {
    const int t = threadIdx.x;
    const int E = (m + kPlanThreads - 1) / kPlanThreads;
    // this thread's four counters in scan order (digit by digit, inside a digit warp by warp)
    uint16_t* mine = cnt + (t % (kPlanWarps / 4)) * 4 * kCntStride + t / (kPlanWarps / 4);
#pragma unroll 1
    for (int shift = 16; shift < 16 + label_bits; shift += kDigitBits) {
        for (int c = t; c < kCntEntries; c += kPlanThreads) cnt[c] = 0;
        __syncthreads();
        digit_walk(a, nullptr, E, m, shift, cnt);
        __syncthreads();
        const uint32_t c0 = mine[0], c1 = mine[kCntStride], c2 = mine[2 * kCntStride], c3 = mine[3 * kCntStride];
        uint32_t total;
        const uint32_t b0 = block_exclusive_sum(c0 + c1 + c2 + c3, warp_sums, total);
        mine[0] = (uint16_t)b0;
        mine[kCntStride] = (uint16_t)(b0 + c0);
        mine[2 * kCntStride] = (uint16_t)(b0 + c0 + c1);
        mine[3 * kCntStride] = (uint16_t)(b0 + c0 + c1 + c2);
        __syncthreads();
        digit_walk(a, b, E, m, shift, cnt);
        __syncthreads();
        uint32_t* s = a;
        a = b;
        b = s;
    }
    return a;
}

// The plan by one stable counting pass: labels get dense numbers (presence flags, one scan), every warp ranks its tokens inside
// their cluster (one match per 32 tokens and a counter per (warp, cluster)), one scan over the counters turns ranks into
// positions.  Taken up to count_seg(E) clusters that have non-elite tokens: 5 % of the tokens that E stands for, rounded up to
// what divides the threads.  E: rows of 32 tokens per warp.  lab, take: this thread's tokens (labels; bit e: not an elite).
// smem: flags / numbers uint16 [n rounded up to 8], counters uint16 [32][clusters + 2].
__host__ __device__ constexpr int count_seg(int E) { return E <= 4 ? 256 : E <= 8 ? 512 : 1024; }
__host__ __device__ constexpr size_t plan_count_bytes(int Nv_cap, int E) {
    return ((size_t)((Nv_cap + 7) & ~7) + (size_t)kPlanWarps * (count_seg(E) + 2)) * sizeof(uint16_t);
}
__device__ __forceinline__ void zero_counters(uint16_t* cnt, int clusters) {
    for (int i = threadIdx.x; i < kPlanWarps * (clusters + 2) / 2; i += kPlanThreads) reinterpret_cast<uint32_t*>(cnt)[i] = 0u;
}
// The first sixteen of a run's members (the low halves of the entries) into its header.
template <typename Entry>
__device__ __forceinline__ void store_first(const Entry* run, int count, MergeHeader* h) {
    uint32_t w[8];
#pragma unroll
    for (int g = 0; g < 4; ++g)
#pragma unroll
        for (int k = 0; k < 2; ++k) {
            const int r = 8 * k + g;                       // first[g][2 k], first[g][2 k + 1]: members r and r + 4
            w[2 * g + k] = (r < count ? (uint32_t)run[r] & 0xFFFFu : 0u) | (r + 4 < count ? (uint32_t)run[r + 4] << 16 : 0u);
        }
    uint4* const to = reinterpret_cast<uint4*>(h->first);
    to[0] = make_uint4(w[0], w[1], w[2], w[3]);
    to[1] = make_uint4(w[4], w[5], w[6], w[7]);
}
// Behind the dense numbers, for up to SEG clusters; the counters are zero.
template <int E, int SEG>
__device__ __forceinline__ void plan_positions(const uint32_t (&lab)[E], uint32_t take, int n, int n_seg, int Mcap,
                                               int32_t* merged_count, uint16_t* members, MergeHeader* headers,
                                               uint16_t* id_of, uint16_t* cnt, uint16_t* seg_start, uint16_t* seg_slot,
                                               uint32_t* warp_sums) {
    constexpr int kStride = SEG + 2, kPer = kPlanThreads / SEG, kOf = kPlanWarps / kPer;     // threads per cluster, counters of one
    static_assert(kPer * SEG == kPlanThreads && kPer * kOf == kPlanWarps && kPer <= 32, "threads and counters of a cluster");
    const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
    const uint32_t lt = (1u << lane) - 1u;
    const int rows = (n + kPlanThreads - 1) / kPlanThreads;
    const int bits = n_seg > 1 ? 32 - __clz(n_seg - 1) : 0;
    uint32_t at[E];                                        // cluster << 16 | rank among the warp's tokens of the cluster
#pragma unroll
    for (int e = 0; e < E; ++e) {
        at[e] = 0;
        if (e < rows) {                                    // (uniform)
            const bool mine = (take >> e & 1u) != 0;
            const uint32_t c = mine ? id_of[lab[e]] : 0u;
            // the lanes of the same cluster: a ballot per bit of its number (a match takes as many steps as the row has different
            // clusters: 16384 tokens in 820 clusters 50.4 us, so 45.7)
            const uint32_t all = __ballot_sync(0xffffffffu, mine);
            uint32_t peers = mine ? all : 0u;
#pragma unroll 1
            for (int k = 0; k < bits; ++k) {
                const uint32_t bk = __ballot_sync(0xffffffffu, c >> k & 1u);
                peers &= (c >> k & 1u) ? bk : ~bk;
            }
            uint32_t before = 0;
            if (mine) before = cnt[warp * kStride + c];
            __syncwarp();
            if (mine && lane == __ffs(peers) - 1) cnt[warp * kStride + c] = (uint16_t)(before + __popc(peers));
            __syncwarp();
            at[e] = (c << 16) | (before + __popc(peers & lt));
        }
    }
    __syncthreads();
    uint32_t m;
    {
        // counters in (cluster, warp) order -> positions
        const int c = tid / kPer, w0 = tid % kPer * kOf;
        uint32_t sum = 0;
#pragma unroll
        for (int q = 0; q < kOf; ++q) sum += cnt[(w0 + q) * kStride + c];
        uint32_t pos = block_exclusive_sum(sum, warp_sums, m);
        const uint32_t start = __shfl_sync(0xffffffffu, pos, lane & ~(kPer - 1));
        const uint32_t end = __shfl_sync(0xffffffffu, pos + sum, lane | (kPer - 1));
        const bool row = tid % kPer == 0 && c < n_seg && c < Mcap, many = row && end - start >= (uint32_t)kManyMembers;
        uint32_t totals;
        const uint32_t before = block_exclusive_sum((row ? 1u : 0u) | (many ? 0x10000u : 0u), warp_sums, totals);
        if (row) {
            const uint32_t many_before = before >> 16, few_before = (before & 0xFFFFu) - many_before;
            const uint32_t slot = many ? many_before : (totals >> 16) + few_before;
            seg_slot[c] = (uint16_t)slot;
            seg_start[c] = (uint16_t)start;
            *reinterpret_cast<int4*>(headers + slot) = make_int4((int)(end - start), (int)start, c, 0);
            merged_count[c] = (int32_t)(end - start);
        }
#pragma unroll
        for (int q = 0; q < kOf; ++q) {
            const uint32_t v = cnt[(w0 + q) * kStride + c];
            cnt[(w0 + q) * kStride + c] = (uint16_t)pos;
            pos += v;
        }
    }
    __syncthreads();
    // the member list is put together in shared memory and leaves in words of eight: tokens of a warp go to as many places as they
    // have clusters (16384 tokens in 820 clusters: 45.7 us with scattered two-byte stores, 27.3 so; 4608 in 231: 18.7, 14.6)
    uint16_t* const sorted = id_of;                        // (the numbers have been read)
#pragma unroll
    for (int e = 0; e < E; ++e)
        if (take >> e & 1u)
            sorted[cnt[warp * kStride + (at[e] >> 16)] + (at[e] & 0xFFFFu)] = (uint16_t)((warp * rows + e) * 32 + lane);
    __syncthreads();
    for (int q = tid; q < ((int)m + 7) / 8; q += kPlanThreads) reinterpret_cast<uint4*>(members)[q] = reinterpret_cast<const uint4*>(sorted)[q];
    if (tid < min(n_seg, Mcap)) {
        const int start = seg_start[tid], end = tid + 1 < min(n_seg, Mcap) ? seg_start[tid + 1] : start + 16;
        store_first(sorted + start, min(end, (int)m) - start, headers + seg_slot[tid]);
    }
    for (int c = n_seg + tid; c < Mcap; c += kPlanThreads) headers[c].count = 0;
}
// Returns false, nothing written, when there are more clusters than that.
template <int E>
__device__ __forceinline__ bool plan_by_count(const uint32_t (&lab)[E], uint32_t take, int n, int Mcap,
                                              int32_t* merged_label, int32_t* merged_count, int32_t* n_merged_b,
                                              uint16_t* members, MergeHeader* headers, uint16_t* smem, uint32_t* warp_sums) {
    constexpr int kSeg = count_seg(E), kNarrow = 256;
    __shared__ uint16_t seg_start[kSeg], seg_slot[kSeg];   // slot: place of the cluster's header
    const int tid = threadIdx.x;
    const int n_al = (n + 7) & ~7;
    uint16_t* const id_of = smem;                          // by label: 1 = present, then its dense number
    uint16_t* const cnt = smem + n_al;
    for (int i = tid; i < n_al / 8; i += kPlanThreads) reinterpret_cast<uint4*>(id_of)[i] = make_uint4(0u, 0u, 0u, 0u);
    zero_counters(cnt, kNarrow);
    __syncthreads();
#pragma unroll
    for (int e = 0; e < E; ++e)
        if (take >> e & 1u) id_of[lab[e]] = 1;
    __syncthreads();
    uint32_t n_seg;
    {
        const int words = (n + kPlanThreads * 8 - 1) / (kPlanThreads * 8);      // of eight labels per thread: 1 or 2
        uint4 w[2];
        uint32_t c = 0;
#pragma unroll
        for (int v = 0; v < 2; ++v) {
            const int l = (tid * words + v) * 8;
            w[v] = v < words && l < n ? *reinterpret_cast<const uint4*>(id_of + l) : make_uint4(0u, 0u, 0u, 0u);
            c += __popc(w[v].x) + __popc(w[v].y) + __popc(w[v].z) + __popc(w[v].w);
        }
        uint32_t next = block_exclusive_sum(c, warp_sums, n_seg);
        if (n_seg > (uint32_t)kSeg) return false;          // uniform
#pragma unroll
        for (int v = 0; v < 2; ++v) {
            const int l = (tid * words + v) * 8;
            if (v < words && l < n && (w[v].x | w[v].y | w[v].z | w[v].w)) {
                uint32_t* f = &w[v].x;
#pragma unroll
                for (int q = 0; q < 8; ++q) {
                    const uint32_t here = (q & 1) ? f[q >> 1] >> 16 : f[q >> 1] & 1u;
                    if (here) {
                        if (next < (uint32_t)Mcap) merged_label[next] = l + q;
                        id_of[l + q] = (uint16_t)next++;
                    }
                }
            }
        }
    }
    if (kSeg > kNarrow && n_seg > (uint32_t)kNarrow) zero_counters(cnt, kSeg);
    __syncthreads();
    if (kSeg > kNarrow && n_seg > (uint32_t)kNarrow)
        plan_positions<E, kSeg>(lab, take, n, (int)n_seg, Mcap, merged_count, members, headers, id_of, cnt, seg_start, seg_slot, warp_sums);
    else
        plan_positions<E, kNarrow>(lab, take, n, (int)n_seg, Mcap, merged_count, members, headers, id_of, cnt, seg_start, seg_slot, warp_sums);
    if (tid == 0) *n_merged_b = (int32_t)n_seg;
    return true;
}

template <int E>
__global__ void __launch_bounds__(kPlanThreads)
merge_plan_kernel(const int32_t* label, const uint8_t* keep_mask,
                  const int32_t* vis_len, int vis_len_uniform, int Nv_cap, int Mcap,
                  int32_t* __restrict__ merged_label, int32_t* __restrict__ merged_count,
                  int32_t* __restrict__ n_merged, uint16_t* members, MergeHeader* headers,
                  int* __restrict__ status) {
    extern __shared__ __align__(16) uint32_t smem_items[];   // two item buffers of Nv_cap (rounded up to 4), then the counters
    __shared__ uint32_t warp_sums[32];
    grid_dependency_wait();
    const int b = blockIdx.x, tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
    if (b == 0 && tid == 0) *status = VITCOP_OK;
    const uint32_t lt = (1u << lane) - 1u;
    int n = vis_len ? __ldcg(vis_len + b) : vis_len_uniform;
    n = max(0, min(n, Nv_cap));
    const int cap4 = (Nv_cap + 3) & ~3;
    uint32_t* buf0 = smem_items;
    uint32_t* buf1 = smem_items + cap4;
    uint16_t* cnt = reinterpret_cast<uint16_t*>(smem_items + 2 * cap4);
    label += (size_t)b * Nv_cap;
    keep_mask += (size_t)b * Nv_cap;
    merged_label += (size_t)b * Mcap;
    merged_count += (size_t)b * Mcap;
    members += (size_t)b * member_stride(Nv_cap);
    headers += (size_t)b * Mcap;

    // this thread's tokens: warp w owns [w * 32 rows, (w + 1) * 32 rows), row by row, so that entry order is (warp, row, lane) order
    uint32_t it[E], take = 0;
    {
        const int rows = (n + kPlanThreads - 1) / kPlanThreads;
#pragma unroll
        for (int e = 0; e < E; ++e) {
            const int i = (warp * rows + e) * 32 + lane;
            it[e] = 0;
            if (e < rows && i < n) {
                const uint32_t lab = (uint32_t)label[i];
                it[e] = lab >= (uint32_t)n ? (uint32_t)n - 1 : lab;        // out-of-range labels are clamped, never indexed
                if (!keep_mask[i]) take |= 1u << e;
            }
        }
    }
    if (plan_by_count<E>(it, take, n, Mcap, merged_label, merged_count, n_merged + b, members, headers,
                         reinterpret_cast<uint16_t*>(smem_items), warp_sums)) {
        grid_dependency_launch_dependents();
        return;
    }
    __syncthreads();
    // ---- more clusters than that: the non-elite tokens, in token order (count per warp, one scan, then place)
    uint32_t m;
    {
        const int rows = (n + kPlanThreads - 1) / kPlanThreads;
        uint32_t mine = 0;
#pragma unroll
        for (int e = 0; e < E; ++e) mine += __popc(__ballot_sync(0xffffffffu, take >> e & 1u));
        uint32_t pos = warp_totals_scan(mine, warp_sums, m);
#pragma unroll
        for (int e = 0; e < E; ++e) {
            const uint32_t bal = __ballot_sync(0xffffffffu, take >> e & 1u);
            if (take >> e & 1u) buf0[pos + __popc(bal & lt)] = (it[e] << 16) | (uint32_t)((warp * rows + e) * 32 + lane);
            pos += __popc(bal);
        }
    }
    __syncthreads();
    // ---- members of a cluster side by side, in ascending token order; clusters in ascending label order
    const uint32_t* items = sort_by_label(buf0, buf1, (int)m, n > 1 ? 32 - __clz(n - 1) : 0, cnt, warp_sums);

    // ---- run heads -> merged rows; run tails close them; the sorted indices are the member list
    const int rows = ((int)m + kPlanThreads - 1) / kPlanThreads;
    uint32_t wh = 0, wt = 0;
#pragma unroll 1
    for (int e = 0; e < rows; ++e) {
        const int p = (warp * rows + e) * 32 + lane;
        bool head = false, tail = false;
        if (p < (int)m) {
            const uint32_t c = items[p], lab = c >> 16;
            head = p == 0 || (items[p - 1] >> 16) != lab;
            tail = p + 1 >= (int)m || (items[p + 1] >> 16) != lab;
            members[p] = (uint16_t)(c & 0xFFFFu);
        }
        wh += __popc(__ballot_sync(0xffffffffu, head));
        wt += __popc(__ballot_sync(0xffffffffu, tail));
    }
    // (two 16-bit counts in a word: neither can exceed 16384)
    uint32_t totals;
    const uint32_t before = warp_totals_scan(wh | (wt << 16), warp_sums, totals);
    uint32_t hs = before & 0xFFFFu, ts = before >> 16;
    const uint32_t heads = totals & 0xFFFFu;
#pragma unroll 1
    for (int e = 0; e < rows; ++e) {
        const int p = (warp * rows + e) * 32 + lane;
        bool head = false, tail = false;
        uint32_t lab = 0;
        if (p < (int)m) {
            lab = items[p] >> 16;
            head = p == 0 || (items[p - 1] >> 16) != lab;
            tail = p + 1 >= (int)m || (items[p + 1] >> 16) != lab;
        }
        const uint32_t hb = __ballot_sync(0xffffffffu, head), tb = __ballot_sync(0xffffffffu, tail);
        const uint32_t h = hs + __popc(hb & lt), t = ts + __popc(tb & lt);
        if (head && h < (uint32_t)Mcap) {
            merged_label[h] = (int32_t)lab;
            headers[h].start = p;
        }
        if (tail && t < (uint32_t)Mcap) merged_count[t] = p;            // position of the run's last member for now
        hs += __popc(hb);
        ts += __popc(tb);
    }
    __syncthreads();
    for (int mm = tid; mm < Mcap; mm += kPlanThreads) {
        int count = 0, start = 0;
        if (mm < (int)heads) {
            start = headers[mm].start;
            count = merged_count[mm] - start + 1;
            merged_count[mm] = count;
            store_first(items + start, count, headers + mm);
        }
        *reinterpret_cast<int4*>(headers + mm) = make_int4(count, start, mm, 0);
    }
    if (tid == 0) n_merged[b] = (int32_t)heads;
    grid_dependency_launch_dependents();
}

__device__ __forceinline__ uint4 ld_stream(const uint4* p) {
    uint4 v;
    asm("ld.global.nc.L1::no_allocate.v4.u32 {%0,%1,%2,%3}, [%4];" : "=r"(v.x), "=r"(v.y), "=r"(v.z), "=r"(v.w) : "l"(p));
    return v;
}
// a[q] += the bf16 pair q of v, both halves with one instruction (each rounded like a scalar addition).
__device__ __forceinline__ void add8(unsigned long long (&a)[4], const uint4& v) {
    const uint32_t w[4] = {v.x, v.y, v.z, v.w};
#pragma unroll
    for (int q = 0; q < 4; ++q) {
        unsigned long long x;
        asm("mov.b64 %0, {%1, %2};" : "=l"(x) : "r"(w[q] << 16), "r"(w[q] & 0xffff0000u));
        asm("add.rn.f32x2 %0, %0, %1;" : "+l"(a[q]) : "l"(x));
    }
}

// A CTA lives for its trips to memory, so the planner leaves, beside the member list, a header per merged row that holds the
// run and its first sixteen members, four for each warp: one trip leads to the data.  (Run, member list and rows in three
// dependent trips: 36 us for 121 MB of rows, 4 x 4608 tokens x 4096.)
// P: 16-byte pieces of a row per lane; R: members a warp has in flight.
template <int P, int R>
__global__ void __launch_bounds__(kRowsThreads)
merge_rows_kernel(const uint4* __restrict__ hidden, int B, int N, int dh8, int slices, int vis_start, int Nv_cap, int Mcap,
                  const MergeHeader* headers, const uint16_t* members,
                  void* __restrict__ merged_bf16, float* __restrict__ merged_f32) {
    constexpr int G = kRowsThreads / 32;                  // warps sharing the members
    static_assert(G == 4, "a header lists members for four warps");
    __shared__ unsigned long long partial[P][G][32][5];      // padded against bank conflicts
    grid_dependency_wait();
    // slices of a row side by side, then the samples, then the rows in header order: the long ones of all samples come first
    const int tid = threadIdx.x, g = tid >> 5, lane = tid & 31;
    const int slice = (int)(blockIdx.x % (unsigned)slices), xb = (int)(blockIdx.x / (unsigned)slices);
    const int b = xb % B, x = xb / B;
    const MergeHeader* h = headers + (size_t)b * Mcap + x;
    const int4 run = __ldcg(reinterpret_cast<const int4*>(h));
    const uint2 four = __ldcg(reinterpret_cast<const uint2*>(h->first[g]));
    const int count = run.x, m = run.z;
    if (count == 0) return;                               // no such merged row
    const uint16_t* mem = members + (size_t)b * member_stride(Nv_cap) + run.y;
    const int piece = slice * (32 * P) + lane;      // 16-byte pieces of the hidden row this lane owns: + 32 p
    unsigned long long acc[P][4];               // pairs of fp32 sums
#pragma unroll
    for (int p = 0; p < P; ++p)
#pragma unroll
        for (int u = 0; u < 4; ++u) acc[p][u] = 0ull;
    {
        const uint4* src = hidden + ((size_t)b * N + vis_start) * dh8 + piece;
        uint32_t idx[4] = {four.x & 0xFFFFu, four.x >> 16, four.y & 0xFFFFu, four.y >> 16};
        for (int r = g; r < count; r += R * G) {
            uint4 v[R][P];
#pragma unroll
            for (int u = 0; u < R; ++u)
#pragma unroll
                for (int p = 0; p < P; ++p)
                    if (r + u * G < count && piece + 32 * p < dh8) v[u][p] = ld_stream(src + (size_t)idx[u] * dh8 + 32 * p);
#pragma unroll
            for (int u = 0; u < 4; ++u) {                 // the header's list, then the next ones, which travel with the data
                if (R < 4 && u < 4 - R) idx[u] = idx[u + R];
                else if (r + (4 + (u - (4 - R))) * G < count) idx[u] = __ldcg(mem + r + (4 + (u - (4 - R))) * G);
            }
#pragma unroll
            for (int u = 0; u < R; ++u)
#pragma unroll
                for (int p = 0; p < P; ++p)
                    if (r + u * G < count && piece + 32 * p < dh8) add8(acc[p], v[u][p]);
        }
    }
#pragma unroll
    for (int p = 0; p < P; ++p)
#pragma unroll
        for (int u = 0; u < 4; ++u) partial[p][g][lane][u] = acc[p][u];
    __syncthreads();
    // each thread finishes a pair of elements of its lane's pieces: g, so that a row is written in 4- and 8-byte words
#pragma unroll
    for (int p = 0; p < P; ++p) {
        if (piece + 32 * p >= dh8) break;
        float sum[2] = {0.f, 0.f};
#pragma unroll
        for (int q = 0; q < G; ++q) {                     // warp order: fixed
            const unsigned long long pair = partial[p][q][lane][g];
            sum[0] += __uint_as_float((uint32_t)pair);
            sum[1] += __uint_as_float((uint32_t)(pair >> 32));
        }
        sum[0] = sum[0] / (float)count;
        sum[1] = sum[1] / (float)count;
        const size_t o = (((size_t)b * Mcap + m) * dh8 + piece + 32 * p) * 8 + 2 * g;
        if (merged_f32) *reinterpret_cast<float2*>(merged_f32 + o) = make_float2(sum[0], sum[1]);
        if (merged_bf16)
            *reinterpret_cast<__nv_bfloat162*>(static_cast<__nv_bfloat16*>(merged_bf16) + o) =
                __nv_bfloat162(__float2bfloat16_rn(sum[0]), __float2bfloat16_rn(sum[1]));
    }
}

// Dynamic shared memory of the planner: the counting pass, or the sort's two buffers and counters.
size_t plan_smem(int Nv_cap, int E) {
    const size_t sort_bytes = 2 * (size_t)((Nv_cap + 3) & ~3) * sizeof(uint32_t) + (size_t)kCntEntries * sizeof(uint16_t);
    const size_t count_bytes = plan_count_bytes(Nv_cap, E);
    return sort_bytes > count_bytes ? sort_bytes : count_bytes;
}

// Workspace: status | members uint16 [B, Nv_cap rounded up to 8] | headers [B, Mcap]
struct MergeWs {
    size_t off_members, off_headers, total;
    MergeWs(int B, int Nv_cap, int Mcap) {
        size_t o = kStatusBytes;
        off_members = o; o += align_up((size_t)B * member_stride(Nv_cap) * sizeof(uint16_t), 256);
        off_headers = o; o += align_up((size_t)B * Mcap * sizeof(MergeHeader), 256);
        total = o;
    }
};

}  // namespace

size_t merge_workspace_bytes(int B, int Nv_cap, int Mcap) { return MergeWs(B, Nv_cap, Mcap).total; }

int launch_merge(const void* hidden, int B, int N, int Dh, int vis_start, const int32_t* vis_len, int vis_len_uniform,
                 int Nv_cap, const int32_t* label, const uint8_t* keep_mask, void* merged_bf16, float* merged_f32,
                 int32_t* merged_label, int32_t* merged_count, int32_t* n_merged, int Mcap, void* workspace,
                 cudaStream_t stream) {
    if (B <= 0) return VITCOP_OK;
    const MergeWs lay(B, Nv_cap, Mcap);
    char* ws = static_cast<char*>(workspace);
    uint16_t* members = reinterpret_cast<uint16_t*>(ws + lay.off_members);
    MergeHeader* headers = reinterpret_cast<MergeHeader*>(ws + lay.off_headers);
    cudaLaunchAttribute attr[1];
    attr[0].id = cudaLaunchAttributeProgrammaticStreamSerialization;
    attr[0].val.programmaticStreamSerializationAllowed = 1;
    {
        const int v = Nv_cap <= kPlanThreads ? 0 : Nv_cap <= 4 * kPlanThreads ? 1 : Nv_cap <= 8 * kPlanThreads ? 2 : 3;
        auto kern = v == 0 ? merge_plan_kernel<1> : v == 1 ? merge_plan_kernel<4> : v == 2 ? merge_plan_kernel<8> : merge_plan_kernel<16>;
        const int E = v == 0 ? 1 : v == 1 ? 4 : v == 2 ? 8 : 16;
        const size_t smem = plan_smem(Nv_cap, E);
        if (v > 0) {                                       // (up to 1024 tokens 19 KB)
            static DoneOnDevice attr_done[4];
            const int rc = allow_dynamic_smem(kern, plan_smem(E * kPlanThreads, E), attr_done[v]);
            if (rc != VITCOP_OK) return rc;
        }
        cudaLaunchConfig_t cfg = {};
        cfg.gridDim = dim3(B);
        cfg.blockDim = dim3(kPlanThreads);
        cfg.dynamicSmemBytes = smem;
        cfg.stream = stream;
        cfg.attrs = attr;
        cfg.numAttrs = pdl_allowed(true) ? 1 : 0;
        KernelTimeScope timed("merge_plan_kernel", stream);
        int rc = record_cuda(cudaLaunchKernelEx(&cfg, kern, label, keep_mask, vis_len, vis_len_uniform,
                                                Nv_cap, Mcap, merged_label, merged_count, n_merged, members, headers,
                                                static_cast<int*>(workspace)));
        if (rc != VITCOP_OK) return rc;
    }
    if (Mcap <= 0 || Dh <= 0 || (!merged_bf16 && !merged_f32)) return VITCOP_OK;
    const int dh8 = Dh / 8;
    cudaLaunchConfig_t cfg = {};
    // Two pieces a lane halve the CTAs and their trips to the plan; a few rows keep the chip better busy cut into more CTAs.  With
    // many CTAs and few members a row, two members in flight a warp instead of four let more CTAs share an SM.  (Pieces, members in
    // flight; us of the kernel under event brackets.  240 CTAs of 400 members: 1,4 123, 2,4 142.  2304 of 18: 1,4 60, 2,4 70.  3712 of 16:
    // 1,4 21, 2,4 19, 2,2 21.  7392 of 16: 1,4 35, 2,4 31, 2,2 29.  20000 of 3: 2,4 50, 2,2 39.  9600 of 44: 2,4 76, 2,2 95.)
    const long long wide = (long long)Mcap * B * ((dh8 + 63) / 64), sms = gram_num_sms();
    const bool few = wide < 16 * sms, shorter = !few && wide >= 28 * sms && Nv_cap <= 24LL * Mcap;
    const int pieces = few ? 1 : 2, slices = (dh8 + 32 * pieces - 1) / (32 * pieces);
    auto kern = few ? merge_rows_kernel<1, 4> : shorter ? merge_rows_kernel<2, 2> : merge_rows_kernel<2, 4>;
    const long long ctas = (long long)Mcap * B * slices;
    if (ctas > 0x7fffffffLL) return VITCOP_ERR_UNSUPPORTED;
    cfg.gridDim = dim3((unsigned)ctas);
    cfg.blockDim = dim3(kRowsThreads);
    cfg.stream = stream;
    cfg.attrs = attr;
    cfg.numAttrs = pdl_allowed(true) ? 1 : 0;
    KernelTimeScope timed("merge_rows_kernel", stream);
    return record_cuda(cudaLaunchKernelEx(&cfg, kern, static_cast<const uint4*>(hidden), B, N, dh8, slices,
                                          vis_start, Nv_cap, Mcap, (const MergeHeader*)headers, (const uint16_t*)members, merged_bf16,
                                          merged_f32));
}

}  // namespace vitcop
