// Cluster-quota selection (Eq. 5) of a sample of up to kRankTokens tokens by one CTA that holds their labels and scores in registers: of
// the tokens of a call (select.cu), or of a thread's own tokens right behind their labels (filter.cu).
//
// The tokens are counted by label (the count in front of a token is its place), the clusters laid out one behind the other in label
// order as segments of (score key, index), and every token counts the members of its segment that precede it.  A CTA alone on
// its SM: what counts is the number of dependent steps, here six barriers and two scans.  (By dense cluster numbers, which longer samples
// need for their other searches, 576 tokens took 4.9 us; 3.9 so.)
#pragma once

#include "select_quota.cuh"

namespace vitcop {

constexpr int kRankTokens = 2 * kSelThreads;

struct RankShared {
    uint32_t warp_sums[kSelWarps];
    uint32_t work;                                         // comparisons, if every cluster has to be searched; those that have to be
};
// Dynamic shared memory: seg uint64 [n_al] | count uint32 [n_al] | size uint16 [n_al] | keep uint8 [n_al], n_al = n rounded up to 8.
__host__ __device__ constexpr size_t rank_smem(int n) { return (size_t)((n + 7) & ~7) * (8 + 4 + 2 + 1); }

// lab, key: label and score key of the thread's tokens e * 1024 + thread, e < E.  Returns false, nothing written, when the clusters are
// too uneven: a sort is faster then.
template <int E>
__device__ __forceinline__ bool select_by_rank(const int (&lab)[E], const uint32_t (&key)[E], int n, int budget, RankShared& sh, uint8_t* smem,
                                               int32_t* keep_idx, int keep_stride, int32_t* n_keep_b, uint8_t* keep_mask, int* status_word) {
    static_assert(E * kSelThreads <= kRankTokens && kRankTokens <= 1 << 14, "a position and an index in 28 bits");
    const int tid = threadIdx.x, n_al = (n + 7) & ~7;
    unsigned long long* const seg = reinterpret_cast<unsigned long long*>(smem);
    uint32_t* const count = reinterpret_cast<uint32_t*>(seg + n_al);       // later: where the label's segment starts
    uint16_t* const size_at = reinterpret_cast<uint16_t*>(count + n_al);   // of the segment that starts there
    uint8_t* const keepf = reinterpret_cast<uint8_t*>(size_at + n_al);
    if (tid < n_al / 4) reinterpret_cast<uint4*>(count)[tid] = make_uint4(0u, 0u, 0u, 0u);
    if (tid < n_al / 8) reinterpret_cast<uint2*>(keepf)[tid] = make_uint2(0u, 0u);
    if (tid == 0) sh.work = 0u;
    __syncthreads();
    uint32_t place[E];
#pragma unroll
    for (int e = 0; e < E; ++e) place[e] = e * kSelThreads + tid < n ? atomicAdd(&count[lab[e]], 1u) : 0u;
    __syncthreads();
    // ---- a run of E labels to a thread: members, and where their segments start
    uint32_t size[E], sum = 0, work = 0;
#pragma unroll
    for (int q = 0; q < E; ++q) {
        const int l = tid * E + q;
        size[q] = l < n ? count[l] : 0u;
        sum += size[q] + (size[q] ? 0x10000u : 0u);        // (clusters in the upper half)
        work += size[q] * size[q];
    }
    work = __reduce_add_sync(0xffffffffu, work);
    if ((tid & 31) == 0 && work) atomicAdd(&sh.work, work);
    uint32_t total;
    uint32_t at = block_exclusive_sum(sum, sh.warp_sums, total) & 0xFFFFu;
    const int n_seg = (int)(total >> 16);
    if (budget < n_seg) {                                  // nothing is kept
        if (tid == 0) {
            if (status_word) atomicMax(status_word, VITCOP_ERR_BUDGET);
            *n_keep_b = 0;
        }
        if (keep_mask)
            for (int i = tid; i < n; i += kSelThreads) keep_mask[i] = 0;
        return true;
    }
    // (a budget of n or more keeps every cluster whole, as n does: the product fits 32 bits)
    const uint32_t elites = (uint32_t)min(budget - n_seg, n);
    auto quota_of = [&](uint32_t members) { return members * elites / (uint32_t)n; };
    if (sh.work > (uint32_t)kRankWork * (uint32_t)n) {     // (uniform) too many?  Clusters of which none or all stay need no search
        work = 0;
#pragma unroll
        for (int q = 0; q < E; ++q) {
            const uint32_t quota = quota_of(size[q]);
            if (quota > 0 && quota < size[q]) work += size[q] * size[q];
        }
        __syncthreads();
        if (tid == 0) sh.work = 0u;
        __syncthreads();
        work = __reduce_add_sync(0xffffffffu, work);
        if ((tid & 31) == 0 && work) atomicAdd(&sh.work, work);
        __syncthreads();
        if (sh.work > (uint32_t)kRankWork * (uint32_t)n) return false;
    }
#pragma unroll
    for (int q = 0; q < E; ++q) {
        if (size[q]) {
            count[tid * E + q] = at;
            size_at[at] = (uint16_t)size[q];
            at += size[q];
        }
    }
    __syncthreads();
#pragma unroll
    for (int e = 0; e < E; ++e) {
        const int i = e * kSelThreads + tid;
        if (i < n) {
            const uint32_t from = count[lab[e]];
            seg[from + place[e]] = ((unsigned long long)key[e] << 32) | (unsigned long long)(from << 14 | (uint32_t)i);
        }
    }
    __syncthreads();
    // ---- the thread of segment position p ranks the token stored there.  The lanes of a warp mostly sit in one cluster: equal trip
    // counts and broadcast reads.  Bound by instruction issue, and a comparison of whole pairs with its count is three instructions.  (The keys
    // alone first, counted below and equal, and the pairs where that leaves too many: the same without ties, 4 x 1319 tokens of six
    // different scores 12.4 us, 10.3 so.)
#pragma unroll 1
    for (int p = tid; p < n; p += kSelThreads) {
        const uint2 mine = *reinterpret_cast<const uint2*>(seg + p);
        const int from = (int)(mine.x >> 14);
        const uint32_t sz = size_at[from], quota = quota_of(sz);
        bool keep = quota >= sz;
        if (!keep && quota > 0) {
            const unsigned long long* other = seg + from;
            const unsigned long long pair = seg[p];
            uint32_t before = 0, m = 0;
            if (from & 1) {                                // (pairs of members from here on)
                before = *other < pair ? 1u : 0u;
                ++other;
                m = 1;
            }
            for (; m + 4 <= sz; m += 4, other += 4) {
                const ulonglong2 x = *reinterpret_cast<const ulonglong2*>(other), y = *reinterpret_cast<const ulonglong2*>(other + 2);
                before += (x.x < pair ? 1u : 0u) + (x.y < pair ? 1u : 0u) + (y.x < pair ? 1u : 0u) + (y.y < pair ? 1u : 0u);
            }
            for (; m < sz; ++m, ++other) before += *other < pair ? 1u : 0u;
            keep = before < quota;                         // (one segment: the order of (score key, index))
        }
        if (keep) keepf[mine.x & ((1u << 14) - 1u)] = 1;
    }
    __syncthreads();
    const uint32_t kept = emit_flags_ascending(n, keepf, keep_idx, keep_stride, keep_mask, sh.warp_sums);
    if (tid == 0) *n_keep_b = (int32_t)kept;
    return true;
}

// Dynamic shared memory of that and of the sort, for a span capacity of Nv_cap tokens; *P_cap receives the sort's padded key count.
inline size_t rank_or_sort_smem(int Nv_cap, int* P_cap) {
    const int cap = Nv_cap > 0 ? Nv_cap : 1;
    int P = 256;
    while (P < cap) P <<= 1;
    *P_cap = P;
    const size_t sort_bytes = (size_t)P * 8 + (size_t)cap * (2 + 2 + 1) + 16;
    return rank_smem(cap) > sort_bytes ? rank_smem(cap) : sort_bytes;
}

}  // namespace vitcop
