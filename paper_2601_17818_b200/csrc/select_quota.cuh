// Cluster-quota selection (Eq. 5 / Algorithm 3 up to the elite set) as a device routine of one to eight CTAs, called by
// select_quota_kernel (select.cu) for more than 2048 tokens (select_rank.cuh: up to there).
#pragma once

#include "async_copy.cuh"
#include "block_sort.cuh"
#include "internal.cuh"

namespace vitcop {

constexpr int kSelThreads = 1024;
constexpr int kSelWarps = kSelThreads / 32;   // block_prefix_count (internal.cuh) is written for this size

// Ascending key order == the selection order: smaller scores first (or larger, when `largest`),
// -0 == +0, NaN after everything.
__device__ __forceinline__ uint32_t order_key(float s, int largest) {
    if (s != s) return 0xFFFFFFFFu;
    uint32_t u = __float_as_uint(s);
    if (u == 0x80000000u) u = 0u;
    const uint32_t asc = (u & 0x80000000u) ? ~u : (u | 0x80000000u);
    return largest ? ~asc : asc;
}

// Writes keep flags (already decided per element) out in ascending index order.
// flag_of(i) -> bool for i < n.  All threads call.
template <typename F>
__device__ __forceinline__ uint32_t emit_ascending(int n, F flag_of, int32_t* keep_idx, int keep_stride,
                                                   uint8_t* keep_mask, uint32_t* warp_sums) {
    uint32_t running = 0;
    for (int base = 0; base < n; base += kSelThreads) {
        const int i = base + threadIdx.x;
        const bool f = i < n && flag_of(i);
        uint32_t total;
        const uint32_t r = running + block_prefix_count(f, warp_sums, total);
        if (f && r < (uint32_t)keep_stride) keep_idx[r] = i;
        if (keep_mask && i < n) keep_mask[i] = f ? 1 : 0;
        running += total;
    }
    return running;
}

// Loads the composite keys (label, score key, index) of one sequence, padded with ~0 up to P, and sorts them.
template <int E>
__device__ void sort_composites(const float* score, const int32_t* label, int n, int T,
                                unsigned long long* comp) {
    unsigned long long r[E];
    const int t = threadIdx.x;
#pragma unroll
    for (int e = 0; e < E; ++e) {
        const int i = t * E + e;
        unsigned long long c = ~0ull;
        if (t < T && i < n) {
            uint32_t lab = (uint32_t)label[i];
            if (lab >= (uint32_t)n) lab = (uint32_t)n - 1;          // out-of-range labels are clamped, never indexed
            c = ((unsigned long long)lab << 48) | ((unsigned long long)order_key(score[i], 0) << 16) |
                (unsigned long long)i;
        }
        r[e] = c;
    }
    block_bitonic_sort<E>(r, comp, T);
}

// ------------------------------------------------------------------------------------------ per-cluster select
// Cluster-quota selection without a global sort, for up to kMaxSeg clusters.  Tokens get dense cluster ids, the
// clusters their sizes and quotas; then one of two searches finds, per cluster, the q_c smallest (score key, index)
// pairs:
//   rank   -- the tokens are scattered into per-cluster segments and every token counts the members of its own
//             segment that precede it: sum of |C_c|^2 comparisons, taken when that sum is a small multiple of n
//             (clusters of similar size, the usual outcome of Algorithm 2).  On longer samples this is most of the work, and
//             the CTAs of a thread-block cluster share the segments out: each prepares everything for itself (a microsecond
//             or two), ranks its part and sends every verdict to the CTA that will emit the token.  (One CTA per sample:
//             10 us on 576 tokens, 16 on 2880, 47 on 16384; now 7.3, 11.7 and 32);
//   radix  -- every cluster runs its own radix select (4-bit digits) for its q_c-th smallest pair, all clusters at
//             once: one shared histogram row per cluster, one thread per cluster to pick the digit, O(n) work per
//             pass whatever the sizes.  Pairs are unique, so ties need no extra pass; a cluster stops as soon as a
//             whole histogram bin is wanted, the loop when all clusters have stopped.
constexpr int kMaxSeg = 1024;
constexpr uint32_t kSegDone = 0xFFFFFFFFu;
// The rank search is taken when no searched cluster is larger than kRankMaxSize and the comparisons of the busiest CTA are few enough:
// a million of them take 28 us, and the other searches on 2880 / 4608 / 8192 / 16384 tokens 18 / 8 / 10 / 20 us longer than what is
// left of the rank search.  (Counting all comparisons against 64 n per CTA of the cluster, as if they were shared out evenly, took
// uneven clusters to the rank search: 8 x 8192 tokens 47 us instead of 27, 32 x 16384 160 instead of 47.)  A CTA of several ranks
// the segments that start in its n / R positions, so it has at most (n / R + largest) * largest, and at most all of them; where
// that bound leaves it open, the CTAs' parts are added up (a third of a microsecond).
constexpr int kRankWork = 64;                             // of one CTA, times n
__host__ __device__ constexpr uint32_t rank_part(int n, bool sorted_otherwise) {         // of one of several
    return sorted_otherwise ? 600000u : 40u * (uint32_t)n + 100000u;
}
constexpr int kRankMaxSize = 2048;
constexpr int kRadixMinTokens = 4096;                     // below this a sort beats the radix passes (fewer barriers)

// Writes the tokens whose flag is set in keepf[0..n) to keep_idx in ascending order (every thread scans a run of
// consecutive tokens, one block-wide scan places the runs); returns their number.
__device__ __forceinline__ uint32_t emit_flags_ascending(int n, const uint8_t* keepf, int32_t* keep_idx,
                                                         int keep_stride, uint8_t* keep_mask, uint32_t* warp_sums) {
    const int per = (n + kSelThreads - 1) / kSelThreads;
    const int i0 = threadIdx.x * per;
    uint32_t cnt = 0;
    for (int j = 0; j < per; ++j) cnt += (i0 + j < n && keepf[i0 + j]) ? 1u : 0u;
    uint32_t total;
    uint32_t r = block_exclusive_sum(cnt, warp_sums, total);
    for (int j = 0; j < per; ++j) {
        const int i = i0 + j;
        if (i >= n) break;
        const bool f = keepf[i] != 0;
        if (f) {
            if (r < (uint32_t)keep_stride) keep_idx[r] = i;
            ++r;
        }
        if (keep_mask) keep_mask[i] = f ? 1 : 0;
    }
    return total;
}

// Shared-memory layout of select_quota_by_cluster for a sample of n tokens.
struct ClusterSelSmem {
    size_t off_thr, off_krem, off_quota, off_csize, off_offs, off_misc, off_id, off_keep, total;
    int n_al;
    __host__ __device__ explicit ClusterSelSmem(int n) {
        n_al = (n + 7) & ~7;
        size_t uni = (size_t)n_al * 8;                     // seg u64 [n_al]: tokens grouped by cluster   (rank)
        const size_t hist = (size_t)kMaxSeg * 16 * 4;      // hist u32 [copies][n_seg][16]              (radix)
        if (uni < hist) uni = hist;
        off_thr = uni;
        off_krem = off_thr + (size_t)kMaxSeg * 8;
        off_quota = off_krem + (size_t)kMaxSeg * 4;
        off_csize = off_quota + (size_t)kMaxSeg * 4;
        off_offs = off_csize + (size_t)kMaxSeg * 4;
        off_misc = off_offs + (size_t)kMaxSeg * 4;
        off_id = off_misc + 16;
        off_keep = off_id + (size_t)n_al * 2;
        total = off_keep + (size_t)n_al;
    }
};

// Returns false (having written nothing) when the sample has more than kMaxSeg clusters, or sizes that rule out
// the rank search on a sample too short for the radix search to pay: the caller then sorts.  R CTAs of a thread-block
// cluster call together with the same arguments and return the same; what the rank search does not take is left to the first.
// E: tokens per thread (a CTA that runs once fetches every instruction cold: sixteen unrolled bodies where one is needed cost
// 576 tokens more than two of nine microseconds).
template <int R, int E>
__device__ __forceinline__ bool select_quota_by_cluster(const float* score, const int32_t* label, int n, int budget,
                                                        int32_t* keep_idx, int keep_stride, int32_t* n_keep_b,
                                                        uint8_t* keep_mask, int* status_word, uint8_t* smem,
                                                        uint32_t* warp_sums) {
    __shared__ uint32_t range_kept[R];                     // tokens kept in every CTA's range
    const int part = R > 1 ? (int)cluster_ctarank() : 0;
    const ClusterSelSmem L(n);
    uint32_t* hist = reinterpret_cast<uint32_t*>(smem);
    unsigned long long* seg = reinterpret_cast<unsigned long long*>(smem);
    unsigned long long* thr = reinterpret_cast<unsigned long long*>(smem + L.off_thr);
    uint32_t* krem = reinterpret_cast<uint32_t*>(smem + L.off_krem);
    uint32_t* quota = reinterpret_cast<uint32_t*>(smem + L.off_quota);
    uint32_t* csize = reinterpret_cast<uint32_t*>(smem + L.off_csize);
    uint32_t* offs = reinterpret_cast<uint32_t*>(smem + L.off_offs);
    uint32_t* misc = reinterpret_cast<uint32_t*>(smem + L.off_misc);   // min key, max key, comparisons, largest searched cluster
    uint16_t* id_of = reinterpret_cast<uint16_t*>(smem + L.off_id);
    uint8_t* keepf = smem + L.off_keep;
    const int tid = threadIdx.x;

    // ---- dense cluster ids in ascending label order
    for (int i = tid; i < L.n_al / 8; i += kSelThreads) reinterpret_cast<uint4*>(id_of)[i] = make_uint4(0u, 0u, 0u, 0u);
    if (tid < kMaxSeg) csize[tid] = 0;
    if (tid == 0) {
        misc[0] = 0xFFFFFFFFu;
        misc[1] = 0u;
        misc[2] = 0u;
        misc[3] = 0u;
    }
    __syncthreads();
    // per token: (cluster << 48) | (score key << 16) | low; low = slot inside the cluster first, then the index
    unsigned long long comp[E];
    uint32_t key_lo = 0xFFFFFFFFu, key_hi = 0u;
#pragma unroll
    for (int k = 0; k < E; ++k) {
        const int i = k * kSelThreads + tid;
        comp[k] = 0;
        if (i < n) {
            uint32_t lab = (uint32_t)__ldcg(label + i);
            if (lab >= (uint32_t)n) lab = (uint32_t)n - 1;          // out-of-range labels are clamped, never indexed
            id_of[lab] = 1;
            const uint32_t key = order_key(__ldcg(score + i), 0);
            key_lo = min(key_lo, key);
            key_hi = max(key_hi, key);
            comp[k] = ((unsigned long long)lab << 48) | ((unsigned long long)key << 16);
        }
    }
    key_lo = __reduce_min_sync(0xffffffffu, key_lo);
    key_hi = __reduce_max_sync(0xffffffffu, key_hi);
    if ((tid & 31) == 0) {
        atomicMin(&misc[0], key_lo);
        atomicMax(&misc[1], key_hi);
    }
    __syncthreads();
    // (a thread takes a run of labels; of eight at a time, two flags to a word, on longer samples)
    uint32_t n_seg;
    if (n <= 2 * kSelThreads) {
        const int l0 = 2 * tid;
        const uint32_t pair = l0 < n ? *reinterpret_cast<const uint32_t*>(id_of + l0) : 0u;     // (id_of is padded to eight)
        const uint32_t f0 = pair & 1u, f1 = (pair >> 16 & 1u) && l0 + 1 < n ? 1u : 0u;
        const uint32_t next_id = block_exclusive_sum(f0 + f1, warp_sums, n_seg);
        if (n_seg > (uint32_t)kMaxSeg) return false;       // uniform over the CTAs
        if (l0 < n) *reinterpret_cast<uint32_t*>(id_of + l0) = next_id | (next_id + f0) << 16;
    } else {
        const int words = (n + kSelThreads * 8 - 1) / (kSelThreads * 8);        // of eight labels per thread: 1 or 2
        uint4 w[2];
        uint32_t cnt = 0;
#pragma unroll
        for (int v = 0; v < 2; ++v) {
            const int l = (tid * words + v) * 8;
            w[v] = v < words && l < n ? *reinterpret_cast<const uint4*>(id_of + l) : make_uint4(0u, 0u, 0u, 0u);
            cnt += __popc(w[v].x) + __popc(w[v].y) + __popc(w[v].z) + __popc(w[v].w);
        }
        uint32_t next_id = block_exclusive_sum(cnt, warp_sums, n_seg);
        if (n_seg > (uint32_t)kMaxSeg) return false;       // uniform over the CTAs
#pragma unroll
        for (int v = 0; v < 2; ++v) {
            const int l = (tid * words + v) * 8;
            if (v < words && l < n) {
                uint32_t* f = &w[v].x;
#pragma unroll
                for (int q = 0; q < 4; ++q) {
                    const uint32_t lo = f[q] & 1u, hi = f[q] >> 16;
                    f[q] = next_id | (next_id + lo) << 16;
                    next_id += lo + hi;
                }
                *reinterpret_cast<uint4*>(id_of + l) = w[v];
            }
        }
    }
    __syncthreads();

    // ---- cluster sizes (the atomic's return value is the token's slot inside its cluster) and quotas (Eq. 5)
#pragma unroll
    for (int k = 0; k < E; ++k) {
        if (k * kSelThreads + tid < n) {
            const uint32_t c = id_of[(uint32_t)(comp[k] >> 48)];
            const uint32_t slot = atomicAdd(&csize[c], 1u);
            comp[k] = (comp[k] & 0x0000FFFFFFFF0000ull) | ((unsigned long long)c << 48) | (unsigned long long)slot;
        }
    }
    __syncthreads();
    const long long b_elites = (long long)budget - (long long)n_seg;
    if (b_elites < 0) {
        if (part != 0) return true;
        if (tid == 0 && status_word) atomicMax(status_word, VITCOP_ERR_BUDGET);
        for (int i = tid; i < n; i += kSelThreads) keepf[i] = 0;
        __syncthreads();
        emit_flags_ascending(n, keepf, keep_idx, keep_stride, keep_mask, warp_sums);
        if (tid == 0) *n_keep_b = 0;
        return true;
    }
    {
        uint32_t size = 0, work = 0, largest = 0;
        if (tid < (int)n_seg) {
            size = csize[tid];
            // (a budget of n or more keeps every cluster whole, as n does: the product fits 32 bits)
            const uint32_t q = size * (uint32_t)(b_elites < n ? b_elites : n) / (uint32_t)n;
            quota[tid] = q;
            const bool searched = q > 0 && q < size;                 // none or all of a cluster: nothing to search
            krem[tid] = searched ? q : kSegDone;
            if (searched) {
                largest = size;
                work = size > (uint32_t)kRankMaxSize ? 0u : size * size;
            }
        }
        work = __reduce_add_sync(0xffffffffu, work);
        largest = __reduce_max_sync(0xffffffffu, largest);
        if ((tid & 31) == 0 && largest) {
            atomicAdd(&misc[2], min(work, 0x0FFFFFFFu));             // 32 sizes of at most 2048: below 2^27
            atomicMax(&misc[3], largest);
        }
        uint32_t total;
        const uint32_t o = block_exclusive_sum(size, warp_sums, total);   // its barriers publish misc as well
        if (tid < (int)n_seg) offs[tid] = o;
    }
    const uint32_t largest = misc[3], all = misc[2];
    bool by_rank = largest <= (uint32_t)kRankMaxSize;
    if (R == 1) {
        by_rank = by_rank && all <= (uint32_t)kRankWork * (uint32_t)n;
    } else if (by_rank) {
        const uint32_t most = rank_part(n, n <= kRadixMinTokens);
        if (min(all, ((uint32_t)(n / R) + largest) * largest) > most) {       // (uniform over the CTAs)
            __shared__ uint32_t part_work[R];
            if (tid < R) part_work[tid] = 0u;
            __syncthreads();
            const bool searched = tid < (int)n_seg && krem[tid] != kSegDone;
            const uint32_t size = searched ? csize[tid] : 0u, to = searched ? offs[tid] / (uint32_t)((n + R - 1) / R) : 0u;
#pragma unroll
            for (int u = 0; u < R; ++u) {
                const uint32_t w = __reduce_add_sync(0xffffffffu, to == (uint32_t)u ? size * size : 0u);
                if ((tid & 31) == u && w) atomicAdd(&part_work[u], w);
            }
            __syncthreads();
#pragma unroll
            for (int u = 0; u < R; ++u) by_rank = by_rank && part_work[u] <= most;
        }
    }
    const uint32_t range_lo = misc[0], range_hi = misc[1];
    if (!by_rank && n <= kRadixMinTokens) return false;    // uniform; nothing has been written yet
    if (!by_rank && part != 0) return true;
    __syncthreads();

    if (by_rank) {
        // ---- scatter into per-cluster segments; then the thread of segment position p ranks the token stored
        // there.  The lanes of a warp mostly sit in one cluster: equal trip counts and broadcast reads.
#pragma unroll
        for (int k = 0; k < E; ++k) {
            const int i = k * kSelThreads + tid;
            if (i < n) {
                const uint32_t c = (uint32_t)(comp[k] >> 48);
                seg[offs[c] + (uint32_t)(comp[k] & 0xFFFFull)] = (comp[k] & ~0xFFFFull) | (unsigned long long)i;
            }
        }
        __syncthreads();
        const int range = (n + R - 1) / R;                 // segment positions a CTA ranks, tokens it emits
        if (R > 1) cluster_sync_all();                     // every CTA of the cluster has started: its memory may be written
        for (int p = part * range + tid; p < n; p += kSelThreads) {
            const unsigned long long mine = seg[p];
            const uint32_t c = (uint32_t)(mine >> 48);
            if (R > 1) {
                // a CTA takes the segments that start in its range, whole: inside a segment the members' order is its own
                // (slots were handed out by atomics), only where segments start is common to all CTAs
                const int at = (int)offs[c];
                if (at < part * range) continue;
                if (at >= (part + 1) * range) break;
            }
            const uint32_t q = quota[c], size = csize[c];
            bool keep = q >= size;
            if (!keep && q > 0) {
                const unsigned long long* members = seg + offs[c];
                uint32_t before = 0;
                uint32_t m = 0;
                for (; m + 4 <= size; m += 4) {
                    const unsigned long long m0 = members[m], m1 = members[m + 1], m2 = members[m + 2],
                                             m3 = members[m + 3];
                    before += (m0 < mine ? 1u : 0u) + (m1 < mine ? 1u : 0u) + (m2 < mine ? 1u : 0u) +
                              (m3 < mine ? 1u : 0u);
                }
                for (; m < size; ++m) before += members[m] < mine ? 1u : 0u;
                keep = before < q;                        // same cluster bits: the order of (score key, index)
            }
            const uint32_t i = (uint32_t)(mine & 0xFFFFull);
            if (R == 1) keepf[i] = keep ? 1 : 0;
            else
                asm volatile("st.shared::cluster.u8 [%0], %1;" ::"r"(cluster_map(smem_u32(keepf + i), i / (uint32_t)range)),
                             "r"(keep ? 1u : 0u)
                             : "memory");
        }
        if (R > 1) {
            // ---- every CTA emits its range of tokens, behind the kept ones of the ranges in front of it
            cluster_sync_all();
            const int first = part * range, last = min(n, first + range);
            const int per = (range + kSelThreads - 1) / kSelThreads, i0 = first + tid * per;
            uint32_t cnt = 0;
            for (int j = 0; j < per; ++j) cnt += (i0 + j < last && keepf[i0 + j]) ? 1u : 0u;
            uint32_t total;
            uint32_t r = block_exclusive_sum(cnt, warp_sums, total);
            if (tid < R)
                asm volatile("st.shared::cluster.u32 [%0], %1;" ::"r"(cluster_map(smem_u32(range_kept + part), (uint32_t)tid)), "r"(total)
                             : "memory");
            cluster_sync_all();
            uint32_t all = 0;
#pragma unroll
            for (int u = 0; u < R; ++u) {
                if (u < part) r += range_kept[u];
                all += range_kept[u];
            }
            for (int j = 0; j < per; ++j) {
                const int i = i0 + j;
                if (i >= last) break;
                const bool f = keepf[i] != 0;
                if (f) {
                    if (r < (uint32_t)keep_stride) keep_idx[r] = i;
                    ++r;
                }
                if (keep_mask) keep_mask[i] = f ? 1 : 0;
            }
            if (part == 0 && tid == 0) *n_keep_b = (int32_t)all;
            return true;
        }
    } else {
        // ---- per-cluster radix select of the quota-th smallest pair, 4 bits per pass from the top of the 48-bit
        // (score key, index) value.  The digits above the first bit in which two score keys differ are the same
        // for every token and are skipped.
#pragma unroll
        for (int k = 0; k < E; ++k)
            comp[k] = (comp[k] & ~0xFFFFull) | (unsigned long long)(k * kSelThreads + tid);
        const int same_bits = __clz((int)(range_lo ^ range_hi));                 // 32 when all scores are equal
        const int shift0 = ((47 - same_bits) / 4) * 4;
        const unsigned long long thr0 = (((unsigned long long)range_lo << 16) >> (shift0 + 4)) << (shift0 + 4);
        if (tid < (int)n_seg) thr[tid] = thr0;
        // few clusters: several copies of the histogram, one per group of warps, spread the shared-memory atomics
        int copies = 1;
        while (copies < 8 && (int)n_seg * 2 * copies <= kMaxSeg) copies <<= 1;
        uint32_t* my_hist = hist + (size_t)((tid >> 5) & (copies - 1)) * n_seg * 16;
        for (int shift = shift0; shift >= 0; shift -= 4) {
            for (int h = tid; h < (int)n_seg * 16 * copies; h += kSelThreads) hist[h] = 0;
            __syncthreads();
#pragma unroll
            for (int k = 0; k < E; ++k) {
                if (k * kSelThreads + tid < n) {
                    const uint32_t c = (uint32_t)(comp[k] >> 48);
                    if (krem[c] != kSegDone) {
                        const unsigned long long key = comp[k] & 0xFFFFFFFFFFFFull;
                        if ((key >> (shift + 4)) == (thr[c] >> (shift + 4)))
                            atomicAdd(&my_hist[c * 16 + (uint32_t)((key >> shift) & 15ull)], 1u);
                    }
                }
            }
            __syncthreads();
            int open_left = 0;
            if (tid < (int)n_seg) {
                const int c = tid;
                uint32_t kr = krem[c];
                if (kr != kSegDone) {
                    uint32_t cum = 0;
                    for (int dgt = 0; dgt < 16; ++dgt) {
                        uint32_t h = 0;
                        for (int r = 0; r < copies; ++r) h += hist[((size_t)r * n_seg + c) * 16 + dgt];
                        if (cum + h >= kr) {
                            unsigned long long t = thr[c] | ((unsigned long long)dgt << shift);
                            kr -= cum;
                            if (h == kr || shift == 0) {   // the whole bin is wanted: every pair up to its top is kept
                                t |= (1ull << shift) - 1ull;
                                krem[c] = kSegDone;
                            } else {
                                krem[c] = kr;
                                open_left = 1;
                            }
                            thr[c] = t;
                            break;
                        }
                        cum += h;
                    }
                }
            }
            if (!__syncthreads_or(open_left)) break;
        }
#pragma unroll
        for (int k = 0; k < E; ++k) {
            const int i = k * kSelThreads + tid;
            if (i < n) {
                const uint32_t c = (uint32_t)(comp[k] >> 48);
                const uint32_t q = quota[c];
                const bool keep = q >= csize[c] ? true : (q == 0 ? false : (comp[k] & 0xFFFFFFFFFFFFull) <= thr[c]);
                keepf[i] = keep ? 1 : 0;
            }
        }
    }
    __syncthreads();
    const uint32_t kept = emit_flags_ascending(n, keepf, keep_idx, keep_stride, keep_mask, warp_sums);
    if (tid == 0) *n_keep_b = (int32_t)kept;
    return true;
}

// ------------------------------------------------------------------------------------------ quota by a sort
// For more clusters than the per-cluster searches handle, or a short sample with very uneven clusters: the composites (label, score
// key, index) sorted by one CTA.  Shared memory: comp[P] (uint64), cstart[n] and csize[n] (uint16, indexed by label value), keep[n]
// (uint8).
__device__ __forceinline__ void select_by_sort(const float* score, const int32_t* label, int n, int Nv_cap, int P_cap, int budget,
                                               int32_t* keep_idx, int keep_stride, int32_t* n_keep_b, uint8_t* keep_mask,
                                               int* status_word, uint8_t* smem, uint32_t* warp_sums) {
    unsigned long long* comp = reinterpret_cast<unsigned long long*>(smem);
    uint16_t* cstart = reinterpret_cast<uint16_t*>(comp + P_cap);
    uint16_t* csize = cstart + Nv_cap;
    uint8_t* keepf = reinterpret_cast<uint8_t*>(csize + Nv_cap);
    const int tid = threadIdx.x;
    int P = 256;                                          // at least one warp of 8 keys per thread
    while (P < n) P <<= 1;
    for (int i = tid; i < n; i += kSelThreads) keepf[i] = 0;
    if (P <= 8 * kSelThreads) sort_composites<8>(score, label, n, P / 8, comp);
    else sort_composites<16>(score, label, n, P / 16, comp);

    // cluster heads / tails in the sorted order
    uint32_t heads_here = 0;
    for (int p = tid; p < n; p += kSelThreads) {
        const uint32_t lab = (uint32_t)(comp[p] >> 48);
        if (p == 0 || (uint32_t)(comp[p - 1] >> 48) != lab) {
            cstart[lab] = (uint16_t)p;
            ++heads_here;
        }
    }
    __syncthreads();
    for (int p = tid; p < n; p += kSelThreads) {
        const uint32_t lab = (uint32_t)(comp[p] >> 48);
        if (p == n - 1 || (uint32_t)(comp[p + 1] >> 48) != lab) csize[lab] = (uint16_t)(p - cstart[lab]);  // size - 1
    }
    // N_c = number of heads
    uint32_t nc = heads_here;
#pragma unroll
    for (int off = 16; off > 0; off >>= 1) nc += __shfl_xor_sync(0xffffffffu, nc, off);
    if ((tid & 31) == 0) warp_sums[tid >> 5] = nc;
    __syncthreads();
    nc = 0;
    for (int w = 0; w < kSelWarps; ++w) nc += warp_sums[w];
    __syncthreads();

    const long long b_elites = (long long)budget - (long long)nc;
    if (b_elites < 0) {
        if (tid == 0 && status_word) atomicMax(status_word, VITCOP_ERR_BUDGET);
    } else {
        for (int p = tid; p < n; p += kSelThreads) {
            const unsigned long long c = comp[p];
            const uint32_t lab = (uint32_t)(c >> 48);
            const long long size_c = (long long)csize[lab] + 1;
            const long long q = (size_c * b_elites) / (long long)n;
            if ((long long)(p - (int)cstart[lab]) < q) keepf[(uint32_t)(c & 0xFFFFull)] = 1;
        }
    }
    __syncthreads();
    const uint32_t kept =
        emit_ascending(n, [&](int i) { return keepf[i] != 0; }, keep_idx, keep_stride, keep_mask, warp_sums);
    if (tid == 0) *n_keep_b = (int32_t)kept;
}

// For more than 2048 tokens a function of its own: in the middle of the kernel the searches in front of it came out with fewer registers or
// more spills (8 x 16384 tokens in even clusters 24.4 us, 22.7 so; 1 x 9000 18.1, 17.0; uneven clusters 5 x 4372 26.3, 24.7, 2 x 7508 32.9, 31.0).
// Not so with four CTAs and sixteen tokens a thread, which spills more that way (32 x 16345 in uneven clusters 47.3, 48.8).
static __device__ __noinline__ void select_by_sort_apart(const float* score, const int32_t* label, int n, int Nv_cap, int P_cap, int budget,
                                                         int32_t* __restrict__ keep_idx, int keep_stride, int32_t* __restrict__ n_keep_b,
                                                         uint8_t* __restrict__ keep_mask, int* __restrict__ status_word) {
    extern __shared__ __align__(16) uint32_t quota_smem[];
    __shared__ uint32_t warp_sums[kSelWarps];
    select_by_sort(score, label, n, Nv_cap, P_cap, budget, keep_idx, keep_stride, n_keep_b, keep_mask, status_word,
                   reinterpret_cast<uint8_t*>(quota_smem), warp_sums);
}

// ------------------------------------------------------------------------------------------ quota
// Cluster-quota selection of sample b by R whole CTAs (kSelThreads threads each); uses the dynamic shared memory.
template <int R, int E>
__device__ __forceinline__ void select_quota_body(const float* score, const int32_t* label,
                                                  const int32_t* vis_len, int vis_len_uniform,
                                                  int Nv_cap, int P_cap, int budget, int32_t* __restrict__ keep_idx,
                                                  int keep_stride, int32_t* __restrict__ n_keep,
                                                  uint8_t* __restrict__ keep_mask, int* __restrict__ status_word,
                                                  int b) {
    extern __shared__ __align__(16) uint32_t quota_smem[];
    __shared__ uint32_t warp_sums[kSelWarps];

    int n = vis_len ? __ldcg(vis_len + b) : vis_len_uniform;
    n = max(0, min(n, Nv_cap));
    score += (int64_t)b * Nv_cap;
    label += (int64_t)b * Nv_cap;
    keep_idx += (int64_t)b * keep_stride;
    if (keep_mask) keep_mask += (int64_t)b * Nv_cap;

    if (select_quota_by_cluster<R, E>(score, label, n, budget, keep_idx, keep_stride, n_keep + b, keep_mask, status_word,
                                   reinterpret_cast<uint8_t*>(quota_smem), warp_sums))
        return;
    if (R > 1 && cluster_ctarank() != 0) return;
    __syncthreads();
    if constexpr (R == 4 && E == 16)
        select_by_sort(score, label, n, Nv_cap, P_cap, budget, keep_idx, keep_stride, n_keep + b, keep_mask, status_word,
                       reinterpret_cast<uint8_t*>(quota_smem), warp_sums);
    else
        select_by_sort_apart(score, label, n, Nv_cap, P_cap, budget, keep_idx, keep_stride, n_keep + b, keep_mask, status_word);
}


// Dynamic shared memory select_quota_body needs for a span capacity of Nv_cap tokens; *P_cap receives the padded key count.
inline size_t select_quota_smem(int Nv_cap, int* P_cap) {
    const int cap = Nv_cap > 0 ? Nv_cap : 1;
    int P = 256;
    while (P < cap) P <<= 1;
    *P_cap = P;
    const size_t sort_bytes = (size_t)P * 8 + (size_t)cap * (2 + 2 + 1) + 16;
    const size_t seg_bytes = ClusterSelSmem(cap).total;
    return sort_bytes > seg_bytes ? sort_bytes : seg_bytes;
}

}  // namespace vitcop
