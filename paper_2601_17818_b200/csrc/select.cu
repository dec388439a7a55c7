// Budgeted selection of visual tokens: one CTA per sequence.
//
//  plain mode (Algorithm 1, Stage III / Stage I): the k smallest pairs (32-bit order-preserving score key, index).  The cut is
//    found with one or two histogram passes of 11 bits that start at the highest bit in which two keys differ; the pairs left in
//    the cut's bin are ranked by counting.  The kept indices leave in ascending order: a ballot ranks a token inside its warp,
//    one scan over the warps' counts the rest.
//  quota mode (Eq. 5 / Algorithm 3 up to the elite set): select_rank.cuh up to 2048 tokens, select_quota.cuh beyond.
#include "select_rank.cuh"

namespace vitcop {
namespace {

// ------------------------------------------------------------------------------------------ plain
// A CTA alone on its SM: what counts is the number of dependent steps.  Scores are loaded all at once and stay in registers as
// keys.  (Keys in shared memory, 8-bit passes with one match per 32 keys: 5.3 us on 128 tokens, 11.1 on 2880.)
constexpr int kPlainBits = 11, kPlainBins = 1 << kPlainBits;
constexpr int kPlainRankLanes = 4;
constexpr int kPlainRank = kSelThreads / kPlainRankLanes;  // bins of up to this many pairs are ranked by counting
static_assert(kPlainBins == 2 * kSelThreads, "two bins per thread");

// E: tokens per thread; token e * 1024 + thread.  `status`: word to clear, or null.
template <int E>
__global__ void __launch_bounds__(kSelThreads)
select_plain_kernel(const float* score, const int32_t* vis_len, int vis_len_uniform,
                    int Nv_cap, int largest, int budget, int32_t* __restrict__ keep_idx, int keep_stride,
                    int32_t* __restrict__ n_keep, uint8_t* __restrict__ keep_mask, int* __restrict__ status) {
    extern __shared__ __align__(16) uint8_t won[];         // [Nv_cap] tokens chosen among the ranked ones
    __shared__ uint32_t hist[kPlainBins];
    __shared__ unsigned long long cand[kPlainRank];        // key, index
    __shared__ uint32_t cnt[E * 32];                       // kept tokens per (round of 1024 tokens, warp)
    __shared__ uint32_t warp_sums[kSelWarps];
    __shared__ uint32_t s_lo, s_hi, s_digit, s_krem, s_count, s_cands;
    const int b = blockIdx.x, tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;

    // The compaction that follows may start at once: it copies the rows that do not depend on the selection and
    // waits for this kernel to complete before it reads the kept indices.
    grid_dependency_launch_dependents();
    hist[2 * tid] = 0;
    hist[2 * tid + 1] = 0;
    if (tid == 0) { s_lo = 0xFFFFFFFFu; s_hi = 0u; s_cands = 0u; }
    grid_dependency_wait();
    if (status && b == 0 && tid == 0) *status = VITCOP_OK;
    int n = vis_len ? __ldcg(vis_len + b) : vis_len_uniform;
    n = max(0, min(n, Nv_cap));
    const int k = max(0, min(budget, n));
    score += (int64_t)b * Nv_cap;
    keep_idx += (int64_t)b * keep_stride;
    if (keep_mask) keep_mask += (int64_t)b * Nv_cap;

    uint32_t key[E], in = 0, sel = 0, ranked = 0;          // in: tokens (bit e) on the cut; sel: chosen ones
    {
        float s[E];
#pragma unroll
        for (int e = 0; e < E; ++e) {
            const int i = e * kSelThreads + tid;
            s[e] = i < n ? __ldcg(score + i) : 0.f;
        }
        uint32_t lo = 0xFFFFFFFFu, hi = 0u;
#pragma unroll
        for (int e = 0; e < E; ++e) {
            key[e] = order_key(s[e], largest);
            if (e * kSelThreads + tid < n) {
                in |= 1u << e;
                lo = min(lo, key[e]);
                hi = max(hi, key[e]);
            }
        }
        lo = __reduce_min_sync(0xffffffffu, lo);
        hi = __reduce_max_sync(0xffffffffu, hi);
        __syncthreads();                                   // (s_lo, s_hi and the histogram are set)
        if (lane == 0 && lo <= hi) {
            atomicMin(&s_lo, lo);
            atomicMax(&s_hi, hi);
        }
    }
    __syncthreads();
    if (k >= n) {
        sel = in;
    } else if (k > 0) {
        uint32_t krem = (uint32_t)k;
        bool by_index = false;                             // the keys on the cut are all equal: the index decides
        int top = 32 - __clz(s_lo ^ s_hi);                 // bits not yet looked at
        for (;;) {
            if (top == 0) {
                by_index = true;
                top = 14;
            }
            const int shift = top > kPlainBits ? top - kPlainBits : 0;
            auto digit = [&](int e) {
                const uint32_t v = by_index ? (uint32_t)(e * kSelThreads + tid) : key[e];
                return (v >> shift) & ((1u << (top - shift)) - 1u);
            };
#pragma unroll
            for (int e = 0; e < E; ++e)
                if (in >> e & 1u) atomicAdd(&hist[digit(e)], 1u);
            __syncthreads();
            const uint32_t h0 = hist[2 * tid], h1 = hist[2 * tid + 1];
            uint32_t total;
            const uint32_t before = block_exclusive_sum(h0 + h1, warp_sums, total);
            if (before < krem && krem <= before + h0 + h1) {
                const bool second = krem > before + h0;
                s_digit = 2 * tid + (second ? 1 : 0);
                s_krem = krem - before - (second ? h0 : 0u);
                s_count = second ? h1 : h0;
            }
            hist[2 * tid] = 0;                             // for the next pass
            hist[2 * tid + 1] = 0;
            __syncthreads();
            const uint32_t cut = s_digit, count = s_count;
            krem = s_krem;
#pragma unroll
            for (int e = 0; e < E; ++e) {
                if (in >> e & 1u) {
                    const uint32_t d = digit(e);
                    if (d < cut) sel |= 1u << e;
                    if (d != cut) in &= ~(1u << e);
                }
            }
            top = shift;
            if (count == krem) {                           // the whole bin is wanted
                sel |= in;
                in = 0;
                break;
            }
            if (count <= (uint32_t)kPlainRank) {
#pragma unroll
                for (int e = 0; e < E; ++e) {
                    if (in >> e & 1u) {
                        const int i = e * kSelThreads + tid;
                        won[i] = 0;
                        cand[atomicAdd(&s_cands, 1u)] = ((unsigned long long)key[e] << 32) | (unsigned long long)(uint32_t)i;
                    }
                }
                ranked = krem;
                break;
            }
            __syncthreads();                               // (s_digit .. are rewritten)
        }
    }
    if (ranked > 0) {                                      // (uniform) four threads per candidate count the smaller ones
        __syncthreads();
        const int c = tid / kPlainRankLanes, cands = (int)s_cands;
        const unsigned long long mine = c < cands ? cand[c] : 0ull;
        uint32_t rank = 0;
        if (c < cands)
            for (int o = tid % kPlainRankLanes; o < cands; o += kPlainRankLanes) rank += cand[o] < mine ? 1u : 0u;
#pragma unroll
        for (int off = 1; off < kPlainRankLanes; off <<= 1) rank += __shfl_xor_sync(0xffffffffu, rank, off);
        if (c < cands && tid % kPlainRankLanes == 0 && rank < ranked) won[(uint32_t)mine] = 1;
        __syncthreads();
#pragma unroll
        for (int e = 0; e < E; ++e)
            if ((in >> e & 1u) && won[e * kSelThreads + tid]) sel |= 1u << e;
    }
    // ---- kept indices in ascending order
#pragma unroll
    for (int e = 0; e < E; ++e) {
        const uint32_t bal = __ballot_sync(0xffffffffu, sel >> e & 1u);
        if (lane == 0) cnt[e * 32 + warp] = __popc(bal);
    }
    __syncthreads();
    uint32_t kept;
    const uint32_t excl = block_exclusive_sum(tid < E * 32 ? cnt[tid] : 0u, warp_sums, kept);
    if (tid < E * 32) cnt[tid] = excl;
    __syncthreads();
#pragma unroll
    for (int e = 0; e < E; ++e) {
        const int i = e * kSelThreads + tid;
        const bool f = (sel >> e & 1u) != 0;
        const uint32_t bal = __ballot_sync(0xffffffffu, f);
        const uint32_t at = cnt[e * 32 + warp] + __popc(bal & ((1u << lane) - 1u));
        if (f && at < (uint32_t)keep_stride) keep_idx[at] = i;
        if (keep_mask && i < n) keep_mask[i] = f ? 1 : 0;
    }
    if (tid == 0) n_keep[b] = (int32_t)kept;
}

// ------------------------------------------------------------------------------------------ quota
// R CTAs (a thread-block cluster) per sequence, E tokens per thread.
template <int R, int E>
__global__ void __launch_bounds__(kSelThreads)
select_quota_kernel(const float* score, const int32_t* label,
                    const int32_t* vis_len, int vis_len_uniform, int Nv_cap, int P_cap, int budget,
                    int32_t* __restrict__ keep_idx, int keep_stride, int32_t* __restrict__ n_keep,
                    uint8_t* __restrict__ keep_mask, int* __restrict__ status_word) {
    grid_dependency_launch_dependents();                  // see select_plain_kernel
    grid_dependency_wait();
    if constexpr (E * kSelThreads <= kRankTokens) {
        extern __shared__ __align__(16) uint8_t rank_dyn[];
        __shared__ RankShared sh;
        const int b = blockIdx.x, n = max(0, min(vis_len ? __ldcg(vis_len + b) : vis_len_uniform, Nv_cap));
        score += (int64_t)b * Nv_cap;
        label += (int64_t)b * Nv_cap;
        keep_idx += (int64_t)b * keep_stride;
        if (keep_mask) keep_mask += (int64_t)b * Nv_cap;
        int lab[E];
        uint32_t key[E];
#pragma unroll
        for (int e = 0; e < E; ++e) {
            const int i = e * kSelThreads + threadIdx.x;
            lab[e] = i < n ? __ldcg(label + i) : 0;
            key[e] = i < n ? order_key(__ldcg(score + i), 0) : 0u;
            if ((uint32_t)lab[e] >= (uint32_t)n) lab[e] = max(n - 1, 0);     // out-of-range labels are clamped, never indexed
        }
        if (select_by_rank<E>(lab, key, n, budget, sh, rank_dyn, keep_idx, keep_stride, n_keep + b, keep_mask, status_word)) return;
        select_by_sort(score, label, n, Nv_cap, P_cap, budget, keep_idx, keep_stride, n_keep + b, keep_mask, status_word, rank_dyn,
                       sh.warp_sums);
    } else {
        select_quota_body<R, E>(score, label, vis_len, vis_len_uniform, Nv_cap, P_cap, budget, keep_idx, keep_stride, n_keep,
                                keep_mask, status_word, blockIdx.x / R);
    }
}

typedef void (*QuotaKernel)(const float*, const int32_t*, const int32_t*, int, int, int, int, int32_t*, int, int32_t*, uint8_t*, int*);
QuotaKernel quota_kernel(int R, int E) {
    return E == 1   ? select_quota_kernel<1, 1>
           : E == 2 ? select_quota_kernel<1, 2>
           : E == 4 ? (R == 1 ? select_quota_kernel<1, 4> : select_quota_kernel<4, 4>)
           : E == 8 ? (R == 1 ? select_quota_kernel<1, 8> : select_quota_kernel<4, 8>)
           : R == 1 ? select_quota_kernel<1, 16> : R == 4 ? select_quota_kernel<4, 16> : select_quota_kernel<8, 16>;
}
size_t quota_smem(int E, int Nv_cap, int* P_cap) {
    return E * kSelThreads <= kRankTokens ? rank_or_sort_smem(Nv_cap, P_cap) : select_quota_smem(Nv_cap, P_cap);
}
size_t quota_most_smem(int E) {
    int p = 0;
    return quota_smem(E, E * kSelThreads, &p);
}
int quota_allow_smem(int R, int E) {
    static DoneOnDevice attr_done[9][17];
    return allow_dynamic_smem(quota_kernel(R, E), quota_most_smem(E), attr_done[R][E]);
}
// Beyond as many clusters as the device runs at a time the ones behind wait for a whole selection: 16 x 16384 tokens 45 us on clusters of
// eight, 26 on clusters of four; 40 x 2880 20 us on clusters of four, 13 on single CTAs.
int quota_clusters_at_once(int R, int E) {
    static KnownOnDevice known[9][17];
    return clusters_at_once(quota_kernel(R, E), R, kSelThreads, quota_most_smem(E), [=] { return quota_allow_smem(R, E); }, known[R][E]);
}

}  // namespace

int launch_select(const float* score, const int32_t* label, int B, const int32_t* vis_len, int vis_len_uniform,
                  int Nv_cap, int mode, int largest, int budget, int32_t* keep_idx, int keep_stride,
                  int32_t* n_keep, uint8_t* keep_mask, int* status_word, cudaStream_t stream, bool pdl,
                  int* clear_status) {
    if (B <= 0) return VITCOP_OK;
    cudaLaunchConfig_t cfg = {};
    cfg.gridDim = dim3(B);
    cfg.blockDim = dim3(kSelThreads);
    cfg.stream = stream;
    cudaLaunchAttribute attr[1];
    attr[0].id = cudaLaunchAttributeProgrammaticStreamSerialization;
    attr[0].val.programmaticStreamSerializationAllowed = 1;
    cfg.attrs = attr;
    cfg.numAttrs = pdl_allowed(pdl) ? 1 : 0;
    if (mode == 0) {
        const size_t smem = ((size_t)Nv_cap + 15) & ~(size_t)15;   // (at most 16 KB beside 12 KB of static arrays)
        auto kern = Nv_cap <= kSelThreads       ? select_plain_kernel<1>
                    : Nv_cap <= 4 * kSelThreads ? select_plain_kernel<4>
                    : Nv_cap <= 8 * kSelThreads ? select_plain_kernel<8> : select_plain_kernel<16>;
        static_assert(VITCOP_MAX_VISUAL_TOKENS <= 16 * kSelThreads, "tokens of the longest sample");
        cfg.dynamicSmemBytes = smem;
        KernelTimeScope timed("select_plain_kernel", stream);
        return record_cuda(cudaLaunchKernelEx(&cfg, kern, score, vis_len, vis_len_uniform, Nv_cap,
                                              largest, budget, keep_idx, keep_stride, n_keep, keep_mask, clear_status));
    }
    int P = 0;
    const int E = Nv_cap <= kSelThreads ? 1 : Nv_cap <= 2 * kSelThreads ? 2 : Nv_cap <= 4 * kSelThreads ? 4 : Nv_cap <= 8 * kSelThreads ? 8 : 16;
    const size_t smem = quota_smem(E, Nv_cap, &P);
    // CTAs per sequence: one up to 2048 tokens (the others would be done preparing when the first is done), four, and eight
    // beyond 8192; fewer where the batch would not be on the chip at once
    int R = E <= 2 ? 1 : E <= 8 ? 4 : 8;
    while (R > 1 && B > quota_clusters_at_once(R, E)) R = R == 8 ? 4 : 1;
    auto kern = quota_kernel(R, E);
    {
        const int rc = quota_allow_smem(R, E);
        if (rc != VITCOP_OK) return rc;
    }
    cudaLaunchAttribute attrs[2];
    attrs[0] = attr[0];
    int n_attr = cfg.numAttrs;
    if (R > 1) {
        attrs[n_attr].id = cudaLaunchAttributeClusterDimension;
        attrs[n_attr].val.clusterDim.x = R;
        attrs[n_attr].val.clusterDim.y = 1;
        attrs[n_attr].val.clusterDim.z = 1;
        ++n_attr;
    }
    cfg.attrs = attrs;
    cfg.numAttrs = n_attr;
    cfg.gridDim = dim3((unsigned)(B * R));
    cfg.dynamicSmemBytes = smem;
    KernelTimeScope timed("select_quota_kernel", stream);
    return record_cuda(cudaLaunchKernelEx(&cfg, kern, score, label, vis_len, vis_len_uniform, Nv_cap,
                                          P, budget, keep_idx, keep_stride, n_keep, keep_mask, status_word));
}

}  // namespace vitcop
