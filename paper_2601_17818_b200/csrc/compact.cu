// Order-preserving compaction of hidden states and the K/V cache (bit-exact row gather).
//
// A group of 32 to 256 threads per (output row, sample).  The source position of the row comes from the ascending
// keep list; the group then moves the hidden row and the row of every K and V head with 128-bit
// loads, up to eight of them issued before the first store and taken from all three tensors alike, so that
// each thread keeps several independent 16-byte requests in flight.  Dropped rows are never read.
// The group is the largest that leaves its threads four pieces each: a row of 1024 bf16 values alone (2 KB) moved by 256
// threads kept one request per thread in flight on half of them (16 x 289 such rows 16 us).
//
// With scores in place of the list every CTA selects for itself: no kernel in between, and none of the rows outside the span waits.
#include "gram.cuh"
#include "select_quota.cuh"

namespace vitcop {
namespace {

constexpr int kCompactThreads = 256;

__device__ __forceinline__ uint4 ld_stream(const uint4* p) {
    uint4 v;
    asm volatile("ld.global.nc.L1::no_allocate.v4.u32 {%0,%1,%2,%3}, [%4];"
                 : "=r"(v.x), "=r"(v.y), "=r"(v.z), "=r"(v.w)
                 : "l"(p));
    return v;
}
__device__ __forceinline__ void st_stream(uint4* p, const uint4& v) {
    asm volatile("st.global.L1::no_allocate.v4.u32 [%0], {%1,%2,%3,%4};" ::"l"(p), "r"(v.x), "r"(v.y), "r"(v.z),
                 "r"(v.w)
                 : "memory");
}

// Moves one token: its hidden row (dh8 pieces of 16 bytes, one run) and its row in each of the H heads of K and of
// V (d8 pieces per head, heads head_in / head_out pieces apart).  The pieces of all three tensors form one index
// space, so that a thread has up to eight loads from any of them in flight before its first store: the row costs
// one round trip to memory, not one per tensor.  Null tensors are skipped.
template <int G>
__device__ __forceinline__ void copy_token(int lane, const uint4* __restrict__ hid_src, uint4* __restrict__ hid_dst, int dh8,
                                           const uint4* __restrict__ k_src, uint4* __restrict__ k_dst,
                                           const uint4* __restrict__ v_src, uint4* __restrict__ v_dst, int H, int d8,
                                           int d8_shift, int64_t head_in, int64_t head_out) {
    const int n_hid = hid_src ? dh8 : 0;
    const int n_kv = H * d8;
    const int n_k = k_src ? n_kv : 0;
    const int total = n_hid + n_k + (v_src ? n_kv : 0);
    constexpr int kInFlight = 8;
    for (int q0 = lane; q0 < total; q0 += kInFlight * G) {
        uint4 v[kInFlight];
        uint4* d[kInFlight];
#pragma unroll
        for (int u = 0; u < kInFlight; ++u) {
            int q = q0 + u * G;
            d[u] = nullptr;
            if (q < total) {
                if (q < n_hid) {
                    v[u] = ld_stream(hid_src + q);
                    d[u] = hid_dst + q;
                } else {
                    q -= n_hid;
                    const bool is_k = q < n_k;
                    if (!is_k) q -= n_k;
                    const int head = d8_shift >= 0 ? q >> d8_shift : q / d8;
                    const int e = q - head * d8;
                    v[u] = ld_stream((is_k ? k_src : v_src) + head * head_in + e);
                    d[u] = (is_k ? k_dst : v_dst) + head * head_out + e;
                }
            }
        }
#pragma unroll
        for (int u = 0; u < kInFlight; ++u)
            if (d[u]) st_stream(d[u], v[u]);
    }
}

// The k tokens of smallest (score, index) of n <= 32 E, in ascending order, to list, by one warp: the cut is found bit by bit
// from the first in which two keys differ, until as many tokens are left as are wanted.  (Ranks counted by all threads of the CTA: as
// fast up to 128 tokens, 256 tokens x 32 heads of 128 8.8 / 9.9 us.)
template <int E>
__device__ __forceinline__ void warp_smallest(const float* score, int n, int k, uint16_t* list) {
    const int lane = threadIdx.x & 31;
    uint32_t key[E], in = 0, sel = 0;                      // in: tokens (bit e: token 32 e + lane) on the cut; sel: chosen ones
    float s[E];
#pragma unroll
    for (int e = 0; e < E; ++e) s[e] = e * 32 + lane < n ? __ldcg(score + e * 32 + lane) : 0.f;
    uint32_t lo = 0xFFFFFFFFu, hi = 0u;
#pragma unroll
    for (int e = 0; e < E; ++e) {
        key[e] = order_key(s[e], 0);
        if (e * 32 + lane < n) {
            in |= 1u << e;
            lo = min(lo, key[e]);
            hi = max(hi, key[e]);
        }
    }
    int cands = n, left = k;
    if (k > 0 && k < n) {
        lo = __reduce_min_sync(0xffffffffu, lo);
        hi = __reduce_max_sync(0xffffffffu, hi);
        for (int bit = 31 - __clz(lo ^ hi); bit >= 0 && cands != left; --bit) {
            uint32_t ones = 0;
#pragma unroll
            for (int e = 0; e < E; ++e) ones |= (key[e] >> bit & 1u) << e;
            const uint32_t zeros = in & ~ones;
            const int c = (int)__reduce_add_sync(0xffffffffu, (unsigned)__popc(zeros));
            if (left <= c) {
                in = zeros;
                cands = c;
            } else {
                sel |= zeros;
                in &= ones;
                left -= c;
                cands -= c;
            }
        }
    }
    // tokens of equal keys are left: the first ones
    const uint32_t lt = (1u << lane) - 1u;
    int equal = 0, at = 0;
#pragma unroll
    for (int e = 0; e < E; ++e) {
        if (e * 32 >= n) break;
        const bool on = (in >> e & 1u) != 0;
        const uint32_t tie = __ballot_sync(0xffffffffu, on);
        const bool mine = (sel >> e & 1u) != 0 || (on && equal + __popc(tie & lt) < left);
        const uint32_t all = __ballot_sync(0xffffffffu, mine);
        if (mine) list[at + __popc(all & lt)] = (uint16_t)(e * 32 + lane);
        equal += __popc(tie);
        at += __popc(all);
    }
}

template <int G>
__global__ void __launch_bounds__(kCompactThreads, G == kCompactThreads ? 4 : 3)
compact_kernel(const uint4* __restrict__ hidden, const uint4* __restrict__ K, const uint4* __restrict__ V, int B, int H, int N,
               int d8, int dh8, int d8_shift, const int32_t* seq_len, int vis_start,
               const int32_t* vis_len, int vis_len_uniform, const int32_t* keep_idx,
               int keep_stride, const int32_t* n_keep, uint4* __restrict__ hidden_out,
               uint4* __restrict__ K_out, uint4* __restrict__ V_out, int Ncap, int32_t* __restrict__ kept_pos,
               int32_t* __restrict__ out_len, int early) {
    // A copy that stands alone reads rows that the kernel in front may still be writing, so only its launch overlaps (a
    // selection and a copy of 16 x 576 rows: 23.7 -> 19.1 us with both launched this way).
    if (!early) grid_dependency_wait();
    // CTAs are handed out sample by sample within a row: all the rows in front of the visual span, which need not
    // wait for the selection, start before the rows that do
    const int rg = (int)(blockIdx.x / (unsigned)B);
    const int b = (int)(blockIdx.x - (unsigned)rg * (unsigned)B);
    // (uniform over the CTA where one row takes all of it)
    const int r = G == kCompactThreads ? rg : rg * (kCompactThreads / G) + (int)threadIdx.x / G;
    const int lane = G == kCompactThreads ? threadIdx.x : threadIdx.x % G;
    const int L = seq_len ? min(__ldcg(seq_len + b), N) : N;
    const int64_t head_in = (int64_t)N * d8, head_out = (int64_t)Ncap * d8;
    // A row in front of the visual span keeps its place whatever the selection turns out to be: it is copied
    // before this kernel waits for the selection, while the kernels that produce it are still running.  (The
    // tensors copied here are inputs of the whole call, complete before its first kernel started.)
    const bool prefix_row = r < min(vis_start, L) && r < Ncap;
    if (prefix_row) {
        copy_token<G>(lane, hidden ? hidden + ((int64_t)b * N + r) * dh8 : nullptr, hidden_out + ((int64_t)b * Ncap + r) * dh8, dh8,
                   K ? K + ((int64_t)b * H * N + r) * d8 : nullptr, K_out + ((int64_t)b * H * Ncap + r) * d8,
                   V ? V + ((int64_t)b * H * N + r) * d8 : nullptr, V_out + ((int64_t)b * H * Ncap + r) * d8, H, d8,
                   d8_shift, head_in, head_out);
        if (kept_pos && lane == 0) kept_pos[(int64_t)b * Ncap + r] = r;
        if (r != 0) return;                                // row 0 still reports the sample's new length
    }
    grid_dependency_wait();
    // (the row's entry in the list travels with the list's length, whether there is one or not; of one list for all samples,
    // stride 0, nobody knows the end but the length)
    const int slot = r - vis_start;
    const int32_t* const entry = keep_idx + (int64_t)b * keep_stride + slot;
    int ki = slot >= 0 && slot < keep_stride ? __ldcg(entry) : 0;
    int nv = vis_len ? __ldcg(vis_len + b) : vis_len_uniform;
    nv = max(0, min(nv, L - vis_start));
    const int nk = max(0, min(min(__ldcg(n_keep + b), keep_stride > 0 ? keep_stride : nv), nv));
    const int olen = L - nv + nk;
    if (r == 0 && lane == 0) out_len[b] = olen;
    if (r >= Ncap || prefix_row) return;
    if (r >= olen) {
        if (kept_pos && lane == 0) kept_pos[(int64_t)b * Ncap + r] = -1;
        return;
    }
    int src_row;
    if (r < vis_start) src_row = r;
    else if (r < vis_start + nk) {
        if (keep_stride == 0) ki = __ldcg(entry);
        ki = max(0, min(ki, nv - 1));                     // a corrupt index can never leave the span
        src_row = vis_start + ki;
    } else src_row = r - nk + nv;
    if (kept_pos && lane == 0) kept_pos[(int64_t)b * Ncap + r] = src_row;

    copy_token<G>(lane, hidden ? hidden + ((int64_t)b * N + src_row) * dh8 : nullptr, hidden_out + ((int64_t)b * Ncap + r) * dh8,
               dh8, K ? K + ((int64_t)b * H * N + src_row) * d8 : nullptr, K_out + ((int64_t)b * H * Ncap + r) * d8,
               V ? V + ((int64_t)b * H * N + src_row) * d8 : nullptr, V_out + ((int64_t)b * H * Ncap + r) * d8, H, d8,
               d8_shift, head_in, head_out);
}

// The same with the selection inside, from the scores of at most TOKENS tokens a sample; the first CTA of a sample writes the list.  (A
// kernel of its own: four more parameters cost each launch of the other one 0.4 us of the caller's time.)
template <int G, int TOKENS>
__global__ void __launch_bounds__(kCompactThreads, G == kCompactThreads ? 4 : 3)
select_compact_kernel(const uint4* __restrict__ hidden, const uint4* __restrict__ K, const uint4* __restrict__ V, int B, int H, int N,
                      int d8, int dh8, int d8_shift, const int32_t* seq_len, int vis_start, const int32_t* vis_len, int vis_len_uniform,
                      const float* score, int keep_stride, int budget, int32_t* __restrict__ keep_out, int32_t* __restrict__ n_keep_out,
                      uint4* __restrict__ hidden_out, uint4* __restrict__ K_out, uint4* __restrict__ V_out, int Ncap,
                      int32_t* __restrict__ kept_pos, int32_t* __restrict__ out_len) {
    const int rg = (int)(blockIdx.x / (unsigned)B);
    const int b = (int)(blockIdx.x - (unsigned)rg * (unsigned)B);
    const int r = G == kCompactThreads ? rg : rg * (kCompactThreads / G) + (int)threadIdx.x / G;
    const int lane = G == kCompactThreads ? threadIdx.x : threadIdx.x % G;
    const int L = seq_len ? min(__ldcg(seq_len + b), N) : N;
    const int64_t head_in = (int64_t)N * d8, head_out = (int64_t)Ncap * d8;
    const auto copy_row = [&](int from) {
        copy_token<G>(lane, hidden ? hidden + ((int64_t)b * N + from) * dh8 : nullptr, hidden_out + ((int64_t)b * Ncap + r) * dh8,
                      dh8, K ? K + ((int64_t)b * H * N + from) * d8 : nullptr, K_out + ((int64_t)b * H * Ncap + r) * d8,
                      V ? V + ((int64_t)b * H * N + from) * d8 : nullptr, V_out + ((int64_t)b * H * Ncap + r) * d8, H, d8,
                      d8_shift, head_in, head_out);
        if (kept_pos && lane == 0) kept_pos[(int64_t)b * Ncap + r] = from;
    };
    // How many tokens stay follows from the lengths: rows behind the span have their place as early as those in front of it.
    __shared__ uint16_t list[TOKENS];
    const int len = vis_len ? __ldcg(vis_len + b) : vis_len_uniform;
    const int n = max(0, min(len, keep_stride)), k = max(0, min(budget, n));
    const int nv = max(0, min(len, L - vis_start)), nk = min(k, nv), olen = L - nv + nk;
    const bool chosen = r >= vis_start && r < vis_start + nk;
    if (r < Ncap && !chosen) {
        if (r < olen) copy_row(r < vis_start ? r : r - nk + nv);
        else if (kept_pos && lane == 0) kept_pos[(int64_t)b * Ncap + r] = -1;
    }
    constexpr int kRows = kCompactThreads / G;
    if (rg != 0 && (rg * kRows >= vis_start + nk || rg * kRows + kRows <= vis_start)) return;      // (uniform over the CTA)
    grid_dependency_wait();
    if (threadIdx.x < 32) warp_smallest<TOKENS / 32>(score + (int64_t)b * keep_stride, n, k, list);
    __syncthreads();
    if (rg == 0) {
        if ((int)threadIdx.x < k) keep_out[(int64_t)b * keep_stride + threadIdx.x] = (int32_t)list[threadIdx.x];
        if (threadIdx.x == 0) {
            n_keep_out[b] = k;
            out_len[b] = olen;
        }
    }
    if (r < Ncap && chosen) copy_row(vis_start + min((int)list[r - vis_start], nv - 1));
}

// How many threads move a row of so many pieces, and how many CTAs that makes.
struct Split {
    int group;
    long long ctas;
    Split(long long pieces, int B, int Ncap) {
        group = kCompactThreads;
        while (group > 32 && pieces < 4LL * group) group /= 2;
        // rows past min(N, Ncap) cannot exist; one extra CTA row keeps out_len written when Ncap == 0
        const int rows = Ncap > 0 ? Ncap : 1, per_cta = kCompactThreads / group;
        ctas = (long long)B * ((rows + per_cta - 1) / per_cta);
    }
};

}  // namespace

// A copy of few rows is the end of a chain of short kernels: one link less outweighs that every CTA selects (whole calls by
// themselves / in a graph, selection as a kernel -> in the copy, us: 1 x 128 tokens x 32 heads of 128 9.1 -> 6.8 / 7.5 -> 6.5, 1 x 256
// 9.4 -> 8.6 / 8.6 -> 8.6, 4 x 256 12.1 -> 11.4 / 11.6 -> 11.3).  Not where the copy fills the chip (8 x 256: 22.1 -> 23.2, 16 x 256 x 4 of 128
// 16.9 -> 21.4), and not for longer lists (1 x 576 11.2 -> 12.7).
bool compact_selects(bool hidden, bool V, int B, int H, int d, int Dh, int Nv_cap, int Ncap) {
    const Split cut((hidden ? Dh / 8 : 0) + (long long)H * (d / 8) * (V ? 2 : 1), B, Ncap);
    return Nv_cap <= 256 && cut.ctas <= 3LL * gram_num_sms();
}

int launch_compact(const void* hidden, const void* K, const void* V, int B, int H, int N, int d, int Dh,
                   const int32_t* seq_len, int vis_start, const int32_t* vis_len, int vis_len_uniform,
                   const int32_t* keep_idx, int keep_stride, const int32_t* n_keep, void* hidden_out, void* K_out,
                   void* V_out, int Ncap, int32_t* kept_pos, int32_t* out_len, cudaStream_t stream, bool early,
                   const SmallestJob* smallest) {
    if (B <= 0) return VITCOP_OK;
    const int d8 = d / 8;
    int d8_shift = -1;                                    // log2(d / 8) when that is a power of two
    if (d8 > 0 && (d8 & (d8 - 1)) == 0)
        for (d8_shift = 0; (1 << d8_shift) < d8; ++d8_shift) {}
    cudaLaunchConfig_t cfg = {};
    const Split cut((hidden ? Dh / 8 : 0) + (long long)H * d8 * ((K ? 1 : 0) + (V ? 1 : 0)), B, Ncap);
    const int G = cut.group;
    cfg.gridDim = dim3((unsigned)cut.ctas);
    cfg.blockDim = dim3(kCompactThreads);
    cfg.stream = stream;
    cudaLaunchAttribute attr[1];
    attr[0].id = cudaLaunchAttributeProgrammaticStreamSerialization;
    attr[0].val.programmaticStreamSerializationAllowed = 1;
    cfg.attrs = attr;
    cfg.numAttrs = pdl_allowed(true) ? 1 : 0;
    KernelTimeScope timed("compact_kernel", stream);       // (either kernel: a selection inside counts as part of the copy)
    const uint4 *hid = static_cast<const uint4*>(hidden), *k = static_cast<const uint4*>(K), *v = static_cast<const uint4*>(V);
    uint4 *const hid_out = static_cast<uint4*>(hidden_out), *const k_out = static_cast<uint4*>(K_out), *const v_out = static_cast<uint4*>(V_out);
    if (smallest) {
        const bool few = keep_stride <= 128;
        auto kern = G == 256   ? (few ? select_compact_kernel<256, 128> : select_compact_kernel<256, 256>)
                    : G == 128 ? (few ? select_compact_kernel<128, 128> : select_compact_kernel<128, 256>)
                    : G == 64  ? (few ? select_compact_kernel<64, 128> : select_compact_kernel<64, 256>)
                               : (few ? select_compact_kernel<32, 128> : select_compact_kernel<32, 256>);
        return record_cuda(cudaLaunchKernelEx(&cfg, kern, hid, k, v, B, H, N, d8, Dh / 8, d8_shift, seq_len, vis_start, vis_len,
                                              vis_len_uniform, smallest->score, keep_stride, smallest->budget, smallest->keep,
                                              smallest->n_keep, hid_out, k_out, v_out, Ncap, kept_pos, out_len));
    }
    auto kern = G == 256 ? compact_kernel<256> : G == 128 ? compact_kernel<128> : G == 64 ? compact_kernel<64> : compact_kernel<32>;
    return record_cuda(cudaLaunchKernelEx(&cfg, kern, hid, k, v, B, H, N, d8, Dh / 8, d8_shift, seq_len, vis_start, vis_len,
                                          vis_len_uniform, keep_idx, keep_stride, n_keep, hid_out, k_out, v_out, Ncap, kept_pos, out_len,
                                          early ? 1 : 0));
}

}  // namespace vitcop
