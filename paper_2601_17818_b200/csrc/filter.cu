// Redundancy filter = Visual Information Clustering (Algorithm 2, Eq. 2 and Eq. 3) on one B200.
//
// Pipeline (one stream, no host synchronisation; consecutive kernels overlap through programmatic dependent
// launch, each waiting for its predecessor before it reads what that one wrote):
//   1. Gram diagonal          the diagonal tiles only: g_ii -> per-token factors (cosine: 1/sqrt(g_ii);
//                             euclid: g_ii), from the same tensor-core arithmetic as every g_ij (gram.cu)
//   2. density_sweep_kernel   Gram tiles on the tensor cores (density.cu); the epilogue turns each tile into
//                             squared distances, exp(-(d/d_c)^2) and partial sums of Eq. 2, keeps the Gram values in the
//                             workspace and leaves the smallest distance of every token to every block of 32 tokens
//   3. rho_reduce_kernel      fixed-order sum of the partials -> rho (bit-reproducible)
//   4. nearest_denser_kernel  (nearest.cu) searches the few blocks that can hold it for each token's nearest denser
//      nearest_left_kernel    token inside the spatial radius (Eq. 3): packed (d^2, j)
//   (2-4 run sample group by sample group where the Gram values of the whole batch would take more than 1.5 GB)
//   5. vic_finalize_kernel    gamma = rho * delta, radix-select of the centres, pointer jumping over the
//                             parent forest, orphan fallback, labels (Algorithm 2, steps 3-4)
// Small problems replace 1-4 by gram_resident_kernel (gram.cu): one pass over the Gram tiles, accumulators kept in
// tensor memory.
#include "density.cuh"
#include "gram.cuh"

namespace vitcop {
namespace {

// ------------------------------------------------------------------------------------------------
// small kernels
// ------------------------------------------------------------------------------------------------
// rho[b,i] = sum of the partials of the density sweep in a fixed order (reproducible bits): first the later tokens, 256 at a
// time (a tile's columns: the sum of its two 128-token blocks), then the earlier ones, one 128-token block after the other, to
// the end of the token's tile (blocks that hold none of them count as zero).  On samples with T + TI <= 64 tiles and blocks (up to
// 5376 tokens) the entries are added one by one; on longer ones in four equal parts, whose sums are then added.  One CTA per 32
// tokens: its warps fetch the entries, all of them in one trip to memory, and the sums are taken from shared memory.  (One thread
// per token walking its list paid a trip for every sixteen entries.)
// blk_rho[b,k]: bits of the largest density among the tokens of block k (densities are not negative, their bit patterns order
// like the values).  tok[b,i]: what the search needs of a token, in one 16-byte load.
constexpr int kRhoThreads = 256;
constexpr int kRhoOneByOne = 64;
// the longest list: (T - tile) + min(TI, 2 (tile + 1)) entries, most at the last tile
constexpr int kRhoEntries = VITCOP_MAX_VISUAL_TOKENS / kGramBM + 1;
__global__ void __launch_bounds__(kRhoThreads)
rho_reduce_kernel(const __grid_constant__ SweepArgs g, int metric, float* __restrict__ rho_user) {
    constexpr int kWarps = kRhoThreads / 32;
    __shared__ float entry[kRhoEntries][kBlk];
    __shared__ float parts[4][kBlk];
    grid_dependency_launch_dependents();
    grid_dependency_wait();
    const SweepTiling& t = g.t;
    const int n = g.n;
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    const int blk = blockIdx.x, b = blockIdx.y, i = blk * kBlk + lane;
    const size_t at = (size_t)b * n + i;
    float4 tok = make_float4(0.f, 0.f, 0.f, 0.f);
    if (warp == 0 && i < n) {
        tok.x = __ldcg((metric == 1 ? g.a : g.w) + at);
        if (g.pos && g.tau2 >= 0.f) {
            const float2 p = *reinterpret_cast<const float2*>(g.pos + 2 * at);
            tok.z = p.x;
            tok.w = p.y;
        }
    }
    if (blk == 0 && b == 0 && threadIdx.x == 0) *g.n_left = 0;       // for the search behind this kernel
    if (blk == 0 && b == 0 && warp == 1 && any_gave_up(g.status, g.diag_reports) && lane == 0) atomicMax(g.status, VITCOP_ERR_TIMEOUT);
    const int own = blk * kBlk / kGramBM, tile = own / 2;
    const int rows = t.T - tile;                           // entries on the row side, then min(TI, 2 (tile + 1)) more
    const int entries = rows + min(t.TI, 2 * (tile + 1));
    if (i < n) {
        const float* p = g.part + (size_t)b * t.slots() * t.n_pad + i;
        auto slot = [&](int k) { return __ldcg(p + (size_t)k * t.n_pad); };
#pragma unroll 6
        for (int e = warp; e < entries; e += kWarps) {
            float v = 0.f, v2 = 0.f;
            if (e < rows) {
                const int k = 2 * (tile + e);
                if (k >= own) v = slot(k);
                if (k + 1 >= own && k + 1 < t.TI) v2 = slot(k + 1);
            } else {
                const int k = e - rows;
                if (k <= own) v = slot(k == own ? t.TI : k);
            }
            entry[e][lane] = v + v2;
        }
    }
    __syncthreads();
    const int nparts = t.T + t.TI > kRhoOneByOne ? 4 : 1;
    if (warp < nparts) {
        const int per = (entries + nparts - 1) / nparts, e1 = min(entries, (warp + 1) * per);
        float s = 0.f;
#pragma unroll 8
        for (int e = warp * per; e < e1; ++e) s += entry[e][lane];
        parts[warp][lane] = s;
    }
    __syncthreads();
    if (warp != 0) return;
    float s = parts[0][lane];
    for (int q = 1; q < nparts; ++q) s += parts[q][lane];
    if (i < n) {
        g.rho[at] = s;
        if (rho_user) rho_user[at] = s;
        tok.y = s;
    }
    g.tok[(size_t)b * t.n_pad + i] = tok;
    const uint32_t m = __reduce_max_sync(0xffffffffu, i < n ? __float_as_uint(s) : 0u);
    if (lane == 0) g.blk_rho[(size_t)b * t.n_blk() + blk] = m;
}

// ------------------------------------------------------------------------------------------------
// Centres, forest roots and labels: one CTA per sample.
// ------------------------------------------------------------------------------------------------
// The CTA runs alone on its SM, so what counts is the number of dependent steps, not throughput: every thread holds its tokens'
// keys in registers, all global loads are in flight together, the cut among the keys is found with one or two histogram
// passes of 11 bits that start at the highest bit in which two keys differ, and what is left in the cut's bin is ranked by
// counting.  (8-bit passes over the whole 64-bit key with ordered scans for ties and for the list of centres: 9.2 us on 576
// tokens, 14 on 2880, 38 on 16384; the list is needed for surplus orphans only and is built when there are any.)
constexpr int kFinThreads = 1024;
constexpr int kFinBits = 11, kFinBins = 1 << kFinBits;
constexpr int kFinRankLanes = 4;
constexpr int kFinRank = kFinThreads / kFinRankLanes;      // bins of up to this many keys are ranked by counting

// Dynamic shared memory: nxt[n] (uint16), isc[n] (uint8), centre list[nc] (uint16; surplus orphans).  E: tokens per thread.
constexpr size_t finalize_smem(int n, int nc) { return (((size_t)n + 15) & ~(size_t)15) * 3 + (size_t)(nc > 0 ? nc : 1) * 2 + 16; }
template <int E>
__global__ void __launch_bounds__(kFinThreads)
vic_finalize_kernel(const uint16_t* __restrict__ feat, int n, int D, int n_centers, const float* rho, const unsigned long long* best,
                    const float* w, const float* a, int32_t* __restrict__ label, int32_t* __restrict__ n_clusters,
                    float* __restrict__ delta2_user, int32_t* __restrict__ parent_user) {
    extern __shared__ __align__(16) uint8_t fin_smem[];
    const int n_al = (n + 15) & ~15;
    uint16_t* nxt = reinterpret_cast<uint16_t*>(fin_smem);
    uint8_t* isc = fin_smem + (size_t)n_al * 2;
    uint16_t* centres = reinterpret_cast<uint16_t*>(fin_smem + (size_t)n_al * 3);
    __shared__ uint32_t hist[kFinBins];
    __shared__ unsigned long long cand_key[kFinRank];
    __shared__ uint16_t cand_idx[kFinRank];
    __shared__ uint32_t warp_sums[32];
    __shared__ uint32_t s_lo, s_hi, s_digit, s_krem, s_count, s_cands;
    __shared__ unsigned long long orph_best[kFinThreads];
    __shared__ int orph_list[kFinThreads];
    __shared__ int orph_cnt, centre_cnt;

    const int tid = threadIdx.x, lane = tid & 31;
    hist[tid] = 0;
    hist[tid + kFinThreads] = 0;
    if (tid == 0) { s_lo = 0xFFFFFFFFu; s_hi = 0u; s_cands = 0u; centre_cnt = 0; }
    static_assert(kFinBins == 2 * kFinThreads, "two bins per thread");
    grid_dependency_launch_dependents();
    grid_dependency_wait();
    const int b = blockIdx.x;
    rho += (size_t)b * n;
    best += (size_t)b * n;
    w += (size_t)b * n;
    a += (size_t)b * n;
    label += (size_t)b * n;
    feat += (size_t)b * n * D;
    if (delta2_user) delta2_user += (size_t)b * n;
    if (parent_user) parent_user += (size_t)b * n;
    const int nc = min(n_centers, n);

    // (Loads of what the preceding kernels wrote: pointers without __restrict__, so that nothing lets the compiler move one in
    // front of the wait.)
    // rank key, ascending = better centre candidate: ( ~( orphan ? 0xFFFFFFFF : gamma ), ~rho, index )
    uint32_t hi[E];
    {
        unsigned long long p[E];
        float r[E];
#pragma unroll
        for (int e = 0; e < E; ++e) {
            const int i = e * kFinThreads + tid;
            p[e] = i < n ? __ldcg(best + i) : 0ull;
            r[e] = i < n ? __ldcg(rho + i) : 0.f;
        }
        uint32_t lo_k = 0xFFFFFFFFu, hi_k = 0u;
#pragma unroll
        for (int e = 0; e < E; ++e) {
            const int i = e * kFinThreads + tid;
            if (i < n) {
                const bool orphan = p[e] == ~0ull;
                const float d2 = orphan ? __int_as_float(0x7f800000) : __uint_as_float((uint32_t)(p[e] >> 32));
                const int par = orphan ? -1 : (int)(uint32_t)(p[e] & 0xFFFFFFFFull);
                if (delta2_user) delta2_user[i] = d2;
                if (parent_user) parent_user[i] = par;
                nxt[i] = (uint16_t)((par < 0 || par >= n) ? i : par);
                hi[e] = ~(orphan ? 0xFFFFFFFFu : __float_as_uint(r[e] * sqrtf(d2)));
                lo_k = min(lo_k, hi[e]);
                hi_k = max(hi_k, hi[e]);
            }
        }
        lo_k = __reduce_min_sync(0xffffffffu, lo_k);
        hi_k = __reduce_max_sync(0xffffffffu, hi_k);
        __syncthreads();                                   // (s_lo, s_hi and the histogram are set)
        if (lane == 0 && lo_k <= hi_k) {
            atomicMin(&s_lo, lo_k);
            atomicMax(&s_hi, hi_k);
        }
    }
    __syncthreads();

    // ---- the nc smallest keys.  `in`: tokens of this thread (bit e) that still are on the cut; `sel`: chosen ones.
    uint32_t in = 0, sel = 0, ranked = 0;                  // ranked: how many of the listed candidates are wanted
#pragma unroll
    for (int e = 0; e < E; ++e)
        if (e * kFinThreads + tid < n) in |= 1u << e;
    if (nc >= n) {
        sel = in;
    } else if (nc > 0) {
        uint32_t krem = (uint32_t)nc;
        int word = 0, top = 32 - __clz(s_lo ^ s_hi);       // word of the key, bits of it not yet looked at
        for (;;) {
            while (top == 0) top = ++word == 2 ? 14 : 32;  // (indices differ: the last word settles everything)
            const int shift = top > kFinBits ? top - kFinBits : 0;
            auto digit = [&](int e) {
                const int i = e * kFinThreads + tid;
                const uint32_t k = word == 0 ? hi[e] : word == 1 ? ~__float_as_uint(__ldcg(rho + i)) : (uint32_t)i;
                return (k >> shift) & ((1u << (top - shift)) - 1u);
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
                break;
            }
            if (count <= (uint32_t)kFinRank) {
                // few left: listed, and ranked below
#pragma unroll
                for (int e = 0; e < E; ++e) {
                    if (in >> e & 1u) {
                        const int i = e * kFinThreads + tid;
                        const uint32_t at = atomicAdd(&s_cands, 1u);
                        cand_key[at] = ((unsigned long long)hi[e] << 32) | (unsigned long long)~__float_as_uint(__ldcg(rho + i));
                        cand_idx[at] = (uint16_t)i;
                    }
                }
                ranked = krem;
                break;
            }
            __syncthreads();                               // (s_digit .. are rewritten)
        }
    }
    // ---- centres are roots; an orphan is one already
#pragma unroll
    for (int e = 0; e < E; ++e) {
        const int i = e * kFinThreads + tid;
        if (i < n) {
            const bool f = (sel >> e & 1u) != 0;
            isc[i] = f ? 1 : 0;
            if (f) nxt[i] = (uint16_t)i;
        }
    }
    __syncthreads();
    if (ranked > 0) {                                      // (uniform) four threads per candidate count the better ones
        const int c = tid / kFinRankLanes, cands = (int)s_cands;
        uint32_t rank = 0;
        unsigned long long mine = 0ull;
        int idx = 0;
        if (c < cands) {
            mine = cand_key[c];
            idx = cand_idx[c];
            for (int o = tid % kFinRankLanes; o < cands; o += kFinRankLanes)
                rank += (cand_key[o] < mine || (cand_key[o] == mine && cand_idx[o] < idx)) ? 1u : 0u;
        }
#pragma unroll
        for (int off = 1; off < kFinRankLanes; off <<= 1) rank += __shfl_xor_sync(0xffffffffu, rank, off);
        if (c < cands && tid % kFinRankLanes == 0 && rank < ranked) {
            isc[idx] = 1;
            nxt[idx] = (uint16_t)idx;
        }
        __syncthreads();
    }
    // ---- forest roots by pointer jumping: any value read is an ancestor, roots are fixed points
    for (int round = 0; round < 16; ++round) {
        int changed = 0;
#pragma unroll
        for (int e = 0; e < E; ++e) {
            const int i = e * kFinThreads + tid;
            if (i < n) {
                int p = nxt[i];
                const int q = nxt[p];
                if (q != p) {
                    p = nxt[q];
                    nxt[i] = nxt[p];
                    changed = 1;
                }
            }
        }
        if (!__syncthreads_or(changed)) break;
    }
    // ---- a root that is an orphan but not a centre joins the nearest centre (feature distance)
    int any_surplus = 0;
#pragma unroll
    for (int e = 0; e < E; ++e) {
        const int i = e * kFinThreads + tid;
        if (i < n && !isc[i] && nxt[i] == i) any_surplus = 1;
    }
    if (nc > 0 && __syncthreads_or(any_surplus)) {
        // Surplus orphans are rare but each needs its distance to every centre: they are listed, kFinThreads tokens at a time,
        // and the (orphan, centre) pairs are spread over all warps; the nearest centre wins through a packed minimum
        // (distance bits, then the lower centre).
#pragma unroll
        for (int e = 0; e < E; ++e) {
            const int i = e * kFinThreads + tid;
            if (i < n && isc[i]) centres[atomicAdd(&centre_cnt, 1)] = (uint16_t)i;
        }
        for (int base = 0; base < n; base += kFinThreads) {
            __syncthreads();                                        // the previous round's list has been consumed
            if (tid == 0) orph_cnt = 0;
            __syncthreads();
            const int o = base + tid;
            if (o < n && !isc[o] && nxt[o] == o) {
                const int at = atomicAdd(&orph_cnt, 1);
                orph_list[at] = o;
                orph_best[at] = ~0ull;
            }
            __syncthreads();
            const int pairs = orph_cnt * nc;
            for (int pr = tid >> 5; pr < pairs; pr += kFinThreads / 32) {
                const int e = pr / nc, q = pr - e * nc;
                const int oo = orph_list[e], c = centres[q];
                const uint16_t* fo = feat + (size_t)oo * D;
                const uint16_t* fc = feat + (size_t)c * D;
                float dot = 0.f;
                for (int k = lane * 2; k < D; k += 64) {
                    const uint32_t u = *reinterpret_cast<const uint32_t*>(fo + k);
                    const uint32_t v = *reinterpret_cast<const uint32_t*>(fc + k);
                    dot = fmaf(bf16lo(u), bf16lo(v), dot);
                    dot = fmaf(bf16hi(u), bf16hi(v), dot);
                }
#pragma unroll
                for (int off = 16; off > 0; off >>= 1) dot += __shfl_xor_sync(0xffffffffu, dot, off);
                const float d2 = fmaxf(0.f, fmaf(-2.f, (dot * w[oo]) * w[c], a[oo] + a[c]));
                if (lane == 0)
                    atomicMin(&orph_best[e], ((unsigned long long)__float_as_uint(d2) << 32) | (unsigned long long)(uint32_t)c);
            }
            __syncthreads();
            if (tid < orph_cnt) nxt[orph_list[tid]] = (uint16_t)(orph_best[tid] & 0xFFFFFFFFull);   // the adopted centre
        }
        __syncthreads();
    }
    // ---- labels
#pragma unroll
    for (int e = 0; e < E; ++e) {
        const int i = e * kFinThreads + tid;
        if (i < n) {
            const int root = nxt[i];
            label[i] = isc[root] ? root : (int)nxt[root];           // (a surplus orphan's entry is the centre that adopted it)
        }
    }
    if (tid == 0) n_clusters[b] = nc;
}

// In front of the one-kernel sweep: status word, barrier counter and published factors.  The sweep's CTAs have nothing to meet by
// until these are cleared, and the launch's own barrier has no time limit.  Latency: the sweep starts beside this kernel and waits
// for it behind its first MMAs, so 1 x 576 tokens (whole call) take 30.8 us where a memset takes 32.2 and clearing inside the sweep,
// behind the launch's barrier, 32.7; 16 x 576 56.1, 57.2 and 55.2.
// It lets the sweep go only behind its own wait: the sweep's loads, its K-norm and the early parts of the kernels behind it rest on
// everything queued before the call being complete by then.
constexpr int kClearThreads = 256;
__global__ void __launch_bounds__(kClearThreads) clear_kernel(uint4* __restrict__ words, unsigned pieces) {
    grid_dependency_wait();
    grid_dependency_launch_dependents();
    const unsigned i = blockIdx.x * kClearThreads + threadIdx.x;
    if (i < pieces) words[i] = make_uint4(0u, 0u, 0u, 0u);
}

// ------------------------------------------------------------------------------------------------
// host side
// ------------------------------------------------------------------------------------------------
// Workspace of the filter: status block | for the one-kernel sweep the tokens' published factors [B, n] | w | a | rho | best |
// rho partials [B, slots, n_pad] | bounding boxes of the row blocks' positions | and, for problems too large for the one-kernel
// sweep, what is kept of one group of samples (SweepGroupWs).  The first kernel of a call clears the status block, in front of the
// one-kernel sweep the published factors too.  Words of the status block: 0 status, 2 grid barrier.
// A group is as large as the workspace allows, so every workspace serves that holds one sample of it; the size asked for holds
// all samples, or as many as fit 1.5 GB (8 x 2880 tokens take 175 MB: one sample at a time would leave half of the SMs without
// work).  Neither the size asked for nor the least one ever falls when the batch or the samples grow: a workspace for a larger
// problem serves a smaller one.
struct FilterWs {
    size_t off_ready, off_w, off_a, off_rho, off_best, off_part, off_bbox, off_group, total, least;
    bool resident;
    FilterWs(int B, int n) {
        size_t o = kStatusBytes;
        const size_t bn = (size_t)B * n;
        resident = gram_fits_resident(B, n);
        off_ready = o; o += resident ? align_up(bn * 4, 256) : 0;
        off_w = o;    o += align_up(bn * 4, 256);
        off_a = o;    o += align_up(bn * 4, 256);
        off_rho = o;  o += align_up(bn * 4, 256);
        off_best = o; o += align_up(bn * 8, 256);
        // one-kernel sweep: units of 64 columns take the most slots; density sweep: make_sweep_tiling
        const GramTiling t = make_gram_tiling(n);
        const size_t slots = resident ? 5 * (size_t)t.TI : (size_t)make_sweep_tiling(n).slots();
        off_part = o; o += align_up((size_t)B * slots * t.n_pad * 4, 256);
        off_bbox = o;   o += align_up((size_t)B * t.TI * sizeof(float4), 256);
        off_group = least = total = o;
        if (B > 0 && n > 0 && !resident) {
            const size_t one = SweepGroupWs(1, n).total, all = SweepGroupWs((size_t)B, n).total;
            least += one;
            total += all < kSweepGroupBytes ? all : one > kSweepGroupBytes ? one : kSweepGroupBytes;
        }
    }
};

void pdl_config(cudaLaunchConfig_t& cfg, cudaLaunchAttribute* attr, dim3 grid, dim3 block, size_t smem,
                cudaStream_t stream, bool pdl) {
    cfg = {};
    cfg.gridDim = grid;
    cfg.blockDim = block;
    cfg.dynamicSmemBytes = smem;
    cfg.stream = stream;
    attr[0].id = cudaLaunchAttributeProgrammaticStreamSerialization;
    attr[0].val.programmaticStreamSerializationAllowed = 1;
    cfg.attrs = attr;
    cfg.numAttrs = pdl_allowed(pdl) ? 1 : 0;
}

}  // namespace

size_t filter_workspace_bytes(int B, int n, int D) {
    (void)D;
    return FilterWs(B, n).total;
}
size_t filter_workspace_least_bytes(int B, int n) { return FilterWs(B, n).least; }
size_t similarity_workspace_bytes(int B, int n, int D) {
    (void)D;
    return kStatusBytes + 2 * align_up((size_t)B * n * 4, 256);
}

int launch_filter(const void* feat, const float* pos, int B, int n, int D, const vitcop_filter_params& p,
                  int n_centers, int32_t* label, int32_t* n_clusters, float* rho_user, float* delta2_user,
                  int32_t* parent_user, void* workspace, size_t workspace_bytes, cudaStream_t stream, const KnormJob* knorm) {
    const FilterWs l(B, n);
    if (workspace_bytes < l.least) return VITCOP_ERR_WORKSPACE;
    char* ws = static_cast<char*>(workspace);
    float* w = reinterpret_cast<float*>(ws + l.off_w);
    float* a = reinterpret_cast<float*>(ws + l.off_a);
    float* rho = reinterpret_cast<float*>(ws + l.off_rho);
    unsigned long long* best = reinterpret_cast<unsigned long long*>(ws + l.off_best);
    float* part = reinterpret_cast<float*>(ws + l.off_part);

    GramArgs g = {};
    g.B = B; g.n = n; g.D = D; g.row0 = 0; g.row_end = n; g.metric = p.metric;
    g.c2 = -1.4426950408889634f / (p.d_c * p.d_c);
    g.tau2 = (p.tau >= 0.f && pos) ? p.tau * p.tau : -1.f;
    g.w = w; g.a = a; g.rho = rho; g.pos = pos; g.part = part; g.best = best;
    g.w_out = w; g.a_out = a;
    g.sim_out = nullptr; g.status = reinterpret_cast<int*>(ws);

    // Everything queued before the call (the producers of features and keys included) has completed before a kernel of the call
    // other than the first can start: the diagonal is launched without programmatic overlap, and clear_kernel waits
    // before it releases the one-kernel sweep.
    int rc;
    int knorm_in_sweep = 0;                                // leading samples whose K-norm the Gram sweep computes
    if (l.resident) {
        g.rho_out = rho;
        g.rho_user = rho_user;
        g.grid_sync = reinterpret_cast<unsigned int*>(ws) + 2;
        g.ready = reinterpret_cast<uint32_t*>(ws + l.off_ready);
        if (knorm && gram_resident_takes_knorm(knorm->H, knorm->d)) {
            // The sweep's side warps take the K-norm of the first samples; the others follow beside vic_finalize_kernel.
            knorm_in_sweep = gram_resident_knorm_samples(B, n, knorm->H, knorm->d, knorm->Nv);
            if (knorm_in_sweep > 0) {
                g.kn_K = knorm->K; g.kn_score = knorm->score; g.kn_B = knorm_in_sweep;
                g.kn_H = knorm->H; g.kn_N = knorm->N; g.kn_d = knorm->d; g.kn_vis_start = knorm->vis_start; g.kn_Nv = knorm->Nv;
            }
        }
        {
            cudaLaunchConfig_t cfg;
            cudaLaunchAttribute attr[1];
            const unsigned pieces = (unsigned)(l.off_w / sizeof(uint4));
            pdl_config(cfg, attr, dim3((pieces + kClearThreads - 1) / kClearThreads), dim3(kClearThreads), 0, stream, true);
            KernelTimeScope timed("clear_kernel", stream);
            rc = record_cuda(cudaLaunchKernelEx(&cfg, clear_kernel, static_cast<uint4*>(workspace), pieces));
            if (rc != VITCOP_OK) return rc;
        }
        rc = launch_gram_resident(feat, g, make_gram_tiling(n), stream);
        if (rc != VITCOP_OK) return rc;
    } else {
        // with a spatial radius, blocks beyond it are neither kept nor looked into (density.cuh: blocks_outside_radius)
        g.bbox = g.tau2 >= 0.f ? reinterpret_cast<float4*>(ws + l.off_bbox) : nullptr;
        g.best = nullptr;                                  // (the search writes every token's entry)
        const SweepTiling tiling = make_sweep_tiling(n);
        const int diag_ctas = (long long)B * tiling.TI < gram_num_sms() ? B * tiling.TI : gram_num_sms();
        g.reports = diag_ctas <= kMaxReports;
        if (!g.reports) {
            rc = record_cuda(cudaMemsetAsync(workspace, 0, kStatusBytes, stream));
            if (rc != VITCOP_OK) return rc;
        }
        rc = launch_gram_sweep(GRAM_DIAG, feat, g, stream, false);
        if (rc != VITCOP_OK) return rc;
        const int group = sweep_group_samples(B, n, (workspace_bytes < l.total ? workspace_bytes : l.total) - l.off_group);
        const SweepGroupWs kept((size_t)group, n);
        char* const gws = ws + l.off_group;
        for (int b0 = 0; b0 < B; b0 += group) {
            const size_t at = (size_t)b0 * n;
            SweepArgs s = {};
            s.B = B - b0 < group ? B - b0 : group;
            s.n = n; s.D = D; s.c2 = g.c2; s.tau2 = g.tau2;
            s.w = w + at; s.a = a + at; s.rho = rho + at; s.best = best + at;
            s.pos = pos ? pos + 2 * at : nullptr;
            s.bbox = g.bbox ? g.bbox + (size_t)b0 * tiling.TI : nullptr;
            s.part = part + (size_t)b0 * tiling.slots() * tiling.n_pad;
            s.n_left = reinterpret_cast<int32_t*>(gws + kept.off_left);
            s.left = s.n_left + 1;
            s.tok = reinterpret_cast<float4*>(gws + kept.off_tok);
            s.blk_rho = reinterpret_cast<uint32_t*>(gws + kept.off_blk_rho);
            s.blk_min = reinterpret_cast<float*>(gws + kept.off_blk_min);
            s.gram = reinterpret_cast<float*>(gws + kept.off_gram);
            s.status = g.status;
            s.diag_reports = g.reports ? diag_ctas : 0;
            s.t = tiling;
            if (knorm && b0 == 0 && (knorm_in_sweep = sweep_knorm_samples(*knorm, s.B, n, D)) > 0) {
                s.kn = *knorm;
                s.kn.B = knorm_in_sweep;
            }
            rc = launch_density_sweep(static_cast<const uint16_t*>(feat) + at * D, s, p.metric, stream, true);
            if (rc != VITCOP_OK) return rc;
            {
                cudaLaunchConfig_t cfg;
                cudaLaunchAttribute attr[1];
                pdl_config(cfg, attr, dim3((n + kBlk - 1) / kBlk, s.B), dim3(kRhoThreads), 0, stream, true);
                KernelTimeScope timed("rho_reduce_kernel", stream);
                rc = record_cuda(cudaLaunchKernelEx(&cfg, rho_reduce_kernel, s, (int)p.metric, rho_user ? rho_user + at : nullptr));
                if (rc != VITCOP_OK) return rc;
            }
            rc = launch_nearest_denser(s, p.metric, stream, true);
            if (rc != VITCOP_OK) return rc;
        }
    }

    const int nc = n_centers < n ? n_centers : n;
    const size_t smem = finalize_smem(n, nc);
    const int v = n <= kFinThreads ? 0 : n <= 4 * kFinThreads ? 1 : n <= 8 * kFinThreads ? 2 : 3;
    auto fin = v == 0 ? vic_finalize_kernel<1> : v == 1 ? vic_finalize_kernel<4> : v == 2 ? vic_finalize_kernel<8> : vic_finalize_kernel<16>;
    static_assert(VITCOP_MAX_VISUAL_TOKENS <= 16 * kFinThreads, "tokens of the longest sample");
    if (v > 0) {                                           // (up to 1024 tokens 5 KB)
        static DoneOnDevice attr_done[4];
        const int most = (v == 1 ? 4 : v == 2 ? 8 : 16) * kFinThreads;
        rc = allow_dynamic_smem(fin, finalize_smem(most, most), attr_done[v]);
        if (rc != VITCOP_OK) return rc;
    }
    cudaLaunchConfig_t cfg;
    cudaLaunchAttribute attr[1];
    pdl_config(cfg, attr, dim3(B), dim3(kFinThreads), smem, stream, true);
    {
        KernelTimeScope timed("vic_finalize_kernel", stream);
        rc = record_cuda(cudaLaunchKernelEx(&cfg, fin, static_cast<const uint16_t*>(feat), n, D, nc,
                                            (const float*)rho, (const unsigned long long*)best, (const float*)w,
                                            (const float*)a, label, n_clusters, delta2_user, parent_user));
        if (rc != VITCOP_OK) return rc;
    }
    if (knorm && knorm_in_sweep < knorm->B) {
        // vic_finalize_kernel runs one CTA per sample and releases its dependents when it starts: the K-norm, which
        // does not depend on the clustering, streams K from HBM on the other SMs meanwhile and waits for the
        // finalize kernel before it ends.  (Beside a Gram sweep it would not fit: those kernels' CTAs hold most of each SM's
        // registers.)
        const int64_t stride_b = (int64_t)knorm->H * knorm->N * knorm->d;
        rc = launch_knorm(static_cast<const uint16_t*>(knorm->K) + (size_t)knorm_in_sweep * stride_b,
                          knorm->B - knorm_in_sweep, knorm->H, knorm->d, stride_b, (int64_t)knorm->N * knorm->d, knorm->d,
                          knorm->vis_start, nullptr, knorm->Nv, knorm->score + (size_t)knorm_in_sweep * knorm->Nv,
                          knorm->Nv, stream, true);
    }
    return rc;
}

int launch_similarity_rows(const void* feat, int B, int n, int D, int metric, int row_begin, int row_end, float* out,
                           void* workspace, cudaStream_t stream) {
    char* ws = static_cast<char*>(workspace);
    float* w = reinterpret_cast<float*>(ws + kStatusBytes);
    float* a = reinterpret_cast<float*>(ws + kStatusBytes + align_up((size_t)B * n * 4, 256));
    GramArgs g = {};
    g.B = B; g.n = n; g.D = D; g.row0 = row_begin; g.row_end = row_end; g.metric = metric;
    g.c2 = 0.f; g.tau2 = -1.f;
    g.w = w; g.a = a; g.w_out = w; g.a_out = a; g.sim_out = out; g.status = reinterpret_cast<int*>(ws);
    int rc = launch_gram_sweep(GRAM_DIAG, feat, g, stream, false);
    if (rc != VITCOP_OK) return rc;
    return launch_gram_sweep(GRAM_SIM, feat, g, stream, true);
}

}  // namespace vitcop
