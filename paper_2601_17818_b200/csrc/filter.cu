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
#include "select_rank.cuh"
#include "vic_labels.cuh"

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
// Centres, forest roots and labels (vic_labels.cuh): R CTAs per sample, E tokens per thread.  SELECT: right behind them the
// cluster-quota selection of a pruning step (select_rank.cuh) whose scores are there by then: the labels stay in registers, and a launch and a
// trip to memory go (1 x 576 tokens, whole call, 31.5 -> 29.0 us).
// ------------------------------------------------------------------------------------------------
struct QuotaArgs {
    QuotaJob job;
    int P_cap;
    int* status;
};
// (One CTA an SM, said aloud: left to itself ptxas went for two of the form up to 1024 tokens, 32 registers a thread and spills, and the
// filter of 8 x 203 tokens took 21.5 us with the caches flushed; 19.5 so.)
template <int R, int E, bool SELECT>
__global__ void __launch_bounds__(kGroupThreads, 1)
vic_finalize_kernel(const __grid_constant__ VicArgs v, const __grid_constant__ QuotaArgs q) {
    extern __shared__ __align__(16) uint8_t fin_dyn[];
    __shared__ VicShared<R> sh;
    grid_dependency_launch_dependents();
    sh.init();
    grid_dependency_wait();
    const int b = blockIdx.x / R;
    int lab[E];
    if constexpr (SELECT) {
        static_assert(R == 1 && kGroupThreads == kSelThreads, "one CTA, its tokens spread as the selection has them");
        const int n = v.n;
        const float* const score = q.job.score + (size_t)b * n;
        uint32_t key[E];
#pragma unroll
        for (int e = 0; e < E; ++e) {                      // (on their way while the labels are worked out)
            const int i = e * kSelThreads + threadIdx.x;
            key[e] = i < n ? __float_as_uint(__ldcg(score + i)) : 0u;
        }
        vic_labels<R, E>(v, b, sh, fin_dyn, lab);
#pragma unroll
        for (int e = 0; e < E; ++e) key[e] = order_key(__uint_as_float(key[e]), 0);
        __shared__ RankShared rs;
        int32_t *const keep = q.job.keep + (size_t)b * n, *const n_keep = q.job.n_keep + b;
        __syncthreads();                                   // (the table is no longer needed, and all labels are written)
        if (!select_by_rank<E>(lab, key, n, q.job.budget, rs, fin_dyn, keep, n, n_keep, nullptr, q.status))
            select_by_sort(score, v.label + (size_t)b * n, n, n, q.P_cap, q.job.budget, keep, n, n_keep, nullptr, q.status, fin_dyn, rs.warp_sums);
    } else {
        vic_labels<R, E>(v, b, sh, fin_dyn, lab);
    }
}

typedef void (*FinalizeKernel)(VicArgs, QuotaArgs);
FinalizeKernel finalize_kernel(int R, int E, bool select) {
    return select   ? (E == 1 ? vic_finalize_kernel<1, 1, true> : vic_finalize_kernel<1, 2, true>)
           : R == 8 ? vic_finalize_kernel<8, 2, false>
           : E == 1 ? vic_finalize_kernel<1, 1, false>
           : E == 2 ? vic_finalize_kernel<1, 2, false>
           : E == 4 ? vic_finalize_kernel<1, 4, false>
           : E == 8 ? vic_finalize_kernel<1, 8, false> : vic_finalize_kernel<1, 16, false>;
}
size_t finalize_smem(int R, int n, int nc, bool select, int* P_cap) {
    const size_t labels = R == 1 ? vic_smem<1>(n, nc) : vic_smem<8>(n, nc), quota = select ? rank_or_sort_smem(n, P_cap) : 0;
    return labels > quota ? labels : quota;
}
size_t finalize_most_smem(int R, int E, bool select) {
    int p = 0;
    return finalize_smem(R, R * E * kGroupThreads, R * E * kGroupThreads, select, &p);
}
int finalize_allow_smem(int R, int E, bool select) {
    static DoneOnDevice attr_done[2][9][17];
    return allow_dynamic_smem(finalize_kernel(R, E, select), finalize_most_smem(R, E, select), attr_done[select][R][E]);
}
int finalize_clusters_at_once() {
    static KnownOnDevice known;
    return clusters_at_once(finalize_kernel(8, 2, false), 8, kGroupThreads, finalize_most_smem(8, 2, false),
                            [] { return finalize_allow_smem(8, 2, false); }, known);
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
                  int32_t* parent_user, void* workspace, size_t workspace_bytes, cudaStream_t stream, const KnormJob* knorm,
                  QuotaJob* quota) {
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
            if (knorm && b0 == 0 && (knorm_in_sweep = sweep_knorm_samples(*knorm, s.B, n, D, p.metric)) > 0) {
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
    // CTAs per sample: one up to 8192 tokens, eight beyond where the batch is on the chip at once (2 x 16384 tokens 28 us on one, 15
    // on eight; 4 x 4608 9 on one, 12 on eight, which meet a dozen times).
    const int R = n > 8 * kGroupThreads && B <= finalize_clusters_at_once() ? 8 : 1;
    int E = 1;
    while (R * E * kGroupThreads < n) E *= 2;
    static_assert(VITCOP_MAX_VISUAL_TOKENS <= 16 * kGroupThreads, "tokens of the longest sample");
    // With all scores there by then the selection of up to 2048 tokens follows in the same kernel.
    const bool select = quota && n <= kRankTokens && knorm && knorm_in_sweep == knorm->B;
    if (quota) quota->taken = select;
    {
        const VicArgs v = {static_cast<const uint16_t*>(feat), n, D, nc, rho, best, w, a, label, n_clusters, delta2_user, parent_user};
        QuotaArgs q = {};
        if (select) q.job = *quota;
        q.status = g.status;
        const size_t smem = finalize_smem(R, n, nc, select, &q.P_cap);
        rc = finalize_allow_smem(R, E, select);
        if (rc != VITCOP_OK) return rc;
        cudaLaunchConfig_t cfg;
        cudaLaunchAttribute attr[2];
        pdl_config(cfg, attr, dim3((unsigned)B * (unsigned)R), dim3(kGroupThreads), smem, stream, true);
        if (R > 1) {
            attr[cfg.numAttrs].id = cudaLaunchAttributeClusterDimension;
            attr[cfg.numAttrs].val.clusterDim.x = (unsigned)R;
            attr[cfg.numAttrs].val.clusterDim.y = attr[cfg.numAttrs].val.clusterDim.z = 1;
            ++cfg.numAttrs;
        }
        KernelTimeScope timed("vic_finalize_kernel", stream);
        rc = record_cuda(cudaLaunchKernelEx(&cfg, finalize_kernel(R, E, select), v, q));
        if (rc != VITCOP_OK) return rc;
    }
    if (knorm && knorm_in_sweep < knorm->B) {
        // vic_finalize_kernel runs one CTA per sample, eight of a long one, and releases its dependents when it starts: the
        // K-norm, which does not depend on the clustering, streams K from HBM on the other SMs meanwhile and waits for the
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
