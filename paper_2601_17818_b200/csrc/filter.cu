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
// the end of the token's tile (blocks that hold none of them count as zero).  Up to 64 entries are added one by one; longer
// lists (up to 192 on the longest samples) in four equal parts, whose sums are then added.  One CTA per 32 tokens: its warps
// fetch the entries, all of them in one trip to memory, and the sums are taken from shared memory.  (One thread per token
// walking its list paid a trip for every sixteen entries.)
// blk_rho[b,k]: bits of the largest density among the tokens of block k (densities are not negative, their bit patterns order
// like the values).
constexpr int kRhoThreads = 256;
constexpr int kRhoOneByOne = 64;
constexpr int kRhoEntries = 3 * VITCOP_MAX_VISUAL_TOKENS / kSweepTile;       // longest list
__global__ void __launch_bounds__(kRhoThreads)
rho_reduce_kernel(const float* __restrict__ part, int n, SweepTiling t, float* __restrict__ rho,
                  float* __restrict__ rho_user, uint32_t* __restrict__ blk_rho, int32_t* __restrict__ n_left) {
    constexpr int kWarps = kRhoThreads / 32;
    __shared__ float entry[kRhoEntries][kBlk];
    __shared__ float parts[4][kBlk];
    grid_dependency_launch_dependents();
    grid_dependency_wait();
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    const int blk = blockIdx.x, b = blockIdx.y, i = blk * kBlk + lane;
    if (blk == 0 && b == 0 && threadIdx.x == 0) *n_left = 0;         // for the search behind this kernel
    const int own = blk * kBlk / kGramBM, tile = own / 2;
    const int rows = t.T - tile;                           // entries on the row side, then min(TI, 2 (tile + 1)) more
    const int entries = rows + min(t.TI, 2 * (tile + 1));
    if (i < n) {
        const float* p = part + (size_t)b * t.slots() * t.n_pad + i;
        auto slot = [&](int k) { return p[(size_t)k * t.n_pad]; };
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
        rho[(size_t)b * n + i] = s;
        if (rho_user) rho_user[(size_t)b * n + i] = s;
    }
    const uint32_t m = __reduce_max_sync(0xffffffffu, i < n ? __float_as_uint(s) : 0u);
    if (lane == 0) blk_rho[(size_t)b * t.n_blk() + blk] = m;
}

// ------------------------------------------------------------------------------------------------
// Centres, forest roots and labels: one CTA per sample.
// ------------------------------------------------------------------------------------------------
constexpr int kFinThreads = 1024;
constexpr int kFinIters = VITCOP_MAX_VISUAL_TOKENS / kFinThreads;      // tokens per thread at the largest sample

// Shared memory: keys[n] (uint64; later reused as next[n] int32), isc[n] (uint8), centres[nc] (int32).
__global__ void __launch_bounds__(kFinThreads)
vic_finalize_kernel(const uint16_t* __restrict__ feat, int n, int D, int n_centers, const float* __restrict__ rho,
                    const unsigned long long* __restrict__ best, const float* __restrict__ w,
                    const float* __restrict__ a, int32_t* __restrict__ label, int32_t* __restrict__ n_clusters,
                    float* __restrict__ delta2_user, int32_t* __restrict__ parent_user) {
    extern __shared__ __align__(16) uint8_t fin_smem[];
    unsigned long long* keys = reinterpret_cast<unsigned long long*>(fin_smem);
    int32_t* nxt = reinterpret_cast<int32_t*>(fin_smem);              // aliases keys after the selection
    uint8_t* isc = fin_smem + (size_t)n * 8;
    int32_t* centres = reinterpret_cast<int32_t*>(fin_smem + (size_t)n * 8 + (((size_t)n + 15) & ~(size_t)15));
    __shared__ uint32_t hist[256];
    __shared__ uint32_t warp_sums[32];
    __shared__ uint32_t cnt[kFinIters * 32];               // one count per (iteration, warp)
    __shared__ uint32_t s_digit, s_krem, s_whole;
    __shared__ unsigned long long orph_best[kFinThreads];
    __shared__ int orph_list[kFinThreads];
    __shared__ int orph_cnt;

    grid_dependency_launch_dependents();
    grid_dependency_wait();
    const int b = blockIdx.x;
    const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
    rho += (size_t)b * n;
    best += (size_t)b * n;
    w += (size_t)b * n;
    a += (size_t)b * n;
    label += (size_t)b * n;
    feat += (size_t)b * n * D;
    if (delta2_user) delta2_user += (size_t)b * n;
    if (parent_user) parent_user += (size_t)b * n;
    const int nc = min(n_centers, n);

    // rank key, ascending = better centre candidate: ~( orphan ? (0xFFFFFFFF, rho) : (gamma, rho) )
    for (int i = tid; i < n; i += kFinThreads) {
        const unsigned long long p = best[i];
        const bool orphan = p == ~0ull;
        const float d2 = orphan ? __int_as_float(0x7f800000) : __uint_as_float((uint32_t)(p >> 32));
        const int par = orphan ? -1 : (int)(uint32_t)(p & 0xFFFFFFFFull);
        if (delta2_user) delta2_user[i] = d2;
        if (parent_user) parent_user[i] = par;
        const float r = rho[i];
        const uint32_t hi = orphan ? 0xFFFFFFFFu : __float_as_uint(r * sqrtf(d2));
        keys[i] = ~(((unsigned long long)hi << 32) | (unsigned long long)__float_as_uint(r));
    }
    __syncthreads();

    // ---- radix select of the nc smallest keys (8 passes of 8 bits), ties -> lower index
    unsigned long long T = ~0ull;
    uint32_t krem = 0;
    if (nc > 0 && nc < n) {
        unsigned long long prefix = 0;
        krem = (uint32_t)nc;
        for (int pass = 0; pass < 8; ++pass) {
            const int shift = 56 - 8 * pass;
            const unsigned long long hi_mask = pass == 0 ? 0ull : (~0ull << (shift + 8));
            if (tid < 256) hist[tid] = 0;
            __syncthreads();
            for (int base = 0; base < n; base += kFinThreads) {
                const int i = base + tid;
                int dig = -1;
                if (i < n) {
                    const unsigned long long key = keys[i];
                    if ((key & hi_mask) == prefix) dig = (int)((key >> shift) & 255ull);
                }
                const uint32_t peers = __match_any_sync(0xffffffffu, dig);
                if (dig >= 0 && lane == __ffs(peers) - 1) atomicAdd(&hist[dig], (uint32_t)__popc(peers));
            }
            __syncthreads();
            const uint32_t c = tid < 256 ? hist[tid] : 0u;
            uint32_t v = c;
#pragma unroll
            for (int off = 1; off < 32; off <<= 1) {
                const uint32_t t = __shfl_up_sync(0xffffffffu, v, off);
                if (lane >= off) v += t;
            }
            if (lane == 31) warp_sums[warp] = v;
            __syncthreads();
            if (tid < 256) {
                uint32_t basew = 0;
                for (int q = 0; q < warp; ++q) basew += warp_sums[q];
                const uint32_t incl = basew + v, excl = incl - c;
                if (excl < krem && krem <= incl) {
                    s_digit = (uint32_t)tid;
                    s_krem = krem - excl;
                    s_whole = (c == krem - excl) ? 1u : 0u;         // the whole bin is wanted
                }
            }
            __syncthreads();
            prefix |= (unsigned long long)s_digit << shift;
            krem = s_krem;
            const bool whole = s_whole != 0;
            __syncthreads();
            if (whole) {
                // every key that shares the prefix found so far is selected: no need to resolve lower digits
                prefix |= (1ull << shift) - 1ull;
                krem = 0xFFFFFFFFu;
                break;
            }
        }
        T = prefix;
    }
    // ---- centre flags + ascending centre list.  Token i = it * 1024 + tid; ranks in index order come from one count
    //      per (iteration, warp), scanned once for the whole sample, plus the lane's position in its warp's ballot:
    //      first among the keys equal to the cut (ties -> lower index), then among the centres.
    {
        uint32_t eq_mask = 0, f_mask = 0;                  // bit it: this thread's token of iteration it is ... / is a centre
        const int iters = (n + kFinThreads - 1) / kFinThreads;          // <= kFinIters
        const uint32_t lane_below = (1u << lane) - 1u;
        const bool cut = nc > 0 && nc < n;
        if (cut) {
            for (int it = 0; it < iters; ++it) {
                const int i = it * kFinThreads + tid;
                const bool eq = i < n && keys[i] == T;
                const uint32_t bal = __ballot_sync(0xffffffffu, eq);
                if (eq) eq_mask |= 1u << it;
                if (lane == 0) cnt[it * 32 + warp] = __popc(bal);
            }
            __syncthreads();
            uint32_t total;
            const uint32_t excl = block_exclusive_sum(tid < iters * 32 ? cnt[tid] : 0u, warp_sums, total);
            if (tid < iters * 32) cnt[tid] = excl;
            __syncthreads();
        }
        for (int it = 0; it < iters; ++it) {
            const int i = it * kFinThreads + tid;
            bool f;
            if (nc <= 0) f = false;
            else if (nc >= n) f = i < n;
            else {
                const bool eq = (eq_mask >> it & 1u) != 0;
                const uint32_t bal = __ballot_sync(0xffffffffu, eq);
                const uint32_t eq_rank = cnt[it * 32 + warp] + __popc(bal & lane_below);
                f = i < n && (keys[i] < T || (eq && eq_rank < krem));
            }
            if (f) f_mask |= 1u << it;
            if (i < n) isc[i] = f ? 1 : 0;
        }
        __syncthreads();                                   // cnt is reused
        for (int it = 0; it < iters; ++it) {
            const uint32_t bal = __ballot_sync(0xffffffffu, (f_mask >> it & 1u) != 0);
            if (lane == 0) cnt[it * 32 + warp] = __popc(bal);
        }
        __syncthreads();
        uint32_t total;
        const uint32_t excl = block_exclusive_sum(tid < iters * 32 ? cnt[tid] : 0u, warp_sums, total);
        if (tid < iters * 32) cnt[tid] = excl;
        __syncthreads();
        for (int it = 0; it < iters; ++it) {
            const bool f = (f_mask >> it & 1u) != 0;
            const uint32_t bal = __ballot_sync(0xffffffffu, f);
            const uint32_t r = cnt[it * 32 + warp] + __popc(bal & lane_below);
            if (f && r < (uint32_t)nc) centres[r] = it * kFinThreads + tid;
        }
    }
    __syncthreads();   // keys are dead from here on; nxt aliases them

    // ---- forest roots by pointer jumping: a centre or an orphan is its own root
    for (int i = tid; i < n; i += kFinThreads) {
        const unsigned long long p = best[i];
        const int par = (p == ~0ull) ? -1 : (int)(uint32_t)(p & 0xFFFFFFFFull);
        nxt[i] = (isc[i] || par < 0 || par >= n) ? i : par;
    }
    __syncthreads();
    for (int round = 0; round < 16; ++round) {
        int changed = 0;
        for (int i = tid; i < n; i += kFinThreads) {
            const int p = nxt[i];
            const int q = nxt[p];
            if (q != p) {
                nxt[i] = q;       // any value read here is an ancestor of i, roots are fixed points
                changed = 1;
            }
        }
        if (!__syncthreads_or(changed)) break;
    }

    // ---- labels; a root that is an orphan but not a centre joins the nearest centre (feature distance)
    for (int i = tid; i < n; i += kFinThreads) {
        const int root = nxt[i];
        label[i] = isc[root] ? root : -1 - root;
    }
    __syncthreads();
    int any_surplus = 0;                                   // a root that is neither a centre nor below one
    for (int i = tid; i < n; i += kFinThreads) any_surplus |= (!isc[i] && nxt[i] == i) ? 1 : 0;
    any_surplus = __syncthreads_or(any_surplus);
    if (nc > 0 && any_surplus) {
        // Surplus orphans (roots that are not centres) are rare but each needs its distance to every centre: they
        // are listed, kFinThreads tokens at a time, and the (orphan, centre) pairs are spread over all warps; the
        // nearest centre wins through a packed minimum (distance bits, then the lower centre rank).
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
            for (int pr = warp; pr < pairs; pr += kFinThreads / 32) {
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
                    atomicMin(&orph_best[e], ((unsigned long long)__float_as_uint(d2) << 32) | (unsigned long long)q);
            }
            __syncthreads();
            if (tid < orph_cnt)                                     // remember the adopted centre at the root
                nxt[orph_list[tid]] = -1 - centres[(int)(orph_best[tid] & 0xFFFFFFFFull)];
        }
    }
    __syncthreads();
    for (int i = tid; i < n; i += kFinThreads) {
        const int l = label[i];
        if (l < 0) {
            const int root = -1 - l;
            const int adopted = nxt[root];
            label[i] = adopted < 0 ? -1 - adopted : root;
        }
    }
    if (tid == 0) n_clusters[b] = nc;
}

// ------------------------------------------------------------------------------------------------
// host side
// ------------------------------------------------------------------------------------------------
// Workspace of the filter: status block | row-block flags [B, ceil(n / 128)] | w | a | rho | best |
// rho partials [B, slots, n_pad] (sized for either sweep) | bounding boxes of the row blocks' positions | and, for
// problems too large for the one-kernel sweep, of one group of samples: count and list of the search's leftovers, block densities, block minima, Gram values of
// the density sweep (4 bytes per pair of the symmetric half, tile padding included).  The status block and the
// flags are zeroed at the start of every call.  Words of the status block: 0 status, 2 grid barrier.
struct FilterWs {
    size_t off_flags, off_w, off_a, off_rho, off_best, off_part, off_bbox, off_left, off_blk_rho, off_blk_min, off_gram, total;
    FilterWs(int B, int n) {
        size_t o = kStatusBytes;
        const size_t bn = (size_t)B * n;
        off_flags = o; o += align_up((size_t)B * ((n + kGramBM - 1) / kGramBM) * 4, 256);
        off_w = o;    o += align_up(bn * 4, 256);
        off_a = o;    o += align_up(bn * 4, 256);
        off_rho = o;  o += align_up(bn * 4, 256);
        off_best = o; o += align_up(bn * 8, 256);
        const GramTiling t = make_gram_tiling(n, 128);           // (two slots per block: never fewer than the density sweep's)
        off_part = o; o += align_up((size_t)B * t.slots() * t.n_pad * 4, 256);
        off_bbox = o;   o += align_up((size_t)B * t.TI * sizeof(float4), 256);
        off_left = off_blk_rho = off_blk_min = off_gram = o;
        if (B > 0 && n > 0 && !gram_fits_resident(B, n)) {
            const SweepTiling s = make_sweep_tiling(n);
            const size_t group = (size_t)sweep_group_samples(B, n);
            o += align_up((group * n + 1) * 4, 256);
            off_blk_rho = o; o += align_up(group * s.n_blk() * 4, 256);
            off_blk_min = o; o += align_up(group * s.n_blk() * s.n_pad * 4, 256);
            off_gram = o;    o += align_up(group * s.tiles_per_b * kSweepTileFloats * 4, 256);
        }
        total = o;
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

size_t filter_zeroed_bytes(int B, int n) { return FilterWs(B, n).off_w; }

size_t filter_workspace_bytes(int B, int n, int D) {
    (void)D;
    return FilterWs(B, n).total;
}
size_t similarity_workspace_bytes(int B, int n, int D) {
    (void)D;
    return kStatusBytes + 2 * align_up((size_t)B * n * 4, 256);
}

int launch_filter(const void* feat, const float* pos, int B, int n, int D, const vitcop_filter_params& p,
                  int n_centers, int32_t* label, int32_t* n_clusters, float* rho_user, float* delta2_user,
                  int32_t* parent_user, void* workspace, cudaStream_t stream, const KnormJob* knorm) {
    FilterWs l(B, n);
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

    // The first kernel of the call is launched without programmatic overlap, so everything queued before the call
    // (the producer of the features included) has completed when it starts.
    int rc;
    int knorm_in_sweep = 0;                                // leading samples whose K-norm the Gram sweep computes
    const bool resident = gram_fits_resident(B, n);
    if (resident) {
        g.rho_out = rho;
        g.rho_user = rho_user;
        g.grid_sync = reinterpret_cast<unsigned int*>(ws) + 2;       // zeroed with the status word at the start of the call
        g.diag_ready = reinterpret_cast<unsigned int*>(ws + l.off_flags);
        if (knorm && gram_resident_takes_knorm(knorm->H, knorm->d)) {
            // The sweep's two idle warps take the K-norm of the first samples, about as many as they finish while
            // the epilogue warps work on the accumulators; the other samples follow beside vic_finalize_kernel.
            knorm_in_sweep = (5 * knorm->B + 8) / 16;
            if (knorm_in_sweep > 0) {
                g.kn_K = knorm->K; g.kn_score = knorm->score; g.kn_B = knorm_in_sweep;
                g.kn_H = knorm->H; g.kn_N = knorm->N; g.kn_d = knorm->d; g.kn_vis_start = knorm->vis_start; g.kn_Nv = knorm->Nv;
            }
        }
        rc = launch_gram_resident(feat, g, make_gram_tiling(n, 128), stream);
        if (rc != VITCOP_OK) return rc;
    } else {
        // with a spatial radius, blocks beyond it are neither kept nor looked into (density.cuh: blocks_outside_radius)
        g.bbox = g.tau2 >= 0.f ? reinterpret_cast<float4*>(ws + l.off_bbox) : nullptr;
        g.best = nullptr;                                  // (the search writes every token's entry)
        rc = launch_gram_sweep(GRAM_DIAG, feat, g, stream, false);
        if (rc != VITCOP_OK) return rc;
        const SweepTiling tiling = make_sweep_tiling(n);
        const int group = sweep_group_samples(B, n);
        for (int b0 = 0; b0 < B; b0 += group) {
            const size_t at = (size_t)b0 * n;
            SweepArgs s = {};
            s.B = B - b0 < group ? B - b0 : group;
            s.n = n; s.D = D; s.c2 = g.c2; s.tau2 = g.tau2;
            s.w = w + at; s.a = a + at; s.rho = rho + at; s.best = best + at;
            s.pos = pos ? pos + 2 * at : nullptr;
            s.bbox = g.bbox ? g.bbox + (size_t)b0 * tiling.TI : nullptr;
            s.part = part + (size_t)b0 * tiling.slots() * tiling.n_pad;
            s.n_left = reinterpret_cast<int32_t*>(ws + l.off_left);
            s.left = s.n_left + 1;
            s.blk_rho = reinterpret_cast<uint32_t*>(ws + l.off_blk_rho);
            s.blk_min = reinterpret_cast<float*>(ws + l.off_blk_min);
            s.gram = reinterpret_cast<float*>(ws + l.off_gram);
            s.status = g.status;
            s.t = tiling;
            rc = launch_density_sweep(static_cast<const uint16_t*>(feat) + at * D, s, p.metric, stream, true);
            if (rc != VITCOP_OK) return rc;
            {
                cudaLaunchConfig_t cfg;
                cudaLaunchAttribute attr[1];
                pdl_config(cfg, attr, dim3((n + kBlk - 1) / kBlk, s.B), dim3(kRhoThreads), 0, stream, true);
                KernelTimeScope timed("rho_reduce_kernel", stream);
                rc = record_cuda(cudaLaunchKernelEx(&cfg, rho_reduce_kernel, (const float*)s.part, n, tiling, rho + at,
                                                    rho_user ? rho_user + at : nullptr, s.blk_rho, s.n_left));
                if (rc != VITCOP_OK) return rc;
            }
            rc = launch_nearest_denser(s, p.metric, stream, true);
            if (rc != VITCOP_OK) return rc;
        }
    }

    const int nc = n_centers < n ? n_centers : n;
    const size_t smem = (size_t)n * 8 + (((size_t)n + 15) & ~(size_t)15) + (size_t)(nc > 0 ? nc : 1) * 4 + 16;
    if (smem > 32 * 1024) {                                // (the kernel's static arrays take part of the default 48 KB)
        cudaError_t e = cudaFuncSetAttribute(vic_finalize_kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem);
        if (e != cudaSuccess) return record_cuda(e);
    }
    cudaLaunchConfig_t cfg;
    cudaLaunchAttribute attr[1];
    pdl_config(cfg, attr, dim3(B), dim3(kFinThreads), smem, stream, true);
    {
        KernelTimeScope timed("vic_finalize_kernel", stream);
        rc = record_cuda(cudaLaunchKernelEx(&cfg, vic_finalize_kernel, static_cast<const uint16_t*>(feat), n, D, nc,
                                            (const float*)rho, (const unsigned long long*)best, (const float*)w,
                                            (const float*)a, label, n_clusters, delta2_user, parent_user));
        if (rc != VITCOP_OK) return rc;
    }
    if (knorm && knorm_in_sweep < knorm->B) {
        // vic_finalize_kernel runs one CTA per sample and releases its dependents when it starts: the K-norm, which
        // does not depend on the clustering, streams K from HBM on the other SMs meanwhile and waits for the
        // finalize kernel before it ends.  (Beside the Gram sweep it would not fit: that kernel's CTAs hold most
        // of each SM's registers.)
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
