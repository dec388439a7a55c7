// Eq. 3 (Algorithm 2, step 2): per token the nearest denser token inside the spatial radius, searched in what the
// density sweep left behind (density.cuh): every Gram value of the symmetric half, and per (token, block of 32 tokens) the
// smallest squared distance.
//
// A block can hold a token's answer only if its minimum is not above the best denser token found so far.  One warp per token:
// every lane keeps the two smallest minima among its blocks (block % 32 = lane) and the warp looks into the blocks in
// ascending order, two at a time (lane = token of the block: the Gram value, the factors, the density and the spatial test).
// For nine tokens in ten two or three rounds are enough: their nearest neighbours include a denser token (half of all tokens need one
// block).  The few tokens that are the densest of their surroundings may have to look into dozens of blocks; these are listed
// and left to a second kernel, in which several warps share out a token's blocks, passing over those without a denser
// token (largest density of the block): a warp alone would hold up everything behind it.  What is skipped could not have
// changed the minimum, and d^2 is recomputed from the stored value with the arithmetic of the sweep (and of the one-kernel
// sweep), so the result has the same bits as a full pass over the pairs.
//
// Both kernels are bound by the latency of their dependent trips to memory (minima, blocks, blocks again), hence few registers
// and as many warps as fit.
#include "density.cuh"

namespace vitcop {
namespace {

constexpr int kNdThreads = 256, kNdWarps = kNdThreads / 32;
constexpr int kNdRounds = 3;                               // rounds of two blocks that a warp does for its own token
constexpr int kNdAhead = 4;                                // blocks a warp of the second kernel looks into at a time
constexpr uint32_t kInfBits = 0x7f800000u;
// A lane orders its blocks by a key: the bits of the minimum (never negative) with the block's number in the low bits, i.e. a
// bound up to 2^-14 too low.
constexpr uint32_t kBlkMask = VITCOP_MAX_VISUAL_TOKENS / kBlk - 1;
static_assert((kBlkMask & (kBlkMask + 1)) == 0 && kBlkMask < (1u << 10), "block numbers fit the low bits of a key");

// One sample as the search sees it.
template <int METRIC, bool SPATIAL>
struct Sample {
    const float *rho, *w, *a, *gram, *minima;
    const float2* pos;
    const uint32_t* top;                                   // largest density of every block
    int n, nb, row;                                        // tokens, blocks that hold tokens, minima per token
    float tau2;
    __device__ __forceinline__ Sample(const SweepArgs& g, int b) {
        const size_t bo = (size_t)b * g.n;
        rho = g.rho + bo;
        w = g.w + bo;
        a = g.a + bo;
        pos = SPATIAL ? reinterpret_cast<const float2*>(g.pos) + bo : nullptr;
        gram = g.gram + (size_t)b * g.t.tiles_per_b * kSweepTileFloats;
        row = g.t.n_blk();
        minima = g.blk_min + (size_t)b * g.t.n_pad * row;
        top = g.blk_rho + (size_t)b * row;
        n = g.n;
        nb = (n + kBlk - 1) / kBlk;
        tau2 = g.tau2;
    }
    struct Token {
        int i;
        float rho, w, a;
        float2 pos;
    };
    __device__ __forceinline__ Token token(int i) const {
        Token t;
        t.i = i;
        t.rho = rho[i];
        t.w = w[i];
        t.a = METRIC == 1 ? a[i] : 1.f;
        t.pos = SPATIAL ? pos[i] : make_float2(0.f, 0.f);
        return t;
    }
    struct Pair {                                          // what a lane needs of the pair (i, 32 blk + lane)
        float gram, w, rho, a;
        float2 pos;
    };
    __device__ __forceinline__ Pair fetch(int i, int blk, int lane) const {
        Pair p;
        const int j = min(blk * kBlk + lane, n - 1), own = i / kBlk, ri = i % kBlk;
        // the pair's lower index is its row (inside the own block: in either order)
        const bool below = blk < own || (blk == own && lane < ri);
        const int r = below ? lane : ri, c = below ? ri : lane;
        p.gram = gram[gram_block_offset(min(blk, own), max(blk, own)) + gram_elem_offset(r, c)];
        p.w = w[j];
        p.rho = rho[j];
        p.a = METRIC == 1 ? a[j] : 1.f;
        p.pos = SPATIAL ? pos[j] : make_float2(0.f, 0.f);
        return p;
    }
    // Folds the block's nearest denser token into `best` (packed as SweepArgs::best; uniform over the warp).
    __device__ __forceinline__ void finish(const Token& t, const Pair& p, int blk, int lane, unsigned long long& best) const {
        const int j = blk * kBlk + lane;
        // d^2 = a_i + a_j - 2 (g w_col) w_row, row the lower index: the operations and their order as in the sweep
        const float w_row = t.i < j ? t.w : p.w, w_col = t.i < j ? p.w : t.w;
        const float d2 = fmaxf(fmaf(p.gram * w_col, -2.f * w_row, METRIC == 0 ? 2.f : t.a + p.a), 0.f);
        bool usable = j < n && (p.rho > t.rho || (p.rho == t.rho && j < t.i));     // denser: (rho desc, index asc)
        if (SPATIAL) {
            const float dx = p.pos.x - t.pos.x, dy = p.pos.y - t.pos.y;
            usable = usable && fmaf(dx, dx, dy * dy) <= tau2;
        }
        const uint32_t key = usable ? __float_as_uint(d2) : kInfBits;
        const uint32_t m = __reduce_min_sync(0xffffffffu, key);
        if (m < kInfBits) {                                // lowest index among the block's nearest
            const uint32_t who = __ballot_sync(0xffffffffu, key == m);
            const unsigned long long cand =
                ((unsigned long long)m << 32) | (unsigned long long)(uint32_t)(blk * kBlk + __ffs(who) - 1);
            best = cand < best ? cand : best;
        }
    }
};

template <int METRIC, bool SPATIAL>
__global__ void __launch_bounds__(kNdThreads)
nearest_denser_kernel(const __grid_constant__ SweepArgs g) {
    // A kernel queued behind this one that does not depend on it may share the SMs from the start.
    grid_dependency_launch_dependents();
    grid_dependency_wait();                                // densities, factors, Gram values and minima come from the kernels before
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    const int b = blockIdx.y, i = blockIdx.x * kNdWarps + warp;
    if (i >= g.n) return;                                  // (uniform)
    const Sample<METRIC, SPATIAL> s(g, b);
    const float* const row = s.minima + (size_t)i * s.row;
    const auto t = s.token(i);
    uint32_t m1 = kInfBits, m2 = kInfBits;                 // this lane's two smallest keys
    for (int k0 = lane; k0 < s.nb; k0 += 128) {
        uint32_t v[4];
#pragma unroll
        for (int u = 0; u < 4; ++u) v[u] = k0 + u * 32 < s.nb ? __float_as_uint(row[k0 + u * 32]) : kInfBits;
#pragma unroll
        for (int u = 0; u < 4; ++u) {
            const uint32_t key = v[u] >= kInfBits ? kInfBits : ((v[u] & ~kBlkMask) | (uint32_t)(k0 + u * 32));
            m2 = min(m2, max(m1, key));
            m1 = min(m1, key);
        }
    }
    const bool more = lane + 64 < s.nb;                    // this lane has blocks beyond the two it remembers
    int taken = 0;                                         // blocks of this lane looked into
    unsigned long long best = ~0ull;
    // The smallest key left, or kInfBits if no block can hold a token below `best` any more.  A lane whose two blocks are
    // taken stands for the rest of its blocks with the larger key (`known` false).
    auto next = [&](bool& known) {
        const uint32_t least = __reduce_min_sync(0xffffffffu, m1);
        known = true;
        if (least >= kInfBits || (least & ~kBlkMask) > (uint32_t)(best >> 32)) return kInfBits;
        const bool mine = m1 == least;                     // (keys are distinct but for a lane's stand-in)
        known = !__any_sync(0xffffffffu, mine && taken == 2);
        if (known && mine) {
            ++taken;
            m1 = (taken == 2 && !more) ? kInfBits : m2;
        }
        return least;
    };
    bool open = true;
#pragma unroll 1
    for (int round = 0; round < kNdRounds; ++round) {
        bool known0, known1 = false;
        const uint32_t k0 = next(known0);
        open = k0 < kInfBits;
        if (!open || !known0) break;
        const uint32_t k1 = next(known1);
        const int b0 = (int)(k0 & kBlkMask), b1 = (int)(k1 & kBlkMask);
        const auto p0 = s.fetch(i, b0, lane);
        const bool two = k1 < kInfBits && known1;          // (uniform)
        auto p1 = p0;
        if (two) p1 = s.fetch(i, b1, lane);
        s.finish(t, p0, b0, lane, best);
        if (two) s.finish(t, p1, b1, lane, best);
    }
    if (open) {
        const uint32_t least = __reduce_min_sync(0xffffffffu, m1);
        open = least < kInfBits && (least & ~kBlkMask) <= (uint32_t)(best >> 32);
    }
    if (lane == 0) {
        g.best[(size_t)b * g.n + i] = best;
        if (open) g.left[atomicAdd(g.n_left, 1)] = b * g.n + i;
    }
}

// The tokens left over, each shared out over `slices` warps: warp w of a token takes the blocks w, w + slices, .. that are
// still open and hold a denser token.  (Those the first kernel has looked into already cannot improve on its result.)
template <int METRIC, bool SPATIAL>
__global__ void __launch_bounds__(kNdThreads)
nearest_left_kernel(const __grid_constant__ SweepArgs g, const int slices) {
    grid_dependency_launch_dependents();
    grid_dependency_wait();
    const int lane = threadIdx.x & 31;
    const long long items = (long long)*g.n_left * slices;
    for (long long q = (long long)blockIdx.x * kNdWarps + (threadIdx.x >> 5); q < items; q += (long long)gridDim.x * kNdWarps) {
        const int at = g.left[q / slices], slice = (int)(q % slices), b = at / g.n, i = at - b * g.n;
        const Sample<METRIC, SPATIAL> s(g, b);
        const auto t = s.token(i);
        const unsigned long long known = __ldcg(g.best + at);      // (other warps may be lowering it: a stale one is only looser)
        unsigned long long best = known;
        // Can block k, with minimum `lo`, hold a token below `best`?  (An equal distance at a lower index would win.)
        auto can = [&](uint32_t lo, int k) {
            return lo < kInfBits && (((unsigned long long)lo << 32) | (unsigned long long)(uint32_t)(k * kBlk)) < best;
        };
        for (int k0 = slice; k0 < s.nb; k0 += 32 * slices) {
            const int k = k0 + lane * slices;
            uint32_t lo = kInfBits, top = 0u;
            if (k < s.nb) {
                top = s.top[k];
                lo = __float_as_uint(s.minima[(size_t)i * s.row + k]);
            }
            if (top < __float_as_uint(t.rho)) lo = kInfBits;
            uint32_t todo = __ballot_sync(0xffffffffu, can(lo, k));
            while (todo) {
                typename Sample<METRIC, SPATIAL>::Pair p[kNdAhead];
                int blk[kNdAhead];
                int cnt = 0;
#pragma unroll
                for (int u = 0; u < kNdAhead; ++u) {
                    if (todo) {
                        blk[u] = k0 + (__ffs(todo) - 1) * slices;
                        todo &= todo - 1;
                        p[u] = s.fetch(i, blk[u], lane);
                        cnt = u + 1;
                    }
                }
#pragma unroll
                for (int u = 0; u < kNdAhead; ++u)
                    if (u < cnt) s.finish(t, p[u], blk[u], lane, best);
                todo &= __ballot_sync(0xffffffffu, can(lo, k));
            }
        }
        if (lane == 0 && best < known) atomicMin(g.best + at, best);
    }
}

}  // namespace

int launch_nearest_denser(const SweepArgs& args, int metric, cudaStream_t stream, bool pdl) {
    if (args.B <= 0 || args.n <= 0) return VITCOP_OK;
    if (!args.gram || !args.blk_min || !args.blk_rho || !args.best || !args.left || !args.n_left) return VITCOP_ERR_INVALID_ARG;
    const bool spatial = args.tau2 >= 0.f && args.pos != nullptr;
    cudaLaunchConfig_t cfg = {};
    cfg.gridDim = dim3((unsigned)((args.n + kNdWarps - 1) / kNdWarps), (unsigned)args.B);
    cfg.blockDim = dim3(kNdThreads);
    cfg.stream = stream;
    cudaLaunchAttribute attr[1];
    attr[0].id = cudaLaunchAttributeProgrammaticStreamSerialization;
    attr[0].val.programmaticStreamSerializationAllowed = 1;
    cfg.attrs = attr;
    cfg.numAttrs = pdl_allowed(pdl) ? 1 : 0;
    auto kern = metric == 1 ? (spatial ? nearest_denser_kernel<1, true> : nearest_denser_kernel<1, false>)
                            : (spatial ? nearest_denser_kernel<0, true> : nearest_denser_kernel<0, false>);
    int rc;
    {
        KernelTimeScope timed("nearest_denser_kernel", stream);
        rc = record_cuda(cudaLaunchKernelEx(&cfg, kern, args));
        if (rc != VITCOP_OK) return rc;
    }
    int slices = 2;                                        // at most 32 blocks a warp: one per lane
    while (slices * 32 < args.t.n_blk()) slices *= 2;
    const long long most = ((long long)args.B * args.n * slices + kNdWarps - 1) / kNdWarps, ctas = 6LL * gram_num_sms();
    cfg.gridDim = dim3((unsigned)(most < ctas ? most : ctas));
    auto rest = metric == 1 ? (spatial ? nearest_left_kernel<1, true> : nearest_left_kernel<1, false>)
                            : (spatial ? nearest_left_kernel<0, true> : nearest_left_kernel<0, false>);
    KernelTimeScope timed("nearest_left_kernel", stream);
    return record_cuda(cudaLaunchKernelEx(&cfg, rest, args, slices));
}

}  // namespace vitcop
