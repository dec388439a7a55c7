// Eq. 3 (Algorithm 2, step 2): per token the nearest denser token inside the spatial radius, searched in what the
// density sweep left behind (density.cuh): every Gram value of the symmetric half, and per (token, block of 32 tokens) the
// smallest squared distance.
//
// A block can hold a token's answer only if its minimum is not above the best denser token found so far.  One warp per token:
// every lane keeps the two smallest minima among its blocks (block % 32 = lane) and the warp looks into the blocks in
// ascending order, two at a time (lane = token of the block: the Gram value, the factors, the density and the spatial test).
// For nine tokens in ten two rounds are enough: their nearest neighbours include a denser token (half of all tokens need one
// block).  The few tokens that are the densest of their surroundings may have to look into dozens of blocks; these are left to
// the whole CTA, whose warps share out the token's blocks, passing over those without a denser token (largest density of the
// block): a warp alone would hold up the kernel.  What is skipped could not have changed the minimum, and d^2 is recomputed
// from the stored value with the arithmetic of the sweep (and of the one-kernel sweep), so the result has the same bits as a
// full pass over the pairs.
//
// The kernel is bound by the latency of its dependent trips to memory (minima, blocks, blocks again), hence few registers and
// as many warps as fit.
#include "density.cuh"

namespace vitcop {
namespace {

constexpr int kNdThreads = 256, kNdWarps = kNdThreads / 32;
constexpr int kNdRounds = 2;                               // rounds of two blocks that a warp does for its own token
constexpr uint32_t kInfBits = 0x7f800000u;
// A lane orders its blocks by a key: the bits of the minimum (never negative) with the block's number in the low bits, i.e. a
// bound up to 2^-14 too low.
constexpr uint32_t kBlkMask = VITCOP_MAX_VISUAL_TOKENS / kBlk - 1;
static_assert((kBlkMask & (kBlkMask + 1)) == 0 && kBlkMask < (1u << 10), "block numbers fit the low bits of a key");

template <int METRIC, bool SPATIAL>
__global__ void __launch_bounds__(kNdThreads, 5)
nearest_denser_kernel(const __grid_constant__ SweepArgs g) {
    __shared__ unsigned long long s_best[kNdWarps];        // (d^2 bits, index) of the CTA's tokens
    __shared__ int s_list[kNdWarps];                       // tokens left to the CTA
    __shared__ int s_count;
    // A kernel queued behind this one that does not depend on it may share the SMs from the start.
    grid_dependency_launch_dependents();
    if (threadIdx.x == 0) s_count = 0;
    grid_dependency_wait();                                // densities, factors, Gram values and minima come from the kernels before
    __syncthreads();
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    const int b = blockIdx.y, n = g.n;
    const int i0 = blockIdx.x * kNdWarps;
    const int nb = (n + kBlk - 1) / kBlk;                  // blocks that hold tokens
    const size_t bo = (size_t)b * n;
    const float* const rho_b = g.rho + bo;
    const float* const w_b = g.w + bo;
    const float* const a_b = g.a + bo;
    const float2* const pos_b = SPATIAL ? reinterpret_cast<const float2*>(g.pos) + bo : nullptr;
    const float* const blocks = g.gram + (size_t)b * g.t.tiles_per_b * kSweepTileFloats;
    const float* const min_b = g.blk_min + (size_t)b * g.t.n_pad * g.t.n_blk();
    const uint32_t* const blk_rho = g.blk_rho + (size_t)b * g.t.n_blk();

    struct Token {
        int i;
        float rho, w, a;
        float2 pos;
    };
    auto token = [&](int i) {
        Token t;
        t.i = i;
        t.rho = rho_b[i];
        t.w = w_b[i];
        t.a = METRIC == 1 ? a_b[i] : 1.f;
        t.pos = SPATIAL ? pos_b[i] : make_float2(0.f, 0.f);
        return t;
    };
    struct Pair {                                          // what a lane needs of the pair (i, 32 blk + lane)
        float gram, w, rho, a;
        float2 pos;
    };
    auto fetch = [&](int i, int blk) {
        Pair p;
        const int j = min(blk * kBlk + lane, n - 1), own = i / kBlk, ri = i % kBlk;
        // the pair's lower index is its row (inside the own block: in either order)
        const bool below = blk < own || (blk == own && lane < ri);
        const int r = below ? lane : ri, c = below ? ri : lane;
        p.gram = blocks[gram_block_offset(min(blk, own), max(blk, own)) + gram_elem_offset(r, c)];
        p.w = w_b[j];
        p.rho = rho_b[j];
        p.a = METRIC == 1 ? a_b[j] : 1.f;
        p.pos = SPATIAL ? pos_b[j] : make_float2(0.f, 0.f);
        return p;
    };
    // Folds the block's nearest denser token into `best` (uniform).
    auto finish = [&](const Token& t, const Pair& p, int blk, unsigned long long& best) {
        const int j = blk * kBlk + lane;
        // d^2 = a_i + a_j - 2 (g w_col) w_row, row the lower index: the operations and their order as in the sweep
        const float w_row = t.i < j ? t.w : p.w, w_col = t.i < j ? p.w : t.w;
        const float d2 = fmaxf(fmaf(p.gram * w_col, -2.f * w_row, METRIC == 0 ? 2.f : t.a + p.a), 0.f);
        bool usable = j < n && (p.rho > t.rho || (p.rho == t.rho && j < t.i));     // denser: (rho desc, index asc)
        if (SPATIAL) {
            const float dx = p.pos.x - t.pos.x, dy = p.pos.y - t.pos.y;
            usable = usable && fmaf(dx, dx, dy * dy) <= g.tau2;
        }
        const uint32_t key = usable ? __float_as_uint(d2) : kInfBits;
        const uint32_t m = __reduce_min_sync(0xffffffffu, key);
        if (m < kInfBits) {                                // lowest index among the block's nearest
            const uint32_t who = __ballot_sync(0xffffffffu, key == m);
            const unsigned long long cand =
                ((unsigned long long)m << 32) | (unsigned long long)(uint32_t)(blk * kBlk + __ffs(who) - 1);
            best = cand < best ? cand : best;
        }
    };

    // ---- each warp its own token
    const int i = i0 + warp;
    if (i < n) {                                           // (uniform)
        const float* const row = min_b + (size_t)i * g.t.n_blk();
        uint32_t m1 = kInfBits, m2 = kInfBits;             // this lane's two smallest keys
        for (int k0 = lane; k0 < nb; k0 += 128) {
            uint32_t v[4];
#pragma unroll
            for (int u = 0; u < 4; ++u) v[u] = k0 + u * 32 < nb ? __float_as_uint(row[k0 + u * 32]) : kInfBits;
#pragma unroll
            for (int u = 0; u < 4; ++u) {
                const uint32_t key = v[u] >= kInfBits ? kInfBits : ((v[u] & ~kBlkMask) | (uint32_t)(k0 + u * 32));
                m2 = min(m2, max(m1, key));
                m1 = min(m1, key);
            }
        }
        const Token t = token(i);
        const bool more = lane + 64 < nb;                  // this lane has blocks beyond the two it remembers
        int taken = 0;                                     // blocks of this lane looked into
        unsigned long long best = ~0ull;
        // The smallest key left, or kInfBits if no block can hold a token below `best` any more.  A lane whose two blocks are
        // taken stands for the rest of its blocks with the larger key (`known` false).
        auto next = [&](bool& known) {
            const uint32_t least = __reduce_min_sync(0xffffffffu, m1);
            known = true;
            if (least >= kInfBits || (least & ~kBlkMask) > (uint32_t)(best >> 32)) return kInfBits;
            const bool mine = m1 == least;                 // (keys are distinct but for a lane's stand-in)
            known = !__any_sync(0xffffffffu, mine && taken == 2);
            if (known && mine) {
                ++taken;
                m1 = (taken == 2 && !more) ? kInfBits : m2;
            }
            return least;
        };
        bool open = true;
#pragma unroll 1
        for (int round = 0; open && round < kNdRounds; ++round) {
            bool known0, known1 = false;
            const uint32_t k0 = next(known0);
            if (k0 >= kInfBits) { open = false; break; }
            if (!known0) break;
            const uint32_t k1 = next(known1);
            const int b0 = (int)(k0 & kBlkMask), b1 = (int)(k1 & kBlkMask);
            const Pair p0 = fetch(i, b0);
            const bool two = k1 < kInfBits && known1;      // (uniform)
            Pair p1 = p0;
            if (two) p1 = fetch(i, b1);
            finish(t, p0, b0, best);
            if (two) finish(t, p1, b1, best);
            const uint32_t least = __reduce_min_sync(0xffffffffu, m1);
            open = least < kInfBits && (least & ~kBlkMask) <= (uint32_t)(best >> 32);
        }
        if (lane == 0) {
            s_best[warp] = best;
            if (open) s_list[atomicAdd(&s_count, 1)] = warp;
        }
    }
    __syncthreads();
    // ---- the tokens left over: warp w takes the blocks w, w + 8, .. that are still open and hold a denser token.  (Those the
    //      token's own warp has looked into already cannot improve on it.)
    const int left = s_count;
    for (int q = 0; q < left; ++q) {
        const int tw = s_list[q];
        const Token t = token(i0 + tw);
        unsigned long long best = s_best[tw];              // (other warps may be lowering it: a stale one is only looser)
        // Can block k, with minimum `lo`, hold a token below `best`?  (An equal distance at a lower index would win.)
        auto can = [&](uint32_t lo, int k) {
            return lo < kInfBits && (((unsigned long long)lo << 32) | (unsigned long long)(uint32_t)(k * kBlk)) < best;
        };
        for (int k0 = warp; k0 < nb; k0 += 32 * kNdWarps) {
            const int k = k0 + lane * kNdWarps;
            uint32_t lo = kInfBits, top = 0u;
            if (k < nb) {
                top = blk_rho[k];
                lo = __float_as_uint(min_b[(size_t)t.i * g.t.n_blk() + k]);
            }
            if (top < __float_as_uint(t.rho)) lo = kInfBits;
            uint32_t todo = __ballot_sync(0xffffffffu, can(lo, k));
            while (todo) {
                const int b0 = k0 + (__ffs(todo) - 1) * kNdWarps;
                todo &= todo - 1;
                const Pair p0 = fetch(t.i, b0);
                const int b1 = todo ? k0 + (__ffs(todo) - 1) * kNdWarps : -1;
                todo &= todo - 1;
                Pair p1 = p0;
                if (b1 >= 0) p1 = fetch(t.i, b1);
                finish(t, p0, b0, best);
                if (b1 >= 0) finish(t, p1, b1, best);
                todo &= __ballot_sync(0xffffffffu, can(lo, k));
            }
        }
        if (lane == 0) atomicMin(&s_best[tw], best);
    }
    __syncthreads();
    if (threadIdx.x < kNdWarps && i0 + threadIdx.x < n) g.best[bo + i0 + threadIdx.x] = s_best[threadIdx.x];
}

}  // namespace

int launch_nearest_denser(const SweepArgs& args, int metric, cudaStream_t stream, bool pdl) {
    if (args.B <= 0 || args.n <= 0) return VITCOP_OK;
    if (!args.gram || !args.blk_min || !args.blk_rho || !args.best) return VITCOP_ERR_INVALID_ARG;
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
    KernelTimeScope timed("nearest_denser_kernel", stream);
    return record_cuda(cudaLaunchKernelEx(&cfg, kern, args));
}

}  // namespace vitcop
