// Eq. 3 (Algorithm 2, step 2): per token the nearest denser token inside the spatial radius, searched in what the
// density sweep left behind (density.cuh): every Gram value of the symmetric half, and per (token, block of 32 tokens) the
// smallest squared distance.
//
// A block can hold a token's answer only if it has a denser token (largest density of the block) and its minimum is not above
// the best denser token found so far.  One warp per token: every lane keeps the two smallest minima among its blocks
// (block % 32 = lane) and the warp looks into the blocks in ascending order, two at a time (lane = token of the block: the
// Gram value and one 16-byte record with factor, density and position).  For nine tokens in ten a few rounds are enough: their
// nearest neighbours include a denser token (half of all tokens need one block).  The few tokens that are the densest of
// their surroundings may have to look into dozens of blocks; these are listed and left to a second kernel, in which
// several warps share out a token's blocks: a warp alone would hold up everything behind it.  What is skipped could not have
// changed the minimum, and d^2 is recomputed from the stored value with the arithmetic of the sweep (and of the one-kernel
// sweep), so the result has the same bits as a full pass over the pairs.
//
// Both kernels are bound by instruction issue (0.73 and 0.57 per cycle; the data sits in L2), so a lane carries its own best pair
// from block to block and the warp exchanges only the bound; the place of a value is one add and one select away from the
// token's.  Measured on 8 x 2880 tokens, caches warm: 19.7 -> 15.1 us and 18.3 -> 13.9 us against a warp-wide minimum and ballot
// per block and four separate loads per token.  Passing over blocks without a denser token in the first kernel too: 6 us less on
// 4 x 4096 tokens.
#include "density.cuh"

namespace vitcop {
namespace {

constexpr int kNdThreads = 256, kNdWarps = kNdThreads / 32;
// Rounds of two blocks that a warp of the first kernel does for its own token, and blocks that a warp of the second looks into at a time: four and
// three (three, five and six rounds take as long on 8 x 2880 and 4 x 4608 tokens and up to 3 us longer on 2 x 16384).  Three and four where the
// chip holds the tokens' warps (64 an SM), up to 4096 tokens to a sample one and a half times as many: the first kernel lasts as long as its longest
// warps there, and the second has idle SMs for what is left.  64 steps on such calls, four and three / three and four: 44 on videos 1.0 %
// less, 20 on images 1.2 % (4 x 3420 tokens of a video 125.1 / 122.4 us, 3 x 3143 99.5 / 98.5).  Beyond that line 1 to 2 % more (2 x 5600 to 6800
// tokens without structure 4 to 5 %), and beyond 8192 tokens to a sample with few samples too.
bool few_tokens(long long tokens, int n) {
    const long long held = 64LL * gram_num_sms();
    return n <= 8192 && (tokens <= held || (n <= 4096 && 2 * tokens <= 3 * held));
}
constexpr uint32_t kInfBits = 0x7f800000u;
// A lane orders its blocks by a key: the bits of the minimum (never negative) with the block's number in the low bits, above it
// one bit that marks a stand-in; i.e. a bound up to 2^-13 too low.
constexpr uint32_t kBlkMask = VITCOP_MAX_VISUAL_TOKENS / kBlk - 1;
constexpr uint32_t kStandIn = kBlkMask + 1, kKeyMask = kStandIn | kBlkMask;
static_assert((kBlkMask & (kBlkMask + 1)) == 0 && kBlkMask < (1u << 10), "block numbers fit the low bits of a key");
static_assert((size_t)(VITCOP_MAX_VISUAL_TOKENS / kSweepTile) * (VITCOP_MAX_VISUAL_TOKENS / kSweepTile + 1) / 2 * kSweepTileFloats <
                  (1u << 31), "a sample's Gram values are indexed with 32 bits");

// One token's search as one lane sees it: the lane stands for one token of every block that the warp looks into, and keeps the
// nearest denser one it has met (bits of d^2, block; none: kInfBits).
template <int METRIC, bool SPATIAL>
struct Search {
    const float* gram;                                     // of the sample
    const float4* tok;                                     // of the sample, from this lane on
    int i, lane;
    float4 t;                                              // (factor, density, position) of the token
    float rho_next;                                        // the next density above the token's
    float tau2;
    uint32_t base_col, base_row;                           // this lane's value of block (k, own) is at base_col + k * kRowStep ..
    uint32_t best = kInfBits;
    int best_blk = 0;
    static constexpr uint32_t kRowStep = kSweepBlks * kBlk * kBlk;             // block (k, own) to block (k + 1, own)
    __device__ __forceinline__ Search(const SweepArgs& g, int b, int i_, int lane_) : i(i_), lane(lane_), tau2(g.tau2) {
        gram = g.gram + (size_t)b * g.t.tiles_per_b * kSweepTileFloats;
        tok = g.tok + (size_t)b * g.t.n_pad;
        t = tok[i];
        tok += lane;
        rho_next = __uint_as_float(__float_as_uint(t.y) + 1u);
        const int own = i / kBlk, ri = i % kBlk;
        base_col = (uint32_t)gram_block_offset(0, own) + (uint32_t)gram_elem_offset(lane, ri);
        base_row = (uint32_t)own * kRowStep + (uint32_t)gram_elem_offset(ri, lane);
    }
    struct Pair {                                          // of the pair (i, 32 blk + lane)
        float gram;
        float4 t;
    };
    // (in front of the token: a column of block (blk, own), whose rows follow one another tile after tile)
    __device__ __forceinline__ bool below(int blk) const { return blk * kBlk + lane < i; }
    __device__ __forceinline__ Pair fetch(int blk) const {
        const uint32_t tj = (uint32_t)blk / kSweepBlks;
        const uint32_t row = base_row + tj * (tj + 1) / 2 * (uint32_t)kSweepTileFloats + (uint32_t)blk % kSweepBlks * (kBlk * kBlk);
        Pair p;
        p.gram = gram[below(blk) ? base_col + (uint32_t)blk * kRowStep : row];
        p.t = tok[blk * kBlk];
        return p;
    }
    __device__ __forceinline__ void look(const Pair& p, int blk) {
        const bool lower = below(blk);                     // this lane's token has the lower index
        // d^2 = a_i + a_j - 2 (g w_col) w_row, row the lower index: the operations and their order as in the sweep
        float d2;
        if (METRIC == 0) d2 = fmaf(p.gram * (lower ? t.x : p.t.x), -2.f * (lower ? p.t.x : t.x), 2.f);
        else d2 = fmaf(p.gram, -2.f, t.x + p.t.x);
        bool usable = p.t.y >= (lower ? t.y : rho_next);   // denser: (rho desc, index asc)
        if (SPATIAL) {
            const float dx = p.t.z - t.z, dy = p.t.w - t.w;
            usable = usable && fmaf(dx, dx, dy * dy) <= tau2;
        }
        const uint32_t key = __float_as_uint(fmaxf(d2, 0.f));
        if (usable && (key < best || (key == best && blk < best_blk))) {
            best = key;
            best_blk = blk;
        }
    }
    // uniform over the warp: the smallest d^2 so far, and all of it packed as SweepArgs::best
    __device__ __forceinline__ uint32_t bound() const { return __reduce_min_sync(0xffffffffu, best); }
    __device__ __forceinline__ unsigned long long packed(uint32_t bound) const {
        const uint32_t j = __reduce_min_sync(0xffffffffu, best == bound ? (uint32_t)(best_blk * kBlk + lane) : ~0u);
        return bound < kInfBits ? ((unsigned long long)bound << 32) | j : ~0ull;       // (the lowest index among the nearest)
    }
};

template <int METRIC, bool SPATIAL>
__global__ void __launch_bounds__(kNdThreads)
nearest_denser_kernel(const __grid_constant__ SweepArgs g, const int rounds) {
    // A kernel queued behind this one that does not depend on it may share the SMs from the start.
    grid_dependency_launch_dependents();
    grid_dependency_wait();                                // densities, factors, Gram values and minima come from the kernels before
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    const int b = blockIdx.y, i = blockIdx.x * kNdWarps + warp;
    if (i >= g.n) return;                                  // (uniform)
    const int nb = (g.n + kBlk - 1) / kBlk, n_blk = g.t.n_blk();
    const float* const row = g.blk_min + ((size_t)b * g.t.n_pad + i) * n_blk;
    const uint32_t* const top = g.blk_rho + (size_t)b * n_blk;       // largest density of every block
    Search<METRIC, SPATIAL> s(g, b, i, lane);
    uint32_t m1 = kInfBits, m2 = kInfBits;                 // this lane's two smallest keys
    for (int k0 = lane; k0 < nb; k0 += 128) {
        uint32_t v[4], dens[4];
#pragma unroll
        for (int u = 0; u < 4; ++u) {
            v[u] = k0 + u * 32 < nb ? __float_as_uint(__ldcg(row + k0 + u * 32)) : kInfBits;
            dens[u] = k0 + u * 32 < nb ? top[k0 + u * 32] : 0u;
        }
#pragma unroll
        for (int u = 0; u < 4; ++u) {
            const uint32_t key = v[u] >= kInfBits || dens[u] < __float_as_uint(s.t.y) ? kInfBits : ((v[u] & ~kKeyMask) | (uint32_t)(k0 + u * 32));
            m2 = min(m2, max(m1, key));
            m1 = min(m1, key);
        }
    }
    // A lane whose two blocks are taken stands for the rest of its blocks, if it has any, with the larger key.
    const uint32_t rest = lane + 64 < nb ? kStandIn : kInfBits;
    uint32_t bound = kInfBits, least = __reduce_min_sync(0xffffffffu, m1);
    auto can = [&](uint32_t key) { return key < kInfBits && (key & ~kKeyMask) <= bound; };       // may hold a nearer token
    auto take = [&]() {                                    // `least` is looked into; the next one
        if (m1 == least) {                                 // (keys are distinct)
            m1 = m2;
            m2 |= rest;
        }
        least = __reduce_min_sync(0xffffffffu, m1);
    };
#pragma unroll 1
    for (int round = 0; round < rounds && can(least) && !(least & kStandIn); ++round) {
        const int b0 = (int)(least & kBlkMask);
        const auto p0 = s.fetch(b0);
        take();
        const bool two = can(least) && !(least & kStandIn);
        const int b1 = (int)(least & kBlkMask);
        auto p1 = p0;
        if (two) {
            p1 = s.fetch(b1);
            take();
        }
        s.look(p0, b0);
        if (two) s.look(p1, b1);
        bound = s.bound();
    }
    const unsigned long long best = s.packed(bound);
    if (lane == 0) {
        g.best[(size_t)b * g.n + i] = best;
        if (can(least)) g.left[atomicAdd(g.n_left, 1)] = b * g.n + i;
    }
}

// The tokens left over, each shared out over `slices` warps: warp w of a token takes the blocks w, w + slices, .. that are
// still open and hold a denser token.  (Those the first kernel has looked into already cannot improve on its result.)
// Each warp in ascending order of its blocks' minima: in the order of their numbers it looked into more of them (2 x 16384 tokens
// of no structure 128.6 -> 117.5 us; 4 x 4608 of a video, whole call, 212 -> 209).  Two or four times as many or as few blocks per warp
// measured the same or worse.  What one warp finds it tells the token's others at once, and what they have found travels with its
// blocks: alone, a warp goes on below a bound that another one has lowered long since (2 x 16384 tokens 41 -> 25 us;
// of no structure, whole call, 1000 -> 754).
template <int METRIC, bool SPATIAL, int AHEAD>
__global__ void __launch_bounds__(kNdThreads)
nearest_left_kernel(const __grid_constant__ SweepArgs g, const int slices) {
    grid_dependency_launch_dependents();
    grid_dependency_wait();
    const int lane = threadIdx.x & 31;
    const int nb = (g.n + kBlk - 1) / kBlk, n_blk = g.t.n_blk();
    const long long items = (long long)*g.n_left * slices;
    for (long long q = (long long)blockIdx.x * kNdWarps + (threadIdx.x >> 5); q < items; q += (long long)gridDim.x * kNdWarps) {
        const int at = g.left[q / slices], slice = (int)(q % slices), b = at / g.n, i = at - b * g.n;
        const float* const row = g.blk_min + ((size_t)b * g.t.n_pad + i) * n_blk;
        const uint32_t* const top = g.blk_rho + (size_t)b * n_blk;   // largest density of every block
        Search<METRIC, SPATIAL> s(g, b, i, lane);
        // (other warps may be lowering it: a stale one is only looser, but all lanes must go by the same one, as it decides which of
        // them meet in the reductions below)
        unsigned long long best = __shfl_sync(0xffffffffu, lane == 0 ? __ldcg(g.best + at) : 0ull, 0);
        // Can block k, with minimum `lo`, hold a token below `best`?  (An equal distance at a lower index would win.)
        auto can = [&](uint32_t lo, int k) {
            return lo < kInfBits && (((unsigned long long)lo << 32) | (unsigned long long)(uint32_t)(k * kBlk)) < best;
        };
        for (int k0 = slice; k0 < nb; k0 += 32 * slices) {
            const int k = k0 + lane * slices;
            uint32_t lo = kInfBits, dens = 0u;
            if (k < nb) {
                dens = top[k];
                lo = __float_as_uint(__ldcg(row + k));
            }
            if (dens < __float_as_uint(s.t.y)) lo = kInfBits;
            // in ascending order of the minima, several at a time: the first ones are the likeliest to hold the answer, and
            // none behind the first that cannot hold it can
            for (;;) {
                typename Search<METRIC, SPATIAL>::Pair p[AHEAD];
                int blk[AHEAD];
                int cnt = 0;
#pragma unroll
                for (int u = 0; u < AHEAD; ++u) {
                    const uint32_t m = __reduce_min_sync(0xffffffffu, lo);
                    const int who = __ffs(__ballot_sync(0xffffffffu, lo == m)) - 1;
                    blk[u] = k0 + who * slices;
                    if (cnt == u && can(m, blk[u])) {
                        if (lane == who) lo = kInfBits;
                        p[u] = s.fetch(blk[u]);
                        cnt = u + 1;
                    }
                }
                if (cnt == 0) break;
                // (what the token's other warps have found by now travels with the blocks)
                const unsigned long long others = lane == 0 ? __ldcg(g.best + at) : 0ull;
#pragma unroll
                for (int u = 0; u < AHEAD; ++u)
                    if (u < cnt) s.look(p[u], blk[u]);
                const unsigned long long found = s.packed(s.bound());
                if (found < best) {
                    best = found;
                    if (lane == 0) atomicMin(g.best + at, best);
                }
                const unsigned long long theirs = __shfl_sync(0xffffffffu, others, 0);
                best = theirs < best ? theirs : best;
            }
        }
    }
}

}  // namespace

int launch_nearest_denser(const SweepArgs& args, int metric, cudaStream_t stream, bool pdl) {
    if (args.B <= 0 || args.n <= 0) return VITCOP_OK;
    if (!args.gram || !args.blk_min || !args.blk_rho || !args.tok || !args.best || !args.left || !args.n_left) return VITCOP_ERR_INVALID_ARG;
    const bool spatial = args.tau2 >= 0.f && args.pos != nullptr, few = few_tokens((long long)args.B * args.n, args.n);
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
        rc = record_cuda(cudaLaunchKernelEx(&cfg, kern, args, few ? 3 : 4));
        if (rc != VITCOP_OK) return rc;
    }
    int slices = 2;                                        // at most 32 blocks a warp: one per lane
    while (slices * 32 < args.t.n_blk()) slices *= 2;
    const long long most = ((long long)args.B * args.n * slices + kNdWarps - 1) / kNdWarps, ctas = 6LL * gram_num_sms();
    cfg.gridDim = dim3((unsigned)(most < ctas ? most : ctas));
    auto pick = [&](auto four, auto three) { return few ? four : three; };
    auto rest = metric == 1 ? (spatial ? pick(nearest_left_kernel<1, true, 4>, nearest_left_kernel<1, true, 3>)
                                       : pick(nearest_left_kernel<1, false, 4>, nearest_left_kernel<1, false, 3>))
                            : (spatial ? pick(nearest_left_kernel<0, true, 4>, nearest_left_kernel<0, true, 3>)
                                       : pick(nearest_left_kernel<0, false, 4>, nearest_left_kernel<0, false, 3>));
    KernelTimeScope timed("nearest_left_kernel", stream);
    return record_cuda(cudaLaunchKernelEx(&cfg, rest, args, slices));
}

}  // namespace vitcop
