// Density sweep (Algorithm 2, step 1 and Eq. 2) of problems too large for the one-kernel sweep: every Gram value of the
// symmetric half on the tensor cores, partial sums of Eq. 2, and what the search of Eq. 3 needs (density.cuh: Gram values and
// block minima).
//
// Persistent clusters of two CTAs, one CTA per SM, each cluster on one 256 x 256 tile at a time (tcgen05 cta_group::2): a CTA
// stages its 128 row tokens and half of the column tokens, 32 KB per k-block instead of the 48 KB that a 128 x 256 tile of
// its own would take, so six k-blocks are in flight and the operand traffic from the L2, which bounds the main loop next to the
// tensor cores, falls by a third.  Warp 0 loads, one thread of the leader's warp 1 issues the MMAs into one of two
// accumulators, 16 epilogue warps per CTA drain the other, in two roles; warp (q, h) of either takes rows 32 q .. + 31 of the CTA
// and columns 128 h .. + 127, in four blocks of 32 x 32 pairs:
//   row warps      one row per thread: store the Gram values, take the row tokens' block minima and their sums of Eq. 2, column
//                  by column (that order of the sums is part of the result).
//   column warps   the column tokens' block minima and sums.  They read the accumulator in the 16-lanes x 256-bit shape: a
//                  thread holds 4 rows x 8 columns of a block, so that columns reduce partly inside the thread and only 8 values
//                  go through shuffles.  (With one row per thread every column costs a butterfly or a redux over 32 lanes.)
// Distances and exponentials are computed by both, which is cheaper than passing them on.  Two more warps fetch the factors of the
// next tile's tokens and join the column warps' parts of the previous one, so that neither the trip to the L2 nor the joining
// stands between two tiles.
//
// The sweep leaves the HBM mostly idle, so four warps more may compute a K-norm (Eq. 4) meanwhile, fed by tensor copies through the
// shared memory of one of the six stages.  (With plain loads the warps have too few of them in flight: 112 us for 188 MB of keys beside a sweep
// of 70; one warp with the copies, in the place of an auxiliary one, takes 126.  With more than five warps to a quarter of the SM a
// thread has 80 registers instead of 96.)
//
// Measured: 8 x 2880 x 1024 75 us (60 us with an empty epilogue), 2 x 16384 x 1280 519 us (433 us with an empty epilogue:
// 0.69 Tflop at the rate cuBLAS reaches in a burst; the stores of the Gram values are about 30 of the rest).  Sixteen warps of
// one role: 70 and 517 us, but another order of the sums.  A sweep of single SMs on 128 x 256 tiles, without the minima: 68 and
// 549 us.
//
// A last round of tiles that would occupy at most half of the clusters is cut into tiles of 128 columns.
// Every wait is bounded; on expiry both CTAs of the cluster leave in order and the call reports VITCOP_ERR_TIMEOUT.
#include "async_copy.cuh"
#include "density.cuh"
#include "f32x2.cuh"
#include "knorm.cuh"
#include "tcgen05.cuh"

namespace vitcop {
namespace {

constexpr int BM = kGramBM, BN = kSweepTile;
constexpr int kBoxRows = 64;                      // column tokens per load: a CTA stages one or two boxes
constexpr int kABytes = BM * BK * 2, kBBytes = BN / 2 * BK * 2, kStageBytes = kABytes + kBBytes;
constexpr int kHalfBlks = BM / kBlk;              // blocks of a warp: 128 columns
constexpr int kEpiWarps = 16, kEpiThreads = kEpiWarps * 32, kAuxThreads = 64;
constexpr int kTileThreads = kEpiThreads + kAuxThreads;   // meet once per tile
// A K-norm on the side has four warps more, and one of the six stages is its buffers.
constexpr int kKnWarps = 4, kKnHeads = 4, kKnBufBytes = 64 * kKnHeads * 16;
__host__ __device__ constexpr int threads(bool knorm) { return 64 + kTileThreads + (knorm ? kKnWarps * 32 : 0); }
constexpr float kInf = __builtin_huge_valf();
constexpr int kRoleLoad = 1, kRoleMma = 2, kRoleEpi = 4;

// Epilogue scratch, per parity of the tile: the factors of its tokens, which of its two 128-column halves lie beyond the spatial
// radius, sums and minima of the columns per row quarter, and the row minima of the block on the diagonal.
template <int METRIC>
struct EpiSmem {
    float colw[2][BN], rowm2w[2][BM];             // w_j; -2 w_i
    float cola[2][METRIC == 1 ? BN : 4], rowa[2][METRIC == 1 ? BM : 4];
    float colsum[2][4][BN], colmin[2][4][BN];
    float rowmin[2][BM][4];
    int far[2][4];
};
constexpr int kMaxStages = 6;
__host__ __device__ constexpr int stages(bool knorm) { return knorm ? kMaxStages - 1 : kMaxStages; }
static_assert(kKnWarps * 2 * kKnBufBytes == kStageBytes, "the K-norm's buffers");
template <int METRIC>
__host__ __device__ constexpr int smem_bytes() { return 1024 + kMaxStages * kStageBytes + (int)sizeof(EpiSmem<METRIC>) + 256; }
static_assert(smem_bytes<0>() <= 227 * 1024 && smem_bytes<1>() <= 227 * 1024, "shared memory of an SM");

struct KernelArgs {
    SweepArgs g;
    int n_full, n_items;           // tiles taken whole; work items (the other tiles count twice)
    float inv_tiles;               // 1 / tiles_per_b
    unsigned long long wait_ns;
    int expire_roles;
    __device__ __forceinline__ unsigned long long limit_of(int role) const { return (expire_roles & role) ? 0ull : wait_ns; }
};

// Work item: row tile tp against column tile tj of sample b, or the 128 columns of it that start at `half`.
struct Item {
    int b, tp, tj, half, halves;
    __device__ __forceinline__ bool one_operand() const { return tp == tj && halves == 2; }   // rows and columns are the same tokens
};
__device__ __forceinline__ Item decode_item(const KernelArgs& k, int t) {
    const int x = t - k.n_full;
    const int tile = x < 0 ? t : k.n_full + (x >> 1);
    Item it;
    it.halves = x < 0 ? 2 : 1;
    it.half = x < 0 ? 0 : (x & 1);
    // (every warp decodes every item, so without divisions: the estimates are off by one at most)
    const int per = k.g.t.tiles_per_b;
    int b = (int)((float)tile * k.inv_tiles);
    int r = tile - b * per;
    if (r < 0) { --b; r += per; }
    if (r >= per) { ++b; r -= per; }
    int q = (int)((__fsqrt_rn(8.f * (float)r + 1.f) - 1.f) * 0.5f);
    if (q * (q + 1) / 2 > r) --q;
    if ((q + 1) * (q + 2) / 2 <= r) ++q;
    it.b = b;
    it.tj = q;
    it.tp = r - q * (q + 1) / 2;
    return it;
}

// Smallest of the values, or NaN if one of them is none.
__device__ __forceinline__ float min2(float a, float b) {
    float r;
    asm("min.NaN.f32 %0, %1, %2;" : "=f"(r) : "f"(a), "f"(b));
    return r;
}
__device__ __forceinline__ float min3(float a, float b, float c) {
    float r;
    asm("min.NaN.f32 %0, %1, %2, %3;" : "=f"(r) : "f"(a), "f"(b), "f"(c));
    return r;
}

// 16 lanes x 32 columns of the accumulator: register 4 k + 2 p + r holds row T / 4 + 8 p, column 8 k + 2 (T % 4) + r.
__device__ __forceinline__ void tmem_ld_16x32_issue(uint32_t taddr, uint32_t* r) {
    asm volatile(
        "tcgen05.ld.sync.aligned.16x256b.x4.b32 {%0, %1, %2, %3, %4, %5, %6, %7, %8, %9, %10, %11, %12, %13, %14, %15}, [%16];"
        : "=r"(r[0]), "=r"(r[1]), "=r"(r[2]), "=r"(r[3]), "=r"(r[4]), "=r"(r[5]), "=r"(r[6]), "=r"(r[7]), "=r"(r[8]),
          "=r"(r[9]), "=r"(r[10]), "=r"(r[11]), "=r"(r[12]), "=r"(r[13]), "=r"(r[14]), "=r"(r[15])
        : "r"(taddr)
        : "memory");
}
// Completes the loads issued so far; names their registers, so that no use of them can be moved in front of it.
__device__ __forceinline__ void tmem_ld_wait32(uint32_t (&r)[32]) {
    asm volatile("tcgen05.wait::ld.sync.aligned;"
                 : "+r"(r[0]), "+r"(r[1]), "+r"(r[2]), "+r"(r[3]), "+r"(r[4]), "+r"(r[5]), "+r"(r[6]), "+r"(r[7]),
                   "+r"(r[8]), "+r"(r[9]), "+r"(r[10]), "+r"(r[11]), "+r"(r[12]), "+r"(r[13]), "+r"(r[14]), "+r"(r[15]),
                   "+r"(r[16]), "+r"(r[17]), "+r"(r[18]), "+r"(r[19]), "+r"(r[20]), "+r"(r[21]), "+r"(r[22]), "+r"(r[23]),
                   "+r"(r[24]), "+r"(r[25]), "+r"(r[26]), "+r"(r[27]), "+r"(r[28]), "+r"(r[29]), "+r"(r[30]), "+r"(r[31])
                 :
                 : "memory");
}

template <bool MIN>
__device__ __forceinline__ float join(float a, float b) { return MIN ? min2(a, b) : a + b; }
// Eight values per thread, value 2 k + r for column 8 k + 2 (T % 4) + r: afterwards the thread holds the total over the eight
// lanes with its T % 4 of column column_of(T), joined as a tree over the bits of T / 4, highest first.
template <bool MIN>
__device__ __forceinline__ float reduce_columns(const float (&v)[8], int lane) {
    const bool u16 = lane & 16, u8 = lane & 8, u4 = lane & 4;
    float a[4], b[2];
#pragma unroll
    for (int q = 0; q < 4; ++q)
        a[q] = join<MIN>(u16 ? v[q + 4] : v[q], __shfl_xor_sync(0xffffffffu, u16 ? v[q] : v[q + 4], 16));
#pragma unroll
    for (int q = 0; q < 2; ++q)
        b[q] = join<MIN>(u8 ? a[q + 2] : a[q], __shfl_xor_sync(0xffffffffu, u8 ? a[q] : a[q + 2], 8));
    return join<MIN>(u4 ? b[1] : b[0], __shfl_xor_sync(0xffffffffu, u4 ? b[0] : b[1], 4));
}
__device__ __forceinline__ int column_of(int lane) {
    return 8 * (((lane >> 4) & 1) * 2 + ((lane >> 3) & 1)) + 2 * (lane & 3) + ((lane >> 2) & 1);
}

// The K-norm (Eq. 4) of the job's samples, shared out over the side warps of all CTAs.  A warp takes 64 16-byte lanes of tokens at a time
// (4 tokens of d = 128, 8 of d = 64), kKnHeads heads per copy into one of its two buffers; a lane carries two of the tokens, so
// that two chains of sums are under way, with the arithmetic and the order of the stand-alone kernel (LPR lanes a token).
template <int LPR>
__device__ __forceinline__ void side_knorm(const KnormJob& kn, const CUtensorMap* map_k, const uint8_t* buf_gen, uint32_t buf_smem, uint32_t bars,
                                           int slot, int slots, volatile int* abort_flag, unsigned long long limit_ns) {
    constexpr int kTok = 2 * (32 / LPR);                   // tokens of a unit
    const int lane = threadIdx.x & 31, sub = lane % LPR, tk = lane / LPR;
    const int per_b = (kn.Nv + kTok - 1) / kTok, units = kn.B * per_b, parts = (kn.H + kKnHeads - 1) / kKnHeads;
    const int copies = units > slot ? (units - slot + slots - 1) / slots * parts : 0;
    struct Unit {
        int b, r;                                          // sample, unit of it
        __device__ __forceinline__ void advance(int by, int per) {
            for (r += by; r >= per; r -= per) ++b;
        }
    };
    Unit next = {0, 0}, now = {0, 0};                      // of the next copy (lane 0); of the sums
    now.advance(slot, per_b);
    next = now;
    int part = 0, issued = 0;
    auto issue = [&]() {
        const uint32_t buf = (uint32_t)issued & 1u;
        mbar_expect_tx(bars + 8 * buf, kKnBufBytes);
        tma_load_4d_once(buf_smem + buf * kKnBufBytes, map_k, bars + 8 * buf, 0, kn.vis_start + next.r * kTok, part * kKnHeads, next.b);
        if (++part == parts) { part = 0; next.advance(slots, per_b); }
        ++issued;
    };
    if (lane == 0)
        while (issued < copies && issued < 2) issue();
    int p = 0;
    bool ok = true;
    float a0 = 0.f, a1 = 0.f, b0 = 0.f, b1 = 0.f;
    int c = 0;
#pragma unroll 1
    for (; c < copies; ++c) {
        const uint32_t buf = (uint32_t)c & 1u;
        ok = __all_sync(0xffffffffu, mbar_wait(bars + 8 * buf, (uint32_t)(c >> 1) & 1u, abort_flag, limit_ns));
        if (!ok) break;
        const uint4* rows = reinterpret_cast<const uint4*>(buf_gen + buf * kKnBufBytes) + lane;
        uint4 x[kKnHeads], y[kKnHeads];                    // (heads past the last are zeros: their squares change nothing)
#pragma unroll
        for (int h = 0; h < kKnHeads; ++h) {
            x[h] = rows[h * 64];
            y[h] = rows[h * 64 + 32];
        }
#pragma unroll
        for (int h = 0; h < kKnHeads; ++h) {
            knorm_sq_acc(x[h], a0, a1);
            knorm_sq_acc(y[h], b0, b1);
        }
        __syncwarp();                                      // the buffer has been read by everyone
        if (lane == 0 && issued < copies) {
            asm volatile("fence.proxy.async.shared::cta;" ::: "memory");
            issue();
        }
        if (++p < parts) continue;
        float s0 = a0 + a1, s1 = b0 + b1;
#pragma unroll
        for (int off = LPR / 2; off > 0; off >>= 1) {
            s0 += __shfl_xor_sync(0xffffffffu, s0, off);
            s1 += __shfl_xor_sync(0xffffffffu, s1, off);
        }
        const int i = now.r * kTok + tk;
        if (sub == 0) {
            float* const out = kn.score + (int64_t)now.b * kn.Nv;
            if (i < kn.Nv) out[i] = sqrtf(s0);
            if (i + kTok / 2 < kn.Nv) out[i + kTok / 2] = sqrtf(s1);
        }
        p = 0;
        a0 = a1 = b0 = b1 = 0.f;
        now.advance(slots, per_b);
    }
    if (!ok && lane == 0)                                  // the copies still in flight land before the CTA's shared memory goes away
        for (int j = c; j < issued; ++j) mbar_drain(bars + 8 * (j & 1), (uint32_t)(j >> 1) & 1u);
}

template <int METRIC, bool KNORM>
__global__ void __cluster_dims__(2, 1, 1) __launch_bounds__(threads(KNORM), 1)
density_sweep_kernel(const __grid_constant__ CUtensorMap map_a, const __grid_constant__ CUtensorMap map_b,
                     const __grid_constant__ CUtensorMap map_k, const __grid_constant__ KernelArgs k) {
    constexpr int kStages = stages(KNORM);
    const SweepArgs& g = k.g;
    extern __shared__ uint8_t smem_raw[];
    const uint32_t raw = smem_u32(smem_raw);
    const uint32_t tiles = (raw + 1023u) & ~1023u;                 // 1024-byte aligned for the 128B swizzle
    uint8_t* gen = smem_raw + (tiles - raw);
    EpiSmem<METRIC>& sm = *reinterpret_cast<EpiSmem<METRIC>*>(gen + kMaxStages * kStageBytes);
    uint64_t* bars = reinterpret_cast<uint64_t*>(gen + kMaxStages * kStageBytes + sizeof(EpiSmem<METRIC>));
    // The leader's full barriers count the bytes of both CTAs and its tempty barriers the epilogue warps of both; empty and
    // tfull are signalled in both CTAs by the leader's commits.
    const uint32_t bar_full = smem_u32(bars), bar_empty = bar_full + 8 * kStages;
    const uint32_t bar_tfull = bar_empty + 8 * kStages, bar_tempty = bar_tfull + 16, bar_drain = bar_tempty + 16;
    const uint32_t bar_kn = bar_drain + 8;
    static_assert((2 * kStages + 5 + 2 * kKnWarps) * 8 + 8 <= 256, "barriers");
    uint32_t* tmem_slot = reinterpret_cast<uint32_t*>(bars + 2 * kStages + 5 + 2 * kKnWarps);
    volatile int* abort_flag = reinterpret_cast<volatile int*>(tmem_slot + 1);
    const uint32_t abort_addr = smem_u32(tmem_slot + 1);
    const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
    constexpr uint32_t kTmemCols = 2 * BN;
    const uint32_t rank = cluster_ctarank();
    const int cluster = blockIdx.x >> 1, n_clusters = gridDim.x >> 1;

    if (threadIdx.x == 0) {
        for (int s = 0; s < kStages; ++s) {
            mbar_init(bar_full + 8 * s, 1);
            mbar_init(bar_empty + 8 * s, 1);
        }
        for (int a = 0; a < 2; ++a) {
            mbar_init(bar_tfull + 8 * a, 1);
            mbar_init(bar_tempty + 8 * a, 2 * kEpiWarps);
        }
        mbar_init(bar_drain, 1);
        for (int a = 0; a < 2 * kKnWarps; ++a) mbar_init(bar_kn + 8 * a, 1);
        *abort_flag = 0;
        asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
        asm volatile("prefetch.tensormap [%0];" ::"l"(reinterpret_cast<uint64_t>(&map_a)) : "memory");
        asm volatile("prefetch.tensormap [%0];" ::"l"(reinterpret_cast<uint64_t>(&map_b)) : "memory");
    }
    if (warp == 1) tmem_alloc_pair(smem_u32(tmem_slot), kTmemCols);
    tc_fence_before();
    __syncthreads();
    cluster_sync_all();                                    // both CTAs' barriers and tensor memory are ready
    tc_fence_after();
    const uint32_t tmem_base = *tmem_slot;

    // The kernels that follow on the stream may be scheduled from here on; they wait for this grid to complete
    // before they touch anything it writes.
    grid_dependency_launch_dependents();

    const int KB = g.D / BK;
    uint32_t issued = 0, issued_parity = 0;                // thread 0, per stage: a load was issued / parity of its phase

    if (warp == 0) {
        // ------------------------------------------------------------------ TMA producer
        // The features are an input of the whole call (never written by the kernel before this one), so
        // the loads need not wait for the preceding grid.
        if (lane == 0) {
            const unsigned long long lim = k.limit_of(kRoleLoad);
            uint32_t stage = 0, phase = 0;
            bool ok = true;
            for (int t = cluster; ok && t < k.n_items; t += n_clusters) {
                const Item it = decode_item(k, t);
                const int row = (it.tp * 2 + (int)rank) * BM;
                const int col = it.tj * BN + it.half * BM + (int)rank * it.halves * kBoxRows;
                const bool one = it.one_operand();
                const uint32_t bytes = 2u * (uint32_t)(kABytes + (one ? 0 : it.halves * (kBBytes / 2)));      // both CTAs
                for (int kb = 0; kb < KB; ++kb) {
                    if (!mbar_wait(bar_empty + 8 * stage, phase ^ 1u, abort_flag, lim)) { ok = false; break; }
                    const uint32_t sa = tiles + stage * kStageBytes;
                    const uint32_t full = cluster_map(bar_full + 8 * stage, 0);
                    if (rank == 0) mbar_expect_tx(bar_full + 8 * stage, bytes);    // rows outside the tensor arrive as zeros
                    tma_load_3d_pair(sa, &map_a, full, kb * BK, row, it.b);
                    if (!one) {
                        tma_load_3d_pair(sa + kABytes, &map_b, full, kb * BK, col, it.b);
                        if (it.halves == 2)
                            tma_load_3d_pair(sa + kABytes + kBBytes / 2, &map_b, full, kb * BK, col + kBoxRows, it.b);
                    }
                    issued |= 1u << stage;
                    issued_parity = (issued_parity & ~(1u << stage)) | (phase << stage);
                    if (++stage == kStages) { stage = 0; phase ^= 1u; }
                }
            }
            // the leader's last commits must have reached this CTA's barriers before it goes away
            for (int s = 0; ok && s < kStages; ++s) {
                ok = mbar_wait(bar_empty + 8 * stage, phase ^ 1u, abort_flag, lim);
                if (++stage == kStages) { stage = 0; phase ^= 1u; }
            }
            if (!ok) raise_abort_pair(abort_addr, rank);
        }
    } else if (warp == 1) {
        // ------------------------------------------------------------------ MMA issuer (leader)
        if (lane == 0 && rank == 0) {
            constexpr uint32_t idesc_full = umma_idesc_bf16(2 * BM, BN), idesc_half = umma_idesc_bf16(2 * BM, BN / 2);
            const unsigned long long lim = k.limit_of(kRoleMma);
            uint32_t stage = 0, phase = 0, acc = 0, acc_phase = 0;
            bool ok = true;
            for (int t = cluster; ok && t < k.n_items; t += n_clusters) {
                if (!mbar_wait(bar_tempty + 8 * acc, acc_phase ^ 1u, abort_flag, lim)) { ok = false; break; }
                tc_fence_after();
                const Item it = decode_item(k, t);
                const uint32_t idesc = it.halves == 2 ? idesc_full : idesc_half;
                const uint32_t b_at = it.one_operand() ? 0u : (uint32_t)kABytes;
                const uint32_t d_tmem = tmem_base + acc * BN;
                for (int kb = 0; kb < KB; ++kb) {
                    if (!mbar_wait(bar_full + 8 * stage, phase, abort_flag, lim)) { ok = false; break; }
                    tc_fence_after();
                    const uint32_t sa = tiles + stage * kStageBytes;
                    const uint64_t da = umma_desc_k128(sa), db = umma_desc_k128(sa + b_at);
#pragma unroll
                    for (int kk = 0; kk < BK / UMMA_K; ++kk)
                        tc_mma_bf16_pair(d_tmem, da + (uint64_t)(2 * kk), db + (uint64_t)(2 * kk), idesc,
                                         (kb > 0 || kk > 0) ? 1u : 0u);
                    tc_commit_pair(bar_empty + 8 * stage);
                    if (++stage == kStages) { stage = 0; phase ^= 1u; }
                }
                if (!ok) break;
                tc_commit_pair(bar_tfull + 8 * acc);
                if (++acc == 2) { acc = 0; acc_phase ^= 1u; }
            }
            if (!ok) raise_abort_pair(abort_addr, rank);
            tc_commit_pair(bar_drain);                     // (waited for below)
        }
    } else if (KNORM && warp >= 2 + kTileThreads / 32) {
        // ------------------------------------------------------------------ K-norm (keys are an input of the whole call, as the features)
        const int w = warp - (2 + kTileThreads / 32), at = kStages * kStageBytes + w * 2 * kKnBufBytes;
        const int slot = (int)blockIdx.x * kKnWarps + w, slots = (int)gridDim.x * kKnWarps;
        if (g.kn.d == 64) side_knorm<8>(g.kn, &map_k, gen + at, tiles + at, bar_kn + 16 * w, slot, slots, abort_flag, k.limit_of(0));
        else side_knorm<16>(g.kn, &map_k, gen + at, tiles + at, bar_kn + 16 * w, slot, slots, abort_flag, k.limit_of(0));
    } else {
        // ------------------------------------------------------------------ epilogue (warps 2 .. 17), auxiliary warps
        const int TI = g.t.TI, nb = g.t.n_blk();
        const int quarter = warp & 3, ew = warp - 2;
        const int h = (ew >> 2) & 1;                               // which 128 columns
        const bool row_role = ew >= kEpiWarps / 2, aux = ew >= kEpiWarps;
        const int lrow = lane >> 2, lcol = 2 * (lane & 3);         // column warps: rows lrow + 8 m, columns lcol + 8 k, + 1
        const unsigned long long lim = k.limit_of(kRoleEpi);
        const f32x2 two2 = pack2(2.f, 2.f), c22 = pack2(g.c2, g.c2);
        uint32_t acc = 0, acc_phase = 0, parity = 0;
        bool ok = true;

        // auxiliary warps: the factors of item t's tokens and whether its halves lie beyond the spatial radius
        auto stage_factors = [&](int t, uint32_t par) {
            const Item it = decode_item(k, t);
            const size_t bo = (size_t)it.b * g.n;
            const int R = 2 * it.tp + (int)rank, C0 = 2 * it.tj + it.half, l = threadIdx.x - 64 - kEpiThreads;
            const int j0 = C0 * BM + l, i0 = R * BM + l;
            float wj[BN / kAuxThreads], aj[BN / kAuxThreads], wi[BM / kAuxThreads], ai[BM / kAuxThreads];
#pragma unroll
            for (int u = 0; u < BN / kAuxThreads; ++u) {
                const int j = j0 + u * kAuxThreads;
                wj[u] = j < g.n ? g.w[bo + j] : 0.f;
                aj[u] = (METRIC == 1 && j < g.n) ? g.a[bo + j] : 0.f;
            }
#pragma unroll
            for (int u = 0; u < BM / kAuxThreads; ++u) {
                const int i = i0 + u * kAuxThreads;
                wi[u] = i < g.n ? -2.f * g.w[bo + i] : 0.f;
                ai[u] = (METRIC == 1 && i < g.n) ? g.a[bo + i] : 0.f;
            }
            if (l < 2) {
                const int C = C0 + l;
                const float4* box = g.bbox + (size_t)it.b * TI;
                sm.far[par][l] = g.bbox && R < TI && C < TI && blocks_outside_radius(box[R], box[C], g.tau2);
            }
#pragma unroll
            for (int u = 0; u < BN / kAuxThreads; ++u) {
                sm.colw[par][l + u * kAuxThreads] = wj[u];
                if (METRIC == 1) sm.cola[par][l + u * kAuxThreads] = aj[u];
            }
#pragma unroll
            for (int u = 0; u < BM / kAuxThreads; ++u) {
                sm.rowm2w[par][l + u * kAuxThreads] = wi[u];
                if (METRIC == 1) sm.rowa[par][l + u * kAuxThreads] = ai[u];
            }
        };
        // auxiliary warps: column side of item t, one column at a time: the sums of the four row quarters in order, the minima as
        // they are
        auto join_columns = [&](int t, uint32_t par) {
            const Item it = decode_item(k, t);
            const int R = 2 * it.tp + (int)rank, C0 = 2 * it.tj + it.half;
            const float(*cs)[BN] = sm.colsum[par];
            const float(*cm)[BN] = sm.colmin[par];
#pragma unroll
            for (int u = 0; u < BN / kAuxThreads; ++u) {
                const int e = (int)threadIdx.x - 64 - kEpiThreads + u * kAuxThreads;
                const int half = e / BM, cc = C0 + half, j = cc * BM + e % BM;
                if (half < it.halves && R <= cc && j < g.n) {
                    const int slot = R == cc ? TI : R;             // (slot R of the own block holds the row side)
                    g.part[((size_t)it.b * g.t.slots() + slot) * g.t.n_pad + j] = ((cs[0][e] + cs[1][e]) + cs[2][e]) + cs[3][e];
                    float4 m = make_float4(cm[0][e], cm[1][e], cm[2][e], cm[3][e]);
                    if (R == cc) {                                 // both sides speak about the same blocks
                        const float4 o = *reinterpret_cast<const float4*>(sm.rowmin[par][e % BM]);
                        m = make_float4(fminf(m.x, o.x), fminf(m.y, o.y), fminf(m.z, o.z), fminf(m.w, o.w));
                    }
                    *reinterpret_cast<float4*>(g.blk_min + ((size_t)it.b * g.t.n_pad + j) * nb + 4 * R) = m;
                }
            }
        };

        grid_dependency_wait();                            // w, a and the bounding boxes come from the preceding kernel
        if (aux && cluster < k.n_items) stage_factors(cluster, 0);
        epi_bar_sync<kTileThreads>();
        for (int t = cluster; t < k.n_items; t += n_clusters, parity ^= 1u) {
            if (aux) {
                // between two meetings: join the previous tile, fetch the next one's factors.  (What the epilogue warps write
                // meanwhile has this tile's parity.)
                if (t != cluster) join_columns(t - n_clusters, parity ^ 1u);
                if (t + n_clusters < k.n_items) stage_factors(t + n_clusters, parity ^ 1u);
                if (epi_bar_or<kTileThreads>(false)) { ok = false; break; }
                if (t + n_clusters >= k.n_items) join_columns(t, parity);
                continue;
            }
            const Item it = decode_item(k, t);
            const int R = 2 * it.tp + (int)rank;           // 128-token block of the CTA's rows ...
            const int C0 = 2 * it.tj + it.half;            // ... and of its first 128 columns
            const int C = C0 + h;                          // this warp's
            const bool work = h < it.halves && R <= C && C < TI;           // (R > C: below the diagonal)
            const int i0 = R * BM + quarter * kBlk;
            const int rb = R * 4 + quarter;                                // the warp's rows as a block of 32
            const bool far = sm.far[parity][h] != 0;       // this warp's pairs all lie beyond the spatial radius
            const float* const colw = sm.colw[parity] + h * BM;
            const float* const cola = sm.cola[parity] + (METRIC == 1 ? h * BM : 0);
            const float* const rowm2w = sm.rowm2w[parity] + quarter * kBlk;
            const float* const rowa = sm.rowa[parity] + (METRIC == 1 ? quarter * kBlk : 0);
            if (ok) ok = mbar_wait(bar_tfull + 8 * acc, acc_phase, abort_flag, lim);
            ok = __all_sync(0xffffffffu, ok);
            if (ok) tc_fence_after();
            const uint32_t taddr = tmem_base + acc * BN + ((uint32_t)(quarter * 32) << 16) + h * BM;
            if (ok && work && row_role) {
                // ---- Eq. 2, row side: exp(-d^2 / d_c^2) of this thread's row, added column by column
                const int i = i0 + lane;
                const f32x2 m2w2 = pack2(rowm2w[lane], rowm2w[lane]);
                const f32x2 ai2 = METRIC == 1 ? pack2(rowa[lane], rowa[lane]) : 0ull;
                float* const blocks = g.gram + (size_t)it.b * g.t.tiles_per_b * kSweepTileFloats;
                float sum = 0.f;
                float4 mins = make_float4(kInf, kInf, kInf, kInf); // of the row over each of the four blocks
#pragma unroll 1
                for (int c = 0; c < kHalfBlks; ++c) {
                    const int cb = C * 4 + c;
                    if (cb < rb) continue;                         // (blocks below the diagonal hold no pair i < j)
                    float v[32];
                    tmem_ld32(taddr + c * kBlk, v);
                    if (!far) {
                        float4* dst = reinterpret_cast<float4*>(blocks + gram_block_offset(rb, cb)) + lane;
#pragma unroll
                        for (int q = 0; q < 8; ++q)
                            __stcs(dst + q * 32, make_float4(v[4 * q], v[4 * q + 1], v[4 * q + 2], v[4 * q + 3]));
                    }
#pragma unroll
                    for (int q = 0; q < 8; ++q) {
                        const float4 cw = *reinterpret_cast<const float4*>(colw + c * kBlk + 4 * q);
                        float4 ca = make_float4(0.f, 0.f, 0.f, 0.f);
                        if (METRIC == 1) ca = *reinterpret_cast<const float4*>(cola + c * kBlk + 4 * q);
#pragma unroll
                        for (int p = 0; p < 2; ++p) {              // two neighbouring columns at a time
                            const int u = 4 * q + 2 * p;
                            const f32x2 x = mul2(pack2(v[u], v[u + 1]), p ? pack2(cw.z, cw.w) : pack2(cw.x, cw.y));
                            const f32x2 base = METRIC == 0 ? two2 : add2(ai2, p ? pack2(ca.z, ca.w) : pack2(ca.x, ca.y));
                            const float2 d = unpack2(fma2(x, m2w2, base));
                            v[u] = d.x;
                            v[u + 1] = d.y;
                        }
                    }
                    const bool edge = cb == rb || (cb + 1) * kBlk > g.n;
                    if (edge) {                                    // pairs that are none (j <= i, tokens past the sample): far apart
#pragma unroll
                        for (int u = 0; u < 32; ++u) {
                            const int j = cb * kBlk + u;
                            v[u] = (j > i && j < g.n) ? v[u] : kInf;
                        }
                    }
                    float mn = min3(v[0], v[1], v[2]), mn2 = min3(v[3], v[4], v[5]);
#pragma unroll
                    for (int u = 6; u < 30; u += 4) {
                        mn = min3(mn, v[u], v[u + 1]);
                        mn2 = min3(mn2, v[u + 2], v[u + 3]);
                    }
                    mn = min3(min3(mn, v[30], v[31]), mn2, kInf);
                    // (rounding can leave a near-duplicate's d^2 below zero, and features without a finite norm give none at all,
                    // which counts as zero in the search and in the one-kernel sweep: rare, so looked for before all are clamped)
                    if (__any_sync(0xffffffffu, !(mn >= 0.f))) {
#pragma unroll
                        for (int u = 0; u < 32; ++u) v[u] = fmaxf(v[u], 0.f);
                        mn = fmaxf(mn, 0.f);
                    }
                    if (far) mn = kInf;                            // (a block beyond the spatial radius has no minima)
                    if (c == 0) mins.x = mn;
                    if (c == 1) mins.y = mn;
                    if (c == 2) mins.z = mn;
                    if (c == 3) mins.w = mn;
#pragma unroll
                    for (int u = 0; u < 32; u += 2) {
                        const float2 arg = unpack2(mul2(pack2(v[u], v[u + 1]), c22));
                        v[u] = ex2_approx(arg.x);
                        v[u + 1] = ex2_approx(arg.y);
                    }
                    if (edge) {
#pragma unroll
                        for (int u = 0; u < 32; ++u) {
                            const int j = cb * kBlk + u;
                            v[u] = (j > i && j < g.n) ? v[u] : 0.f;
                        }
                    }
#pragma unroll
                    for (int u = 0; u < 32; ++u) sum += v[u];
                }
                if (i < g.n) g.part[((size_t)it.b * g.t.slots() + C) * g.t.n_pad + i] = sum;
                // (the block on the diagonal: joined with the column side below)
                if (R == C) *reinterpret_cast<float4*>(sm.rowmin[parity][quarter * kBlk + lane]) = mins;
                else if (i < g.n) *reinterpret_cast<float4*>(g.blk_min + ((size_t)it.b * g.t.n_pad + i) * nb + 4 * C) = mins;
            }
            if (ok && work && !row_role) {
                f32x2 m2w2[4], ai2[4];
#pragma unroll
                for (int m = 0; m < 4; ++m) {
                    m2w2[m] = pack2(rowm2w[lrow + 8 * m], rowm2w[lrow + 8 * m]);
                    ai2[m] = METRIC == 1 ? pack2(rowa[lrow + 8 * m], rowa[lrow + 8 * m]) : 0ull;
                }
#pragma unroll 1
                for (int c = 0; c < kHalfBlks; ++c) {
                    const int cb = C * 4 + c;
                    float csum = 0.f, cmin = kInf;
                    if (cb >= rb) {
                        uint32_t r[32];
                        tmem_ld_16x32_issue(taddr + c * kBlk, r);
                        tmem_ld_16x32_issue(taddr + c * kBlk + (16u << 16), r + 16);
                        tmem_ld_wait32(r);
                        // ---- squared distances
                        float d[32];                               // [m][k][r]: row lrow + 8 m, column 8 k + lcol + r
#pragma unroll
                        for (int q = 0; q < 4; ++q) {
                            const float2 cw = *reinterpret_cast<const float2*>(colw + c * kBlk + 8 * q + lcol);
                            float2 ca = make_float2(0.f, 0.f);
                            if (METRIC == 1) ca = *reinterpret_cast<const float2*>(cola + c * kBlk + 8 * q + lcol);
                            const f32x2 cw2 = pack2(cw.x, cw.y), ca2 = pack2(ca.x, ca.y);
#pragma unroll
                            for (int m = 0; m < 4; ++m) {
                                const int at = (m >> 1) * 16 + q * 4 + (m & 1) * 2;
                                const f32x2 x = mul2(pack2(__uint_as_float(r[at]), __uint_as_float(r[at + 1])), cw2);
                                const f32x2 base = METRIC == 0 ? two2 : add2(ai2[m], ca2);
                                const float2 o = unpack2(fma2(x, m2w2[m], base));
                                d[m * 8 + q * 2] = o.x;
                                d[m * 8 + q * 2 + 1] = o.y;
                            }
                        }
                        const bool edge = cb == rb || (cb + 1) * kBlk > g.n;
                        if (edge) {                                // pairs that are none lie infinitely far apart
#pragma unroll
                            for (int u = 0; u < 32; ++u) {
                                const int i = i0 + lrow + 8 * (u >> 3), j = cb * kBlk + 8 * ((u >> 1) & 3) + lcol + (u & 1);
                                d[u] = (j > i && j < g.n) ? d[u] : kInf;
                            }
                        }
                        // ---- block minima (none where the block lies beyond the spatial radius); clamping as in the row warps
                        float cm[8];
#pragma unroll
                        for (int q = 0; q < 8; ++q) cm[q] = min3(min2(d[q], d[8 + q]), d[16 + q], d[24 + q]);
                        cmin = reduce_columns<true>(cm, lane);
                        if (__any_sync(0xffffffffu, !(cmin >= 0.f))) {
#pragma unroll
                            for (int u = 0; u < 32; ++u) d[u] = fmaxf(d[u], 0.f);
                            cmin = fmaxf(cmin, 0.f);
                        }
                        if (far) cmin = kInf;
                        // ---- Eq. 2, column side: the sum of 32 rows as a tree over the bits of the row, highest first
#pragma unroll
                        for (int u = 0; u < 32; u += 2) {
                            const float2 x = unpack2(mul2(pack2(d[u], d[u + 1]), c22));
                            d[u] = ex2_approx(x.x);
                            d[u + 1] = ex2_approx(x.y);
                        }
                        if (edge) {
#pragma unroll
                            for (int u = 0; u < 32; ++u) {
                                const int i = i0 + lrow + 8 * (u >> 3), j = cb * kBlk + 8 * ((u >> 1) & 3) + lcol + (u & 1);
                                d[u] = (j > i && j < g.n) ? d[u] : 0.f;
                            }
                        }
                        float cs[8];
#pragma unroll
                        for (int q = 0; q < 8; q += 2) {
                            const f32x2 even = add2(pack2(d[q], d[q + 1]), pack2(d[16 + q], d[17 + q]));
                            const f32x2 odd = add2(pack2(d[8 + q], d[9 + q]), pack2(d[24 + q], d[25 + q]));
                            const float2 o = unpack2(add2(even, odd));
                            cs[q] = o.x;
                            cs[q + 1] = o.y;
                        }
                        csum = reduce_columns<false>(cs, lane);
                    }
                    const int at = h * BM + c * kBlk + column_of(lane);
                    sm.colsum[parity][quarter][at] = csum;
                    sm.colmin[parity][quarter][at] = cmin;
                }
            }
            // this warp has read all it needs from the accumulator
            if (ok) {
                tc_fence_before();
                __syncwarp();
                if (lane == 0) mbar_arrive_cluster(cluster_map(bar_tempty + 8 * acc, 0));
            }
            if (epi_bar_or<kTileThreads>(!ok)) { ok = false; break; }
            if (++acc == 2) { acc = 0; acc_phase ^= 1u; }
        }
        if (!ok && lane == 0) raise_abort_pair(abort_addr, rank);
    }

    __syncthreads();
    // Another role may have given up behind the last MMA: operands and tensor memory stay until all of them have completed.
    // (Otherwise they have; the wait costs nothing.)
    if (threadIdx.x == 32) mbar_drain(bar_drain, 0);
    if (threadIdx.x == 0 && *abort_flag) {
        // Some role gave up, so loads issued here may never have been consumed: give the copies still in flight into this
        // CTA's shared memory time to land before the CTA goes away.  (The other CTA's land on the leader's barriers.)
        if (rank == 0) {
            for (int s = 0; s < kStages; ++s)
                if (issued >> s & 1u) mbar_drain(bar_full + 8 * s, issued_parity >> s & 1u);
        } else if (issued) {
            const unsigned long long t0 = global_ns();
            while (global_ns() - t0 < kDrainLimitNs) {}
        }
        grid_dependency_wait();                            // (the kernel in front clears the word)
        atomicMax(g.status, VITCOP_ERR_TIMEOUT);
    }
    tc_fence_before();
    __syncthreads();
    cluster_sync_all();                                    // neither CTA leaves while the other may reach into it
    if (warp == 1) {
        tc_fence_after();
        tmem_dealloc_pair(tmem_base, kTmemCols);
    }
}

}  // namespace

// In microseconds.  The sweep runs at 0.9 PFLOP/s or more and has room for 2.6 MB of keys in each (four warps of every SM, 5 us
// slower by them and the missing stage); the stand-alone kernel reads 6.2 MB, the first 4 + n / 600 of them beside
// vic_finalize_kernel.  So worth it where that leaves 8 to be gained.  Whole calls without and with, 32 heads of 128: 8 x 2880 tokens
// 204 -> 193, 4 x 4608 222 -> 212, 16 x 1152 132.6 -> 128.3, 20 x 1500 207 -> 193; not for 2 x 16384 x 4 heads (868 / 896), whose keys
// all fit beside vic_finalize_kernel.
// And where the keys of all samples have room, which saves the kernel and its wait: from 8 MB of keys, where a tenth
// of a microsecond for each MB (saved) exceeds a twentieth of the sweep (slower by its side warps), up to 8192 tokens.  Without and with: 12 x 1779 x 32 heads of 128 189 / 183, 8 x 1920 x
// 768 features, 32 of 64 105 / 97, 3 x 2845 x 16 of 128 119 / 113, 4 x 2473 x 16 of 64 103 / 99, 3 x 4675 x 16 of 128 168 / 162.  Fewer keys
// are hidden beside vic_finalize_kernel, and longer samples hide more (4 x 3393 x 4 of 64 1.8 % slower, above 8192 tokens 1 to 4 %).
// Below some 760 features the sweep takes as long as its epilogue does, and with the Euclidean metric the side warps cost it a little more: by the
// features alone, 14 of 167 problems were 1 to 4 % slower with all (5 x 7252 x 128 features, 4 of 128 294 / 306; 6 x 4092 x 512, 8 of 128 153 /
// 159).  So the line, of 260 problems, leaves 120, 2.5 % faster in the mean, one of them slower (1.7 %).
int sweep_knorm_samples(const KnormJob& job, int samples, int n, int D, int metric) {
    if (!job.K || job.B <= 0 || job.H <= 0 || job.Nv <= 0 || (job.d != 64 && job.d != 128)) return 0;
    const double mb = 2e-6 * job.H * job.d * job.Nv, sweep = 1e-9 / 0.9 * samples * n * (double)n * D;
    const double fits = 2.6 * sweep / mb, hidden = 4.0 + n / 600.0, all_mb = mb * job.B;
    const int s = fits < job.B ? (int)fits : job.B;
    const double lasts = D < 760 ? sweep / D * 760 : sweep;
    if (s == job.B && n <= 8192 && all_mb >= 8.0 && 0.1 * all_mb > (metric == 1 ? 0.06 : 0.05) * lasts) return s;
    auto left = [&](int b) { return b * mb / 6.2 > hidden ? b * mb / 6.2 - hidden : 0.0; };
    return left(job.B) - left(job.B - s) >= 8.0 ? s : 0;
}

int launch_density_sweep(const void* feat, const SweepArgs& args, int metric, cudaStream_t stream, bool pdl) {
    KernelArgs k;
    k.g = args;
    k.wait_ns = gram_wait_limit_ns();
    k.expire_roles = pair_expire_roles();
    const long long total = (long long)args.B * args.t.tiles_per_b;
    if (total <= 0) return VITCOP_OK;
    if (total >= 1 << 22) return VITCOP_ERR_UNSUPPORTED;   // (group sizes keep it far below; decode_item's estimates hold to there)
    const long long pairs = gram_num_sms() / 2 > 0 ? gram_num_sms() / 2 : 1;
    const long long last = total % pairs, cut = 2 * last <= pairs ? last : 0;
    k.n_full = (int)(total - cut);
    k.n_items = (int)(total + cut);
    k.inv_tiles = 1.f / (float)args.t.tiles_per_b;
    CUtensorMap ma, mb, mk = {};
    const bool kn = k.g.kn.K != nullptr;
    if (!make_rowmajor_bf16_map(&ma, feat, args.B, args.n, args.D, BM) ||
        !make_rowmajor_bf16_map(&mb, feat, args.B, args.n, args.D, kBoxRows))
        return VITCOP_ERR_CUDA;
    if (kn && !make_keys_map(&mk, k.g.kn.K, k.g.kn.B, k.g.kn.H, k.g.kn.N, k.g.kn.d, 512 / k.g.kn.d, kKnHeads)) return VITCOP_ERR_CUDA;
    const int smem = metric == 1 ? smem_bytes<1>() : smem_bytes<0>();
    auto kern = metric == 1 ? (kn ? density_sweep_kernel<1, true> : density_sweep_kernel<1, false>)
                            : (kn ? density_sweep_kernel<0, true> : density_sweep_kernel<0, false>);
    static DoneOnDevice attr_done[2][2];
    const int arc = allow_dynamic_smem(kern, smem, attr_done[metric == 1][kn]);
    if (arc != VITCOP_OK) return arc;
    cudaLaunchConfig_t cfg = {};
    cfg.gridDim = dim3((unsigned)(2 * (k.n_items < pairs ? k.n_items : pairs)));
    cfg.blockDim = dim3(threads(kn));
    cfg.dynamicSmemBytes = smem;
    cfg.stream = stream;
    cudaLaunchAttribute attr[1];
    attr[0].id = cudaLaunchAttributeProgrammaticStreamSerialization;
    attr[0].val.programmaticStreamSerializationAllowed = 1;
    cfg.attrs = attr;
    cfg.numAttrs = pdl_allowed(pdl) ? 1 : 0;
    KernelTimeScope timed("density_sweep_kernel", stream);
    return record_cuda(cudaLaunchKernelEx(&cfg, kern, ma, mb, mk, k));
}

}  // namespace vitcop
