// The K-norm of Eq. 4 at the source of K: the key projection K^(h) = W_k^(h) t for all heads as one bf16 GEMM on the
// tensor cores (tcgen05, fp32 accumulators in tensor memory, operands staged by TMA), with rotary position embedding,
// the bf16 rounding of K and the sum of squares of every token's K vectors in the epilogue.  The separate read of K
// that a stand-alone K-norm costs (the largest byte term of a pruning step) disappears.
//
//   A = hidden [B * N, Dh] (rows = tokens), B = W_k [H * d, Dh] (rows = output features, as a linear layer stores its
//   weight): both K-major, so D = A * B^T needs no transposition.  Output tile 256 tokens x 256 features, or 128 x 256.
//
// Bound by the tensor cores at the clock that the power limit leaves.  Persistent clusters of two CTAs, one CTA per SM, each
// cluster on one tile at a time (tcgen05 cta_group::2): a CTA stages its 128 token rows and its half of the weight rows, 32 KB
// per k-block where two CTAs working apart would each stage 48 KB, so six k-blocks fit and a third of the operand traffic from
// the L2 goes (16 x 640 tokens x 4096 -> 4096 back to back, rotary on: 304 us with CTAs working apart, 275 us so; cuBLAS in a
// sustained loop: 253).  CTAs working apart, on 128 x 256 tiles, where that is the shorter way (the rule is in
// launch_kproj_knorm).
// Warp-specialised like the Gram sweep: warp 0 loads, one thread of the leader's warp 1 issues the MMAs into one of two
// accumulators, 8 epilogue warps of each CTA drain the other: a thread owns one token row (its TMEM lane), the two warps of a lane
// quarter share the row's 256 columns.  Per 32-column chunk a thread rounds the values to bf16 (round to nearest even), stores
// them (64 contiguous bytes of K[b, h, t, :]) and adds their squares -- of the ROUNDED values, i.e. Eq. 4 of the K cache as
// written -- to the row's fp32 partial sum.  With rotary embedding the chunks holding the two halves of a head are taken together
// and turned first.  Partial sums go to one slot per 128 columns and are added by a second, tiny kernel in slot order (the same
// bits on every run and with either tile).
// When the last round of tiles would occupy at most half of the clusters, its tiles are cut into two of 128 features each
// (the MMA keeps its rate at N = 128 with two CTAs), so that the round takes half as long
// (2 x 16512 tokens x 3584 -> 512: 3.5 rounds instead of 4; 121 us before, 117 now).
// Every wait is bounded; on expiry all CTAs of the cluster leave in order and the call reports VITCOP_ERR_TIMEOUT.
#include "async_copy.cuh"
#include "gram.cuh"
#include "tcgen05.cuh"

namespace vitcop {
namespace {

constexpr int BM = 128, BN = 256;                 // rows of one CTA, columns of the cluster's tile
constexpr int kABytes = BM * BK * 2;
__host__ __device__ constexpr int stages(int ctas) { return ctas == 2 ? 6 : 4; }      // (192 KB either way)
__host__ __device__ constexpr int stage_bytes(int ctas) { return kABytes + BN / ctas * BK * 2; }
constexpr int kEpiWarps = 8, kEpiThreads = kEpiWarps * 32, kThreads = 64 + kEpiThreads;
constexpr int kSmemBytes = 1024 + stages(2) * stage_bytes(2) + 256;
static_assert(stages(1) * stage_bytes(1) == stages(2) * stage_bytes(2), "shared memory of either form");

struct KprojArgs {
    int B, N, Dh, H, d;
    int M, NO;                      // rows of A (B * N), output features (H * d)
    int TI, TJ;                     // tiles of 128 rows per CTA of a cluster, of 256 columns
    int n_full;                     // tiles taken whole; the others are cut into two column halves
    uint16_t* K_out;                // bf16 [B, H, N, d]
    float* part;                    // [2 TJ, M] sum of squares of a token's values inside 128 columns
    const float* cos_tab;           // [n_pos, d / 2] or null (no rotation)
    const float* sin_tab;
    const int32_t* position;        // [B, N] or null (token index)
    int n_pos;
    int* status;
    int reports;                    // every CTA reports (internal.cuh) to the kernel behind this one, which sets the status word
    unsigned long long wait_ns;
    int expire_roles;               // roles whose waits give up at once: 1 load warp, 2 MMA warp, 4 epilogue warps
    __device__ __forceinline__ unsigned long long limit_of(int role) const { return (expire_roles & role) ? 0ull : wait_ns; }
};

__device__ __forceinline__ uint32_t pack_bf16_rne(float lo, float hi) {
    uint32_t r;
    asm("cvt.rn.bf16x2.f32 %0, %1, %2;" : "=r"(r) : "f"(hi), "f"(lo));
    return r;
}

// Rounds 32 values to bf16, stores them to `dst` (64 bytes, 16-byte aligned) and returns the sum of the squares of the
// rounded values, two running sums side by side.
__device__ __forceinline__ float round_store_sumsq(const float (&v)[32], uint16_t* dst, bool write) {
    uint32_t w[16];
    float s0 = 0.f, s1 = 0.f;
#pragma unroll
    for (int u = 0; u < 16; ++u) {
        w[u] = pack_bf16_rne(v[2 * u], v[2 * u + 1]);
        const float a = bf16lo(w[u]), b = bf16hi(w[u]);
        s0 = fmaf(a, a, s0);
        s1 = fmaf(b, b, s1);
    }
    if (write) {
        uint4* o = reinterpret_cast<uint4*>(dst);
#pragma unroll
        for (int q = 0; q < 4; ++q) o[q] = make_uint4(w[4 * q], w[4 * q + 1], w[4 * q + 2], w[4 * q + 3]);
    }
    return s0 + s1;
}

// Work item t of a cluster: row tile, first column, 128-column halves.
struct KprojItem {
    int ti, col0, halves;
};
__device__ __forceinline__ KprojItem decode_item(const KprojArgs& k, int t) {
    const int x = t - k.n_full;
    const int tile = x < 0 ? t : k.n_full + (x >> 1);
    KprojItem it;
    it.ti = tile / k.TJ;
    it.col0 = (tile - it.ti * k.TJ) * BN + (x < 0 ? 0 : (x & 1) * (BN / 2));
    it.halves = x < 0 ? 2 : 1;
    return it;
}

// CTAS: CTAs of a cluster, 2 or 1 (one form of the tcgen05 instructions per kernel).
template <bool ROPE, int CTAS>
__global__ void __launch_bounds__(kThreads, 1)
kproj_kernel(const __grid_constant__ CUtensorMap map_a, const __grid_constant__ CUtensorMap map_b,
             const __grid_constant__ CUtensorMap map_half, const KprojArgs k, const int n_items) {
    constexpr bool kPair = CTAS == 2;
    constexpr int kStages = stages(CTAS), kStageBytes = stage_bytes(CTAS);
    extern __shared__ uint8_t smem_raw[];
    const uint32_t raw = smem_u32(smem_raw);
    const uint32_t tiles = (raw + 1023u) & ~1023u;
    uint8_t* gen = smem_raw + (tiles - raw);
    uint64_t* bars = reinterpret_cast<uint64_t*>(gen + kStages * kStageBytes);
    // The leader's full barriers count the bytes of both CTAs and its tempty barriers the epilogue warps of both; empty and
    // tfull are signalled in both CTAs by the leader's commits.
    const uint32_t bar_full = smem_u32(bars), bar_empty = bar_full + 8 * kStages;
    const uint32_t bar_tfull = bar_empty + 8 * kStages, bar_tempty = bar_tfull + 16, bar_drain = bar_tempty + 16;
    uint32_t* tmem_slot = reinterpret_cast<uint32_t*>(bars + 2 * kStages + 5);
    volatile int* abort_flag = reinterpret_cast<volatile int*>(tmem_slot + 1);
    const uint32_t abort_addr = smem_u32(tmem_slot + 1);
    const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
    constexpr uint32_t kTmemCols = 2 * BN;
    const uint32_t rank = kPair ? cluster_ctarank() : 0u;
    const int cluster = blockIdx.x / CTAS, n_clusters = gridDim.x / CTAS;

    if (threadIdx.x == 0) {
        for (int s = 0; s < kStages; ++s) {
            mbar_init(bar_full + 8 * s, 1);
            mbar_init(bar_empty + 8 * s, 1);
        }
        for (int a = 0; a < 2; ++a) {
            mbar_init(bar_tfull + 8 * a, 1);
            mbar_init(bar_tempty + 8 * a, CTAS * kEpiWarps);
        }
        mbar_init(bar_drain, 1);
        *abort_flag = 0;
        asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
        asm volatile("prefetch.tensormap [%0];" ::"l"(reinterpret_cast<uint64_t>(&map_a)) : "memory");
        asm volatile("prefetch.tensormap [%0];" ::"l"(reinterpret_cast<uint64_t>(&map_b)) : "memory");
    }
    if (warp == 1) {
        if constexpr (kPair) tmem_alloc_pair(smem_u32(tmem_slot), kTmemCols);
        else tmem_alloc(smem_u32(tmem_slot), kTmemCols);
    }
    tc_fence_before();
    __syncthreads();
    if constexpr (kPair) cluster_sync_all();               // both CTAs' barriers and tensor memory are ready
    tc_fence_after();
    const uint32_t tmem_base = *tmem_slot;

    const int KB = k.Dh / BK;
    uint32_t issued = 0, issued_parity = 0;                // thread 0, per stage: a load was issued / parity of its phase

    // Everything this kernel reads may come from the kernel before it on the stream.
    grid_dependency_wait();

    if (warp == 0) {
        if (lane == 0) {
            const unsigned long long lim = k.limit_of(1);
            uint32_t stage = 0, phase = 0;
            bool ok = true;
            for (int t = cluster; ok && t < n_items; t += n_clusters) {
                const KprojItem it = decode_item(k, t);
                const int row = (it.ti * CTAS + (int)rank) * BM;
                const int cols = it.halves * (BN / 2 / CTAS), col = it.col0 + (int)rank * cols;       // weight rows that this CTA stages
                const CUtensorMap* const mb = it.halves == 2 ? &map_b : &map_half;         // (one load whatever their number)
                const uint32_t bytes = (uint32_t)(CTAS * (kABytes + cols * BK * 2));       // of all CTAs
                for (int kb = 0; kb < KB; ++kb) {
                    if (!mbar_wait(bar_empty + 8 * stage, phase ^ 1u, abort_flag, lim)) { ok = false; break; }
                    const uint32_t sa = tiles + stage * kStageBytes;
                    if (rank == 0) mbar_expect_tx(bar_full + 8 * stage, bytes);    // rows outside the tensors arrive as zeros
                    if constexpr (kPair) {
                        const uint32_t full = cluster_map(bar_full + 8 * stage, 0);
                        tma_load_3d_pair(sa, &map_a, full, kb * BK, row, 0);
                        tma_load_3d_pair(sa + kABytes, mb, full, kb * BK, col, 0);
                    } else {
                        tma_load_3d(sa, &map_a, bar_full + 8 * stage, kb * BK, row, 0);
                        tma_load_3d(sa + kABytes, mb, bar_full + 8 * stage, kb * BK, col, 0);
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
            if (kPair && !ok) raise_abort_pair(abort_addr, rank);
        }
    } else if (warp == 1) {
        if (lane == 0 && rank == 0) {
            constexpr uint32_t idesc_full = umma_idesc_bf16(CTAS * BM, BN), idesc_half = umma_idesc_bf16(CTAS * BM, BN / 2);
            const unsigned long long lim = k.limit_of(2);
            auto commit = [](uint32_t bar) {
                if constexpr (kPair) tc_commit_pair(bar);
                else tc_commit(bar);
            };
            uint32_t stage = 0, phase = 0, acc = 0, acc_phase = 0;
            bool ok = true;
            for (int t = cluster; ok && t < n_items; t += n_clusters) {
                if (!mbar_wait(bar_tempty + 8 * acc, acc_phase ^ 1u, abort_flag, lim)) { ok = false; break; }
                tc_fence_after();
                const uint32_t idesc = decode_item(k, t).halves == 2 ? idesc_full : idesc_half;
                const uint32_t d_tmem = tmem_base + acc * BN;
                for (int kb = 0; kb < KB; ++kb) {
                    if (!mbar_wait(bar_full + 8 * stage, phase, abort_flag, lim)) { ok = false; break; }
                    tc_fence_after();
                    const uint32_t sa = tiles + stage * kStageBytes;
                    const uint64_t da = umma_desc_k128(sa), db = umma_desc_k128(sa + kABytes);
#pragma unroll
                    for (int kk = 0; kk < BK / UMMA_K; ++kk) {
                        const uint32_t add = (kb > 0 || kk > 0) ? 1u : 0u;
                        if constexpr (kPair) tc_mma_bf16_pair(d_tmem, da + (uint64_t)(2 * kk), db + (uint64_t)(2 * kk), idesc, add);
                        else tc_mma_bf16(d_tmem, da + (uint64_t)(2 * kk), db + (uint64_t)(2 * kk), idesc, add);
                    }
                    commit(bar_empty + 8 * stage);
                    if (++stage == kStages) { stage = 0; phase ^= 1u; }
                }
                if (!ok) break;
                commit(bar_tfull + 8 * acc);
                if (++acc == 2) { acc = 0; acc_phase ^= 1u; }
            }
            if (kPair && !ok) raise_abort_pair(abort_addr, rank);
            commit(bar_drain);                     // (waited for below)
        }
    } else {
        // ------------------------------------------------------------------ epilogue
        const int quarter = warp & 3, slice = (warp - 2) >> 2;     // TMEM lane quarter; which half of the columns
        const int rl = quarter * 32 + lane;
        const int half32 = k.d / 64;                               // chunks in half a head (rotation only)
        uint32_t acc = 0, acc_phase = 0;
        bool ok = true;
        for (int t = cluster; ok && t < n_items; t += n_clusters) {
            const KprojItem it = decode_item(k, t);
            const int m = (it.ti * CTAS + (int)rank) * BM + rl;       // token row of this thread
            const bool row_valid = m < k.M;
            const int b = row_valid ? m / k.N : 0, tok = row_valid ? m - b * k.N : 0;
            ok = mbar_wait(bar_tfull + 8 * acc, acc_phase, abort_flag, k.limit_of(4));
            ok = __all_sync(0xffffffffu, ok);
            if (!ok) break;
            tc_fence_after();
            if (slice < it.halves) {                               // (a column half has work for one slice only)
                float ssq = 0.f;
                const uint32_t taddr = tmem_base + acc * BN + ((uint32_t)(quarter * 32) << 16);
                auto dst_of = [&](int chunk) -> uint16_t* {        // K[b, head, tok, e0 ..] of a 32-column chunk
                    const int col = it.col0 + chunk * 32;
                    const int head = col / k.d, e0 = col - head * k.d;
                    return k.K_out + (((size_t)b * k.H + head) * k.N + tok) * k.d + e0;
                };
                if (!ROPE) {
#pragma unroll 1
                    for (int c = 0; c < 4; ++c) {
                        const int chunk = slice * 4 + c;
                        float v[32];
                        tmem_ld32(taddr + chunk * 32, v);
                        const bool write = row_valid && it.col0 + chunk * 32 < k.NO;
                        ssq += round_store_sumsq(v, dst_of(chunk), write);
                    }
                } else {
                    // pairs of chunks that hold columns e and e + d / 2 of one head: two per slice
                    const int p = row_valid ? (k.position ? k.position[(size_t)b * k.N + tok] : tok) : 0;
                    const int pos = min(max(p, 0), k.n_pos - 1);
#pragma unroll 1
                    for (int c = 0; c < 2; ++c) {
                        const int q = slice * 2 + c;                               // pair number inside the tile
                        const int lo = (q / half32) * 2 * half32 + q % half32, hi = lo + half32;
                        float x[32], y[32];
                        tmem_ld32(taddr + lo * 32, x);
                        tmem_ld32(taddr + hi * 32, y);
                        const int e0 = (it.col0 + lo * 32) % k.d;                  // first of the 32 rotation angles
                        const float4* ct = reinterpret_cast<const float4*>(k.cos_tab + (size_t)pos * (k.d / 2) + e0);
                        const float4* st = reinterpret_cast<const float4*>(k.sin_tab + (size_t)pos * (k.d / 2) + e0);
#pragma unroll
                        for (int u4 = 0; u4 < 8; ++u4) {
                            const float4 cc = __ldg(ct + u4), ss = __ldg(st + u4);
                            const float cv[4] = {cc.x, cc.y, cc.z, cc.w}, sv[4] = {ss.x, ss.y, ss.z, ss.w};
#pragma unroll
                            for (int r = 0; r < 4; ++r) {
                                const float a = x[4 * u4 + r], bb = y[4 * u4 + r];
                                x[4 * u4 + r] = fmaf(a, cv[r], -(bb * sv[r]));
                                y[4 * u4 + r] = fmaf(bb, cv[r], a * sv[r]);
                            }
                        }
                        const bool write = row_valid && it.col0 + hi * 32 < k.NO;
                        ssq += round_store_sumsq(x, dst_of(lo), write);
                        ssq += round_store_sumsq(y, dst_of(hi), write);
                    }
                }
                if (row_valid) k.part[(size_t)(it.col0 / (BN / 2) + slice) * k.M + m] = ssq;
            }
            tc_fence_before();
            __syncwarp();
            if (lane == 0) {
                if constexpr (kPair) mbar_arrive_cluster(cluster_map(bar_tempty + 8 * acc, 0));
                else mbar_arrive(bar_tempty + 8 * acc);
            }
            if (++acc == 2) { acc = 0; acc_phase ^= 1u; }
        }
        if (kPair && !ok && lane == 0) raise_abort_pair(abort_addr, rank);
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
        if (!k.reports) atomicMax(k.status, VITCOP_ERR_TIMEOUT);
    }
    if (threadIdx.x == 0 && k.reports) report_gave_up(k.status, *abort_flag != 0);
    tc_fence_before();
    __syncthreads();
    if constexpr (kPair) cluster_sync_all();               // neither CTA leaves while the other may reach into it
    if (warp == 1) {
        tc_fence_after();
        if constexpr (kPair) tmem_dealloc_pair(tmem_base, kTmemCols);
        else tmem_dealloc(tmem_base, kTmemCols);
    }
    grid_dependency_launch_dependents();
}

// score[b, i] = sqrt( sum over the slots, in order, of the partial sums of token vis_start + i ).
__global__ void kproj_score_kernel(const float* __restrict__ part, int M, int slots, int N, int vis_start, int Nv,
                                   float* __restrict__ score, int* __restrict__ status, int reports) {
    grid_dependency_launch_dependents();
    grid_dependency_wait();
    if (reports > 0 && blockIdx.x == 0 && blockIdx.y == 0 && threadIdx.x < 32) {
        const bool gave_up = any_gave_up(status, reports);
        if (threadIdx.x == 0) *status = gave_up ? VITCOP_ERR_TIMEOUT : VITCOP_OK;
    }
    const int i = blockIdx.x * blockDim.x + threadIdx.x, b = blockIdx.y;
    if (i >= Nv) return;
    const size_t m = (size_t)b * N + vis_start + i;
    float s = 0.f;
#pragma unroll 8
    for (int q = 0; q < slots; ++q) s += part[(size_t)q * M + m];
    score[(size_t)b * Nv + i] = sqrtf(s);
}

// Tiles of 128 rows per CTA x 256 columns on clusters of `ctas` CTAs, those of a last round that would occupy at most half of the
// clusters cut in two.
struct TileSplit {
    int TI, units;                  // row tiles; clusters at work together
    long long total, cut;
    double rounds;                  // until the last is done, a cut tile counting half
};
TileSplit split_tiles(int M, int TJ, int ctas, bool may_cut) {
    TileSplit s;
    s.TI = (int)(((long long)M + ctas * BM - 1) / (ctas * BM));
    s.units = gram_num_sms() / ctas > 0 ? gram_num_sms() / ctas : 1;
    s.total = (long long)s.TI * TJ;
    const long long last = s.total % s.units;
    s.cut = 2 * last <= s.units && may_cut ? last : 0;
    s.rounds = (double)(s.total / s.units) + (last == 0 ? 0.0 : s.cut ? 0.5 : 1.0);
    return s;
}

}  // namespace

size_t kproj_workspace_bytes(int B, int N, int H, int d) {
    const size_t TJ = ((size_t)H * d + BN - 1) / BN;
    return kStatusBytes + align_up(2 * TJ * (size_t)B * N * sizeof(float), 256);
}

int launch_kproj_knorm(const void* hidden, const void* W, int B, int N, int Dh, int H, int d, const float* cos_tab,
                       const float* sin_tab, const int32_t* position, int n_pos, void* K_out, int vis_start, int Nv,
                       float* score, void* workspace, cudaStream_t stream) {
    KprojArgs k = {};
    k.B = B; k.N = N; k.Dh = Dh; k.H = H; k.d = d;
    k.M = B * N; k.NO = H * d;
    k.TJ = (k.NO + BN - 1) / BN;
    k.K_out = static_cast<uint16_t*>(K_out);
    k.part = reinterpret_cast<float*>(static_cast<char*>(workspace) + kStatusBytes);
    k.cos_tab = cos_tab; k.sin_tab = sin_tab; k.position = position; k.n_pos = n_pos;
    k.status = static_cast<int*>(workspace);
    k.wait_ns = gram_wait_limit_ns();
    k.expire_roles = pair_expire_roles();
    const bool scores = Nv > 0 && score;
    k.reports = scores && gram_num_sms() <= kMaxReports;
    if (!k.reports) {
        const int rc = record_cuda(cudaMemsetAsync(workspace, 0, kStatusBytes, stream));
        if (rc != VITCOP_OK) return rc;
    }
    const bool rope = cos_tab != nullptr;
    // (a rotated head of 256 columns cannot be cut: its halves are turned together)
    const bool may_cut = !(rope && d > BN / 2);
    const TileSplit two = split_tiles(k.M, k.TJ, 2, may_cut), one = split_tiles(k.M, k.TJ, 1, may_cut);
    // CTAs apart take a tenth longer for a full round, but their rounds are finer: 1152 tokens x 4096 -> 4096 are 144 tiles of 128
    // rows, one round, and 80 of 256 rows, one and a half (30.9 and 48.6 us).  Inside one round they are done sooner up to
    // Dh = 4096 (9000 tokens x 3584 -> 512: 28.7 and 30.8 us; 640 x 8192 -> 4096: 53 and 47): pairs start and stop 2 us slower.
    const bool pair = !(one.rounds * 1.1 < two.rounds || (one.rounds == two.rounds && two.rounds <= 1.0 && Dh <= 4096));
    const TileSplit& split = pair ? two : one;
    if (split.total + split.cut > 0x7fffffffLL) return VITCOP_ERR_UNSUPPORTED;
    k.TI = split.TI;
    k.n_full = (int)(split.total - split.cut);
    const int n_items = (int)(split.total + split.cut), units = split.units;
    const int ctas = pair ? 2 : 1;
    CUtensorMap ma, mb, mh;
    if (!make_rowmajor_bf16_map(&ma, hidden, 1, k.M, Dh, BM) || !make_rowmajor_bf16_map(&mb, W, 1, k.NO, Dh, BN / ctas) ||
        !make_rowmajor_bf16_map(&mh, W, 1, k.NO, Dh, BN / 2 / ctas))
        return VITCOP_ERR_CUDA;
    auto kern = pair ? (rope ? kproj_kernel<true, 2> : kproj_kernel<false, 2>) : (rope ? kproj_kernel<true, 1> : kproj_kernel<false, 1>);
    static DoneOnDevice attr_done[2][2];
    const int arc = allow_dynamic_smem(kern, kSmemBytes, attr_done[pair][rope]);
    if (arc != VITCOP_OK) return arc;
    cudaLaunchConfig_t cfg = {};
    cfg.gridDim = dim3((unsigned)(ctas * (n_items < units ? n_items : units)));
    cudaLaunchAttribute shape[2];
    int n_shape = 0;
    if (pdl_allowed(k.reports)) {                          // (a memset is no kernel to overlap with)
        shape[n_shape].id = cudaLaunchAttributeProgrammaticStreamSerialization;
        shape[n_shape++].val.programmaticStreamSerializationAllowed = 1;
    }
    if (pair) {
        shape[n_shape].id = cudaLaunchAttributeClusterDimension;
        shape[n_shape].val.clusterDim.x = (unsigned)ctas;
        shape[n_shape].val.clusterDim.y = shape[n_shape].val.clusterDim.z = 1;
        ++n_shape;
    }
    cfg.attrs = shape;
    cfg.numAttrs = n_shape;
    cfg.blockDim = dim3(kThreads);
    cfg.dynamicSmemBytes = kSmemBytes;
    cfg.stream = stream;
    int rc;
    {
        KernelTimeScope timed("kproj_kernel", stream);
        rc = record_cuda(cudaLaunchKernelEx(&cfg, kern, ma, mb, mh, k, n_items));
    }
    if (rc != VITCOP_OK || !scores) return rc;
    cudaLaunchAttribute attr[1];
    attr[0].id = cudaLaunchAttributeProgrammaticStreamSerialization;
    attr[0].val.programmaticStreamSerializationAllowed = 1;
    cudaLaunchConfig_t c2 = {};
    c2.gridDim = dim3((Nv + 255) / 256, B);
    c2.blockDim = dim3(256);
    c2.stream = stream;
    c2.attrs = attr;
    c2.numAttrs = pdl_allowed(true) ? 1 : 0;
    KernelTimeScope timed("kproj_score_kernel", stream);
    return record_cuda(cudaLaunchKernelEx(&c2, kproj_score_kernel, (const float*)k.part, k.M, 2 * k.TJ, N, vis_start, Nv,
                                          score, k.status, k.reports ? (int)cfg.gridDim.x : 0));
}

}  // namespace vitcop
