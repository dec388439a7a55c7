// Tensor-core work on the Gram matrix of the visual-token features (Algorithm 2, step 1): its diagonal (per-token factors), rows
// of it (similarity), and, for small problems, the whole of Eq. 2 (density) and Eq. 3 (nearest denser neighbour) in one kernel.
// Larger problems take density.cu and nearest.cu for the two equations.
//
// The Gram matrix f_I . f_J^T is taken on the RAW bf16 features (bf16 x bf16 products are exact in fp32) by
// tcgen05.mma with fp32 accumulators in tensor memory; the L2 normalisation enters as fp32 factors in the epilogue.
//
// Symmetry: d_ij = d_ji, so the one-kernel sweep visits only tiles that hold a pair i < j.  Such a pair serves its
// row token i (a per-thread accumulation along the row) and its column token j (a reduction over the 128
// rows of the tile: inside each warp a shuffle butterfly for the sums of Eq. 2 and one redux.sync per column for
// the minima of Eq. 3, then a fixed-order combination of the four warps that share a column range).
//
// One persistent CTA per SM, warp-specialised (the one-kernel sweep has two warps more behind these):
//   warp 0      TMA producer: feature tiles [128 x 64] (128-byte swizzle) into a ring of stages
//   warp 1      one thread issues tcgen05.mma into one of two TMEM accumulators
//   warps 2..   epilogue: warp w reads TMEM lanes 32 * (w % 4) .. + 31 (its rows) and one slice of the columns
// Every wait is bounded; on expiry the CTA raises an abort flag, all roles leave, TMEM is released and
// VITCOP_ERR_TIMEOUT is written to the status word.
#include <cuda.h>

#include <atomic>

#include "async_copy.cuh"
#include "f32x2.cuh"
#include "gram.cuh"
#include "tcgen05.cuh"
#include "knorm.cuh"

namespace vitcop {
namespace {

constexpr int BM = kGramBM;
// Column slices an output tile of gram_tc_kernel is cut into for the epilogue; every slice is served by four warps (one per
// TMEM lane quarter).
constexpr int kEpiSlices = 2;
constexpr int kGemmThreads = 64 + kEpiSlices * 128;

// ------------------------------------------------------------------------------------------------
// tile numbering
// ------------------------------------------------------------------------------------------------
struct KernelArgs {
    GramArgs g;
    GramTiling t;
    long long total_tiles;         // the resident sweep counts its units here
    int extra_units_per_b;         // resident sweep: units of one sample that do not hold a diagonal tile
    int unit_w;                    // resident sweep: column blocks of a unit, 1 or 2
    unsigned long long wait_ns;    // time limit of every bounded wait
    int expire_roles;              // roles whose waits give up at once: 1 load warp, 2 MMA warp, 4 epilogue warps
    int reports;                   // diagonal: every CTA reports (internal.cuh); rho_reduce_kernel sets the status word
    __device__ __forceinline__ unsigned long long limit_of(int role) const {
        return (expire_roles & role) ? 0ull : wait_ns;
    }
};
constexpr int kRoleLoad = 1, kRoleMma = 2, kRoleEpi = 4;

template <bool DIAG>
__device__ __forceinline__ void decode_tile(const KernelArgs& k, long long t, int& b, int& ti, int& tj) {
    b = (int)(t / k.t.tiles_per_b);
    const int r = (int)(t - (long long)b * k.t.tiles_per_b);
    if (DIAG) {
        ti = tj = r;
        return;
    }
    ti = r / k.t.TJ;
    tj = r - ti * k.t.TJ;
}

// ------------------------------------------------------------------------------------------------
// warp butterflies: lane L ends up with the reduction over the 32 lanes of element L of the array
// ------------------------------------------------------------------------------------------------
template <int HALF>
__device__ __forceinline__ void butterfly_stage(float* v, bool up) {
#pragma unroll
    for (int k = 0; k < HALF; ++k) {
        const float keep = up ? v[k + HALF] : v[k];
        const float send = up ? v[k] : v[k + HALF];
        const float recv = __shfl_xor_sync(0xffffffffu, send, HALF);
        v[k] = keep + recv;
    }
}
// Eight columns held by every lane (one row each): afterwards every lane holds the sum over the 32 lanes of column
// lane & 7, added in a fixed order.
__device__ __forceinline__ float warp_column_sums8(float (&v)[8], int lane) {
    butterfly_stage<4>(v, (lane & 4) != 0);
    butterfly_stage<2>(v, (lane & 2) != 0);
    butterfly_stage<1>(v, (lane & 1) != 0);
    float s = v[0];
    s += __shfl_xor_sync(0xffffffffu, s, 8);
    s += __shfl_xor_sync(0xffffffffu, s, 16);
    return s;
}
// ------------------------------------------------------------------------------------------------
// shared memory
// ------------------------------------------------------------------------------------------------
template <int BN>
struct GemmSmem {
    static constexpr int kStages = (BN == 128) ? 6 : 4;
    static constexpr int kABytes = BM * BK * 2;
    static constexpr int kBBytes = BN * BK * 2;
    static constexpr int kStageBytes = kABytes + kBBytes;
    static constexpr int kTileBytes = kStages * kStageBytes;
    // per column of the tile: w, a, rho, x, y; column reduction scratch: 4 x value, 4 x index;
    // row reduction scratch: 3 x value, 3 x index; per row of the tile: w, a, rho, x, y
    static constexpr int kEpiBytes = (5 + 4 + 4) * BN * 4 + (3 + 3 + 5) * BM * 4;
    static constexpr int kBarBytes = 256;
    static constexpr int kTotal = 1024 /*alignment slack*/ + kTileBytes + kEpiBytes + kBarBytes;
};
// The one-kernel sweep's units of 64 columns: the operand memory of GemmSmem<256> in stages of 128 + 64 rows.
struct HalfUnitSmem {
    static constexpr int kStageBytes = (BM + 64) * BK * 2;
    static constexpr int kStages = 8;
    static constexpr int kEpiBytes = (5 + 4 + 4) * 64 * 4 + (3 + 3 + 5) * BM * 4 + 2 * 16 * BM * 4;
    static_assert(kStages * kStageBytes <= GemmSmem<256>::kTileBytes, "stages");
};

constexpr float kInf = __builtin_huge_valf();

// ------------------------------------------------------------------------------------------------
// epilogue of one output tile (called by all epilogue threads of the CTA)
// ------------------------------------------------------------------------------------------------
struct EpiSmem {
    float *colw, *cola, *colrho, *colx, *coly, *colred, *rowred;
    int *colidx, *rowidx;                                       // (colidx: the rows that attain colred, as a mask)
    float *roww, *rowa, *rowrho, *rowx, *rowy;
    float* half;                                                // [2][16][BM], units of 64 columns only
    // Carves the arrays out of GemmSmem<BN>::kEpiBytes bytes at `base`.
    template <int BN>
    __device__ __forceinline__ void carve(uint8_t* base) {
        colw = reinterpret_cast<float*>(base);
        cola = colw + BN;
        colrho = cola + BN;
        colx = colrho + BN;
        coly = colx + BN;
        colred = coly + BN;                                     // [4][BN]
        colidx = reinterpret_cast<int*>(colred + 4 * BN);       // [4][BN]
        rowred = reinterpret_cast<float*>(colidx + 4 * BN);     // [3][BM]
        rowidx = reinterpret_cast<int*>(rowred + 3 * BM);       // [3][BM]
        roww = reinterpret_cast<float*>(rowidx + 3 * BM);
        rowa = roww + BM;
        rowrho = rowa + BM;
        rowx = rowrho + BM;
        rowy = rowx + BM;
        half = rowy + BM;
    }
};
// A token's factor travels from the diagonal tile's CTA to the others as one word, bits + 1 (0: not there yet), so that value
// and flag arrive in one trip.  (Behind a flag per row block, i.e. stores, fence, flag, poll, fence, loads: 3.9 us from the
// accumulator of the diagonal tile to the factors in every other CTA, instead of 2.0.)
__device__ __forceinline__ void publish_factor(uint32_t* p, float f) {
    const uint32_t v = __float_as_uint(f) + 1u;
    asm volatile("st.relaxed.gpu.global.u32 [%0], %1;" ::"l"(p), "r"(v ? v : 0x80000000u) : "memory");     // (a NaN stays one)
}
// Bounded; gives up (sets the abort flag, returns false) when the limit is over or another role has given up.
__device__ __forceinline__ bool wait_factor(const uint32_t* p, float& f, volatile int* abort_flag, unsigned long long limit_ns) {
    auto load = [&]() {
        uint32_t v;
        asm volatile("ld.relaxed.gpu.global.u32 %0, [%1];" : "=r"(v) : "l"(p) : "memory");
        return v;
    };
    uint32_t v = load();
    bool ok = true;
    if (v == 0u) {
        unsigned long long t0;
        asm volatile("mov.u64 %0, %globaltimer;" : "=l"(t0));
        while ((v = load()) == 0u) {
            unsigned long long now;
            asm volatile("mov.u64 %0, %globaltimer;" : "=l"(now));
            if (limit_ns == 0ull || now - t0 > limit_ns || *abort_flag) {
                *abort_flag = 1;
                ok = false;
                break;
            }
        }
    }
    f = __uint_as_float(v - 1u);
    return ok;
}

struct EpiCall {
    int b, ti, tj;                 // sample, row tile, column tile
    uint32_t tmem_tile;            // TMEM address (lane 0) of the tile's first accumulator column
    uint32_t wait_bar, wait_parity;   // mbarrier that completes when the accumulator is ready (0: it already is)
    uint32_t arrive_bar;           // mbarrier to arrive on once this thread has read the accumulator (0: none)
    volatile int* abort_flag;
    unsigned long long limit_ns;   // time limit of the wait for the accumulator
};

// Returns true when the CTA must give up (a bounded wait expired somewhere).
// GW: columns a warp takes from the accumulator at a time: 8 in the one-kernel sweep, a short rolled loop, because every tile is
// visited once and the instruction cache would otherwise miss all the way; 32 for the diagonal and the similarity rows.
template <int BN, int MODE, int METRIC, bool SPATIAL, int NS, int GW = 32>
__device__ __forceinline__ bool epi_tile(const KernelArgs& k, const EpiSmem& sm, const EpiCall& call, bool& ok) {
    static_assert(GW == 8 || GW == 32, "group width");
    constexpr bool SYM = MODE == GRAM_RHO || MODE == GRAM_DELTA;
    constexpr bool DIAG = MODE == GRAM_DIAG;
    constexpr bool HALF = SYM && BN == 64;             // a unit of the one-kernel sweep: half a tile
    constexpr int kEpiThreads = NS * 128;
    constexpr int kSliceCols = BN / NS;
    constexpr int kGroups = kSliceCols / GW;           // column groups per warp, taken one by one in a rolled loop
    const GramArgs& g = k.g;
    float *colw = sm.colw, *cola = sm.cola, *colrho = sm.colrho, *colx = sm.colx, *coly = sm.coly;
    float *colred = sm.colred, *rowred = sm.rowred;
    int *colidx = sm.colidx, *rowidx = sm.rowidx;
    const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
    const int e = threadIdx.x - 64;                    // 0 .. kEpiThreads - 1
    const int quarter = warp & 3;                      // TMEM lane quarter this warp may read
    const int slice = (warp - 2) >> 2;                 // which slice of the tile's columns this warp handles
    const int rl = quarter * 32 + lane;                // tile-local row == TMEM lane
    const int rows_out = g.row_end - g.row0;
    const int b = call.b, ti = call.ti, tj = call.tj;
    const int I0 = g.row0 + ti * BM, J0 = tj * BN;
    const int i = I0 + rl;
    const bool row_valid = SYM ? (i < g.n) : (i < g.row_end);
    const size_t bo = (size_t)b * g.n;

    // ---- per-column and per-row constants.  One item per thread where the tile allows it -- column factors,
    //      column rho and position, row factors, row rho and position -- so that all the global loads of the tile
    //      are in flight together: one round trip to L2 instead of one per group.
    const float* const part_b = g.part + (size_t)b * (HALF ? 5 * k.t.TI : k.t.slots()) * k.t.n_pad;
    auto sum_rho = [&](int x) {
        return HALF ? rho_from_half_partials(part_b, k.t, g.n, x) : rho_from_partials(part_b + x, k.t, x);
    };
    for (int it = e; it < 2 * BN + 2 * BM && !DIAG; it += kEpiThreads) {
        if (it < BN) {
            const int ce = it, j = J0 + ce;
            const bool cv = j < g.n;
            // (L2 loads: another CTA may have written these factors after this SM last cached their line)
            if (MODE == GRAM_RHO) {
                float f = 0.f;
                if (cv) ok = wait_factor(g.ready + bo + j, f, call.abort_flag, call.limit_ns) && ok;
                colw[ce] = METRIC == 0 ? f : cv ? 1.f : 0.f;
                if (METRIC == 1) cola[ce] = f;
            } else {
                colw[ce] = cv ? __ldcg(g.w + bo + j) : 0.f;
                if (METRIC == 1) cola[ce] = cv ? __ldcg(g.a + bo + j) : 0.f;
            }
        } else if (it < 2 * BN) {
            if (MODE == GRAM_DELTA) {
                const int ce = it - BN, j = J0 + ce;
                const bool cv = j < g.n;
                float rj = 0.f;
                float2 pj = make_float2(0.f, 0.f);
                if (cv) {
                    if (SPATIAL) pj = *reinterpret_cast<const float2*>(g.pos + 2 * (bo + j));
                    rj = sum_rho(j);
                    if (ti == (HALF ? tj / 2 : tj)) {          // the diagonal tile of a row block publishes its tokens' rho
                        g.rho_out[bo + j] = rj;
                        if (g.rho_user) g.rho_user[bo + j] = rj;
                    }
                }
                colrho[ce] = rj;
                if (SPATIAL) { colx[ce] = pj.x; coly[ce] = pj.y; }
            }
        } else if (it < 2 * BN + BM) {
            const int r = it - 2 * BN, ir = I0 + r;
            const bool rv = SYM ? (ir < g.n) : (ir < g.row_end);
            if (MODE == GRAM_RHO) {
                float f = 0.f;
                if (rv) ok = wait_factor(g.ready + bo + ir, f, call.abort_flag, call.limit_ns) && ok;
                sm.roww[r] = METRIC == 0 ? f : rv ? 1.f : 0.f;
                if (METRIC == 1) sm.rowa[r] = f;
            } else {
                sm.roww[r] = rv ? __ldcg(g.w + bo + ir) : 0.f;
                if (METRIC == 1) sm.rowa[r] = rv ? __ldcg(g.a + bo + ir) : 0.f;
            }
        } else if (MODE == GRAM_DELTA) {
            const int r = it - 2 * BN - BM, ir = I0 + r;
            float rr = 0.f;
            float2 pr = make_float2(0.f, 0.f);
            if (ir < g.n) {
                if (SPATIAL) pr = *reinterpret_cast<const float2*>(g.pos + 2 * (bo + ir));
                rr = sum_rho(ir);
            }
            sm.rowrho[r] = rr;
            if (SPATIAL) { sm.rowx[r] = pr.x; sm.rowy[r] = pr.y; }
        }
    }
    // every pair of the tile has i < j < n: no masking needed
    const bool full = SYM && (J0 >= I0 + BM) && (J0 + BN <= g.n);

    epi_bar_sync<kEpiThreads>();
    const float w_i = DIAG ? 0.f : sm.roww[rl];
    const float a_i = METRIC == 1 ? (DIAG ? 0.f : sm.rowa[rl]) : 1.f;
    const float m2w_i = -2.f * w_i;
    float rho_i = 0.f, x_i = 0.f, y_i = 0.f;
    if (MODE == GRAM_DELTA) {
        rho_i = sm.rowrho[rl];
        if (SPATIAL) { x_i = sm.rowx[rl]; y_i = sm.rowy[rl]; }
    }
    // the row's constants, twice each, for the paired arithmetic (the epilogues are bound by instruction issue)
    const unsigned long long m2w2 = pack2(m2w_i, m2w_i), ai2 = pack2(a_i, a_i), two2 = pack2(2.f, 2.f);
    const unsigned long long nxi2 = pack2(-x_i, -x_i), nyi2 = pack2(-y_i, -y_i), c22 = pack2(g.c2, g.c2);
    if (ok && call.wait_bar) ok = mbar_wait(call.wait_bar, call.wait_parity, call.abort_flag, call.limit_ns);
    ok = __all_sync(0xffffffffu, ok);

    // GRAM_DELTA: the tile-local columns j of this row's pairs i < j < n
    const int first_c = i + 1 - J0;
    const uint32_t usable_c = row_valid ? (uint32_t)max(min(BN, g.n - J0) - first_c, 0) : 0u;
    float racc = 0.f;                              // GRAM_RHO: row-side sum
    float rbest = kInf;                            // GRAM_DELTA: row-side minimum and its tile-local column
    int rbest_c = -1;
    if (ok) {
        tc_fence_after();
        const uint32_t taddr = call.tmem_tile + ((uint32_t)(quarter * 32) << 16) + slice * kSliceCols;
        uint32_t ld_cur[8], ld_nxt[8];
        if constexpr (GW == 8) {
            tmem_ld8_issue(taddr, ld_cur);
            tmem_ld8_wait(ld_cur);
        }
#pragma unroll 1
        for (int c = 0; c < kGroups; ++c) {
            float v[GW];
            if constexpr (GW == 8) {
                // the next group's accumulators travel while this one is worked on
                if (c + 1 < kGroups) tmem_ld8_issue(taddr + (c + 1) * 8, ld_nxt);
#pragma unroll
                for (int u = 0; u < 8; ++u) v[u] = __uint_as_float(ld_cur[u]);
            } else {
                tmem_ld32(taddr + c * 32, v);
            }
            if (c == kGroups - 1) {
                // this thread has read all it needs from the accumulator
                tc_fence_before();
                if (call.arrive_bar) mbar_arrive(call.arrive_bar);
            }
            const int cl0 = slice * kSliceCols + c * GW;       // tile-local first column of the group
            const float4* cw4 = reinterpret_cast<const float4*>(colw + cl0);
            const float4* ca4 = reinterpret_cast<const float4*>(cola + cl0);
            if constexpr (MODE == GRAM_DIAG) {
                // g_ii sits in column rl of row rl
                if (J0 + cl0 == I0 + (rl & ~(GW - 1)) && row_valid) {
                    // (selected with explicit selp: left to itself the compiler indexes the array in local
                    // memory, a cold round trip on the path every other tile waits for)
                    float gii = 0.f;
                    const int mine = lane & (GW - 1);
#pragma unroll
                    for (int u = 0; u < GW; ++u)
                        asm("{\n\t.reg .pred p;\n\tsetp.eq.s32 p, %2, %3;\n\tselp.f32 %0, %1, %0, p;\n\t}"
                            : "+f"(gii)
                            : "f"(v[u]), "r"(mine), "r"(u));
                    // The squared norm comes from the same tensor-core arithmetic as every g_ij, so the
                    // rounding of the accumulation cancels in s_ij = g_ij / sqrt(g_ii g_jj) where it
                    // matters: near-duplicates (s -> 1, d^2 = 2 - 2 s -> 0); exact duplicates give s = 1.
                    const float wi = METRIC == 0 ? (gii > 0.f ? 1.0f / sqrtf(gii) : 0.f) : 1.f;
                    if (g.ready) publish_factor(g.ready + bo + i, METRIC == 0 ? wi : gii);
                    g.w_out[bo + i] = wi;
                    g.a_out[bo + i] = METRIC == 0 ? 1.f : gii;
                    if (g.best) g.best[bo + i] = ~0ull;
                }
            } else if constexpr (MODE == GRAM_SIM) {
                if (row_valid) {
                    float* o = g.sim_out + ((size_t)b * rows_out + (i - g.row0)) * g.n;
#pragma unroll
                    for (int u = 0; u < GW; ++u) {
                        const int j = J0 + cl0 + u;
                        if (j < g.n) o[j] = METRIC == 0 ? (v[u] * w_i) * colw[cl0 + u] : v[u];
                    }
                }
            } else if constexpr (MODE == GRAM_RHO) {
                // e_ij = exp(-d_ij^2 / d_c^2), Eq. 2
#pragma unroll
                for (int q4 = 0; q4 < GW / 4; ++q4) {
                    const float4 cw = cw4[q4];
                    float4 ca = make_float4(0.f, 0.f, 0.f, 0.f);
                    if (METRIC == 1) ca = ca4[q4];
#pragma unroll
                    for (int h = 0; h < 2; ++h) {              // two neighbouring columns at a time
                        const int u = 4 * q4 + 2 * h;
                        const unsigned long long cw2 = h ? pack2(cw.z, cw.w) : pack2(cw.x, cw.y);
                        const unsigned long long ca2 = h ? pack2(ca.z, ca.w) : pack2(ca.x, ca.y);
                        const unsigned long long x2 = mul2(pack2(v[u], v[u + 1]), cw2);
                        const unsigned long long base2 = METRIC == 0 ? two2 : add2(ai2, ca2);
                        const float2 d2 = unpack2(fma2(x2, m2w2, base2));
                        const float2 arg = unpack2(mul2(pack2(fmaxf(d2.x, 0.f), fmaxf(d2.y, 0.f)), c22));
                        v[u] = ex2_approx(arg.x);
                        v[u + 1] = ex2_approx(arg.y);
                    }
                }
                if (!full) {
#pragma unroll
                    for (int u = 0; u < GW; ++u) {
                        const int j = J0 + cl0 + u;
                        v[u] = (j > i && j < g.n && row_valid) ? v[u] : 0.f;
                    }
                }
                if (HALF && (slice & 1)) {             // the second half of a 32-column sum: added by the warp that holds the first
#pragma unroll
                    for (int u = 0; u < GW; ++u) sm.half[((slice >> 1) * 16 + c * GW + u) * BM + rl] = v[u];
                } else {
#pragma unroll
                    for (int u = 0; u < GW; ++u) racc += v[u];
                }
                const float cs = warp_column_sums8(v, lane);
                if (lane < GW) colred[quarter * BN + cl0 + lane] = cs;
            } else {  // GRAM_DELTA, Eq. 3
                const float4* cr4 = reinterpret_cast<const float4*>(colrho + cl0);
                const float4* cx4 = reinterpret_cast<const float4*>(colx + cl0);
                const float4* cy4 = reinterpret_cast<const float4*>(coly + cl0);
                uint32_t kc[GW];                   // column-side keys: d^2 >= 0 orders like its bit pattern
#pragma unroll
                for (int q4 = 0; q4 < GW / 4; ++q4) {
                    const float4 cw = cw4[q4];
                    const float4 cr = cr4[q4];
                    float4 ca = make_float4(0.f, 0.f, 0.f, 0.f), cx = ca, cy = ca;
                    if (METRIC == 1) ca = ca4[q4];
                    if (SPATIAL) { cx = cx4[q4]; cy = cy4[q4]; }
                    const float crv[4] = {cr.x, cr.y, cr.z, cr.w};
                    float d2v[4], s2v[4];              // squared feature distance (unclamped), squared spatial distance
#pragma unroll
                    for (int h = 0; h < 2; ++h) {              // two neighbouring columns at a time
                        const int u = 4 * q4 + 2 * h;
                        const unsigned long long cw2 = h ? pack2(cw.z, cw.w) : pack2(cw.x, cw.y);
                        const unsigned long long ca2 = h ? pack2(ca.z, ca.w) : pack2(ca.x, ca.y);
                        const unsigned long long x2 = mul2(pack2(v[u], v[u + 1]), cw2);
                        const unsigned long long base2 = METRIC == 0 ? two2 : add2(ai2, ca2);
                        const float2 d2 = unpack2(fma2(x2, m2w2, base2));
                        d2v[2 * h] = d2.x;
                        d2v[2 * h + 1] = d2.y;
                        if (SPATIAL) {
                            const unsigned long long dx2 = add2(h ? pack2(cx.z, cx.w) : pack2(cx.x, cx.y), nxi2);
                            const unsigned long long dy2 = add2(h ? pack2(cy.z, cy.w) : pack2(cy.x, cy.y), nyi2);
                            const float2 s2 = unpack2(fma2(dx2, dx2, mul2(dy2, dy2)));
                            s2v[2 * h] = s2.x;
                            s2v[2 * h + 1] = s2.y;
                        }
                    }
#pragma unroll
                    for (int r = 0; r < 4; ++r) {
                        const int u = 4 * q4 + r;
                        const float d2 = fmaxf(d2v[r], 0.f);
                        // the pair may serve as (child, parent) at all (one comparison, & and not &&: the branches a pair took
                        // before cost the whole call 4 %, on 16 x 576 tokens 64.3 -> 61.9 us)
                        bool usable = (uint32_t)(cl0 + u - first_c) < usable_c;
                        if (SPATIAL) usable = usable & (s2v[r] <= g.tau2);
                        // with i < j: "j denser than i" is rho_j > rho_i, "i denser than j" is its complement
                        const bool jd = crv[r] > rho_i;
                        const float kr = (usable & jd) ? d2 : kInf;     // j as parent candidate of i (row side)
                        kc[u] = __float_as_uint((usable & !jd) ? d2 : kInf);   // i as parent candidate of j (column side)
                        if (kr < rbest) { rbest = kr; rbest_c = cl0 + u; }
                    }
                }
                // column side: minimum over this warp's 32 rows and the rows that attain it
                // (one lane stores what all lanes hold: selecting column u in lane u took three more instructions a column)
                uint32_t m[GW], rows[GW];
#pragma unroll
                for (int u = 0; u < GW; ++u) {
                    m[u] = __reduce_min_sync(0xffffffffu, kc[u]);
                    rows[u] = __ballot_sync(0xffffffffu, kc[u] == m[u]);
                }
                if (lane == 0) {
#pragma unroll
                    for (int u = 0; u < GW; u += 4) {
                        *reinterpret_cast<uint4*>(colred + quarter * BN + cl0 + u) = make_uint4(m[u], m[u + 1], m[u + 2], m[u + 3]);
                        *reinterpret_cast<uint4*>(colidx + quarter * BN + cl0 + u) =
                            make_uint4(rows[u], rows[u + 1], rows[u + 2], rows[u + 3]);
                    }
                }
            }
            if constexpr (GW == 8) {
                if (c + 1 < kGroups) {
                    tmem_ld8_wait(ld_nxt);
#pragma unroll
                    for (int u = 0; u < 8; ++u) ld_cur[u] = ld_nxt[u];
                }
            }
        }
    }

    if (MODE == GRAM_DIAG && g.bbox) {
        // ---- bounding box of the row block's positions: per warp by shuffles, the four row quarters through shared
        //      memory (rows outside the sample and coordinates that are not numbers leave the box alone)
        if (slice == 0) {
            float4 bx = make_float4(kInf, kInf, -kInf, -kInf);
            if (row_valid) {
                const float2 q = *reinterpret_cast<const float2*>(g.pos + 2 * (bo + i));
                bx = make_float4(q.x, q.y, q.x, q.y);
            }
#pragma unroll
            for (int off = 16; off > 0; off >>= 1) {
                bx.x = fminf(bx.x, __shfl_xor_sync(0xffffffffu, bx.x, off));
                bx.y = fminf(bx.y, __shfl_xor_sync(0xffffffffu, bx.y, off));
                bx.z = fmaxf(bx.z, __shfl_xor_sync(0xffffffffu, bx.z, off));
                bx.w = fmaxf(bx.w, __shfl_xor_sync(0xffffffffu, bx.w, off));
            }
            if (lane == 0) reinterpret_cast<float4*>(rowred)[quarter] = bx;
        }
        epi_bar_sync<kEpiThreads>();
        if (e == 0 && ok) {
            float4 bx = reinterpret_cast<const float4*>(rowred)[0];
#pragma unroll
            for (int q = 1; q < 4; ++q) {
                const float4 o = reinterpret_cast<const float4*>(rowred)[q];
                bx = make_float4(fminf(bx.x, o.x), fminf(bx.y, o.y), fmaxf(bx.z, o.z), fmaxf(bx.w, o.w));
            }
            g.bbox[(size_t)b * k.t.TI + ti] = bx;
        }
    }
    if (SYM) {
        // ---- combine the four column slices of every row and the four row quarters of every column
        if (slice > 0 && !(HALF && MODE == GRAM_RHO)) {
            rowred[(slice - 1) * BM + rl] = MODE == GRAM_RHO ? racc : rbest;
            if (MODE == GRAM_DELTA) rowidx[(slice - 1) * BM + rl] = rbest_c;
        }
        epi_bar_sync<kEpiThreads>();
        if (ok) {
            const int slot_base = b * k.t.slots();
            if (HALF && MODE == GRAM_RHO) {
                float* const part = g.part + (size_t)b * 5 * k.t.TI * k.t.n_pad;
                if (!(slice & 1) && row_valid) {
#pragma unroll
                    for (int u = 0; u < 16; ++u) racc += sm.half[((slice >> 1) * 16 + u) * BM + rl];
                    part[((size_t)(tj / 2) * k.t.n_pad + i) * 4 + (tj & 1) * 2 + (slice >> 1)] = racc;
                }
                for (int ce = e; ce < BN; ce += kEpiThreads)
                    if (J0 + ce < g.n)
                        part[(size_t)(4 * k.t.TI + ti) * k.t.n_pad + J0 + ce] =
                            ((colred[ce] + colred[BN + ce]) + colred[2 * BN + ce]) + colred[3 * BN + ce];
            } else if (MODE == GRAM_RHO) {
                if (slice == 0 && row_valid) {
#pragma unroll
                    for (int q = 0; q < NS - 1; ++q) racc += rowred[q * BM + rl];       // fixed order
                    g.part[((size_t)(slot_base + tj)) * k.t.n_pad + i] = racc;
                }
                for (int ce = e; ce < BN; ce += kEpiThreads)
                    if (J0 + ce < g.n)
                        g.part[((size_t)(slot_base + k.t.TJ + ti)) * k.t.n_pad + J0 + ce] =
                            ((colred[ce] + colred[BN + ce]) + colred[2 * BN + ce]) + colred[3 * BN + ce];
            } else {
                if (slice == 0 && row_valid) {
#pragma unroll
                    for (int q = 0; q < NS - 1; ++q) {                             // ascending columns: ties keep the lower one
                        const float other = rowred[q * BM + rl];
                        if (other < rbest) { rbest = other; rbest_c = rowidx[q * BM + rl]; }
                    }
                    if (rbest_c >= 0) {
                        const unsigned long long packed =
                            ((unsigned long long)__float_as_uint(rbest) << 32) |
                            (unsigned long long)(uint32_t)(J0 + rbest_c);
                        atomicMin(g.best + bo + i, packed);
                    }
                }
                for (int ce = e; ce < BN; ce += kEpiThreads) {
                    if (J0 + ce >= g.n) continue;
                    float bk = kInf;
                    int bi = -1;
#pragma unroll
                    for (int q = 0; q < 4; ++q) {                                  // ascending rows: ties keep the lower row
                        const float kk = colred[q * BN + ce];
                        if (kk < bk) { bk = kk; bi = I0 + q * 32 + __ffs(colidx[q * BN + ce]) - 1; }
                    }
                    if (bi >= 0) {
                        const unsigned long long packed =
                            ((unsigned long long)__float_as_uint(bk) << 32) | (unsigned long long)(uint32_t)bi;
                        atomicMin(g.best + bo + J0 + ce, packed);
                    }
                }
            }
        }
    }
    // shared arrays are rewritten for the next tile; all epilogue warps leave together or not at all
    return epi_bar_or<kEpiThreads>(!ok);
}

// ------------------------------------------------------------------------------------------------
// the kernel
// ------------------------------------------------------------------------------------------------
// MODE: GRAM_DIAG or GRAM_SIM.
template <int BN, int MODE, int METRIC>
__global__ void __launch_bounds__(kGemmThreads, 1)
gram_tc_kernel(const __grid_constant__ CUtensorMap map_a, const __grid_constant__ CUtensorMap map_b,
               const KernelArgs k) {
    using S = GemmSmem<BN>;
    constexpr bool DIAG = MODE == GRAM_DIAG;            // BN == BM: a diagonal tile multiplies the row block by itself
    constexpr int NS = kEpiSlices;
    constexpr int kEpiThreads = NS * 128;
    const GramArgs& g = k.g;
    extern __shared__ uint8_t smem_raw[];
    const uint32_t raw = smem_u32(smem_raw);
    const uint32_t tiles = (raw + 1023u) & ~1023u;                 // 1024-byte aligned for the 128B swizzle
    uint8_t* gen = smem_raw + (tiles - raw);
    EpiSmem sm;
    sm.template carve<BN>(gen + S::kTileBytes);
    uint64_t* bars = reinterpret_cast<uint64_t*>(gen + S::kTileBytes + S::kEpiBytes);
    // barriers: full[kStages], empty[kStages], tmem_full[2], tmem_empty[2], drain
    const uint32_t bar_full = smem_u32(bars);
    const uint32_t bar_empty = bar_full + 8 * S::kStages;
    const uint32_t bar_tfull = bar_empty + 8 * S::kStages;
    const uint32_t bar_tempty = bar_tfull + 16;
    const uint32_t bar_drain = bar_tempty + 16;
    uint32_t* tmem_slot = reinterpret_cast<uint32_t*>(bars + 2 * S::kStages + 5);
    volatile int* abort_flag = reinterpret_cast<volatile int*>(tmem_slot + 1);
    const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
    constexpr uint32_t kTmemCols = 2 * BN;

    if (threadIdx.x == 0) {
        for (int s = 0; s < S::kStages; ++s) {
            mbar_init(bar_full + 8 * s, 1);
            mbar_init(bar_empty + 8 * s, 1);
        }
        for (int a = 0; a < 2; ++a) {
            mbar_init(bar_tfull + 8 * a, 1);
            mbar_init(bar_tempty + 8 * a, kEpiThreads);   // every epilogue thread arrives once per tile
        }
        mbar_init(bar_drain, 1);
        *abort_flag = 0;
        asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
        asm volatile("prefetch.tensormap [%0];" ::"l"(reinterpret_cast<uint64_t>(&map_a)) : "memory");
        asm volatile("prefetch.tensormap [%0];" ::"l"(reinterpret_cast<uint64_t>(&map_b)) : "memory");
    }
    if (warp == 1) tmem_alloc(smem_u32(tmem_slot), kTmemCols);
    tc_fence_before();
    __syncthreads();
    tc_fence_after();
    const uint32_t tmem_base = *tmem_slot;

    // The kernels that follow on the stream may be scheduled from here on; they wait for this grid to complete
    // before they touch anything it writes.
    grid_dependency_launch_dependents();
    if (k.reports && blockIdx.x == 0 && threadIdx.x == 0) *g.status = VITCOP_OK;

    const long long total_tiles = k.total_tiles;
    const int KB = g.D / BK;
    uint32_t issued = 0, issued_parity = 0;    // thread 0, per stage: a load was issued / parity of its phase

    if (warp == 0) {
        // ------------------------------------------------------------------ TMA producer
        // The features are an input of the whole call (never written by the kernel before this one), so
        // the loads need not wait for the preceding grid.
        if (lane == 0) {
            const unsigned long long lim = k.limit_of(kRoleLoad);
            uint32_t stage = 0, phase = 0;
            bool ok = true;
            for (long long t = blockIdx.x; ok && t < total_tiles; t += gridDim.x) {
                int b, ti, tj;
                decode_tile<DIAG>(k, t, b, ti, tj);
                const int I0 = g.row0 + ti * BM, J0 = tj * BN;
                for (int kb = 0; kb < KB; ++kb) {
                    if (!mbar_wait(bar_empty + 8 * stage, phase ^ 1u, abort_flag, lim)) { ok = false; break; }
                    const uint32_t sa = tiles + stage * S::kStageBytes;
                    mbar_expect_tx(bar_full + 8 * stage, DIAG ? S::kABytes : S::kStageBytes);
                    tma_load_3d(sa, &map_a, bar_full + 8 * stage, kb * BK, I0, b);
                    if (!DIAG) tma_load_3d(sa + S::kABytes, &map_b, bar_full + 8 * stage, kb * BK, J0, b);
                    issued |= 1u << stage;
                    issued_parity = (issued_parity & ~(1u << stage)) | (phase << stage);
                    if (++stage == S::kStages) { stage = 0; phase ^= 1u; }
                }
            }
        }
    } else if (warp == 1) {
        // ------------------------------------------------------------------ MMA issuer
        if (lane == 0) {
            constexpr uint32_t idesc = umma_idesc_bf16(BM, BN);
            const unsigned long long lim = k.limit_of(kRoleMma);
            uint32_t stage = 0, phase = 0;
            uint32_t acc = 0, acc_phase = 0;
            bool ok = true;
            for (long long t = blockIdx.x; ok && t < total_tiles; t += gridDim.x) {
                if (!mbar_wait(bar_tempty + 8 * acc, acc_phase ^ 1u, abort_flag, lim)) { ok = false; break; }
                tc_fence_after();
                const uint32_t d_tmem = tmem_base + acc * BN;
                for (int kb = 0; kb < KB; ++kb) {
                    if (!mbar_wait(bar_full + 8 * stage, phase, abort_flag, lim)) { ok = false; break; }
                    tc_fence_after();
                    const uint32_t sa = tiles + stage * S::kStageBytes;
                    const uint64_t da = umma_desc_k128(sa), db = DIAG ? da : umma_desc_k128(sa + S::kABytes);
#pragma unroll
                    for (int kk = 0; kk < BK / UMMA_K; ++kk) {
                        // advancing 16 elements (32 bytes) along K inside the swizzle row: +2 in address units
                        tc_mma_bf16(d_tmem, da + (uint64_t)(2 * kk), db + (uint64_t)(2 * kk), idesc,
                                    (kb > 0 || kk > 0) ? 1u : 0u);
                    }
                    tc_commit(bar_empty + 8 * stage);      // frees the smem stage once these MMAs have read it
                    if (++stage == S::kStages) { stage = 0; phase ^= 1u; }
                }
                if (!ok) break;
                tc_commit(bar_tfull + 8 * acc);            // accumulator complete
                if (++acc == 2) { acc = 0; acc_phase ^= 1u; }
            }
            // let the MMAs issued finish before the operands and TMEM are released (the epilogue need not be waiting for them: it
            // may have given up)
            tc_commit(bar_drain);
            mbar_drain(bar_drain, 0);
        }
    } else {
        // ------------------------------------------------------------------ epilogue (warps 2 ..)
        uint32_t acc = 0, acc_phase = 0;
        bool ok = true;
        grid_dependency_wait();                            // w, a, rho, best come from the preceding kernels

        for (long long t = blockIdx.x; t < total_tiles; t += gridDim.x) {
            EpiCall c;
            decode_tile<DIAG>(k, t, c.b, c.ti, c.tj);
            c.tmem_tile = tmem_base + acc * BN;
            c.wait_bar = bar_tfull + 8 * acc;
            c.wait_parity = acc_phase;
            c.arrive_bar = bar_tempty + 8 * acc;
            c.abort_flag = abort_flag;
            c.limit_ns = k.limit_of(kRoleEpi);
            if (epi_tile<BN, MODE, METRIC, false, NS>(k, sm, c, ok)) break;
            if (++acc == 2) { acc = 0; acc_phase ^= 1u; }
        }
    }

    tc_fence_before();
    __syncthreads();
    if (warp == 1) {
        tc_fence_after();
        tmem_dealloc(tmem_base, kTmemCols);
    }
    if (threadIdx.x == 0 && *abort_flag) {
        // Some role gave up, so loads this thread issued may never have been consumed: give the copies still in
        // flight into this CTA's shared memory time to land before the CTA goes away.
        for (int s = 0; s < S::kStages; ++s)
            if (issued >> s & 1u) mbar_drain(bar_full + 8 * s, issued_parity >> s & 1u);
        if (!k.reports) atomicMax(g.status, VITCOP_ERR_TIMEOUT);
    }
    if (threadIdx.x == 0 && k.reports) report_gave_up(g.status, *abort_flag != 0);
}


// ------------------------------------------------------------------------------------------------
// the resident kernel: density and delta from ONE pass over the Gram tiles (small problems)
// ------------------------------------------------------------------------------------------------
// The unit of work is one row block (128 tokens) against two adjacent column blocks -- against one, or half of one, where that
// still leaves no more units than SMs: the epilogue of a unit is most of the kernel's time (one sample of 576 tokens on 9, 15,
// 25 CTAs: 30, 24, 15 us; the last with the factors' faster way to the other CTAs).  Two column blocks: one MMA of N = 256 per
// k-step, the row operand loaded once for both 128 x 128 tiles (a quarter less operand traffic than tile by tile,
// and the tensor cores run N = 256 at twice the rate of N = 128).  Row block ti owns the column blocks ti .. TI - 1,
// paired from the diagonal on; the last unit of a row is half empty when their number is odd (the rows of its
// missing column block lie outside the tensor and are zero-filled at no cost in traffic).  A CTA owns at most
// kResidentUnits units and keeps their accumulators in tensor memory (2 x 256 of the 512 columns).  Units that
// start with a diagonal tile are numbered first, so that these accumulators are the first to complete.
// Half a column block: the sums over 32 columns that the other units form in one warp are handed from the warp with the
// first 16 to the one with the rest, and the four of a tile are stored side by side and joined by the reader, so that every
// unit gives the same bits.
// Phases of the epilogue warps, which treat a unit as two tiles of 128 x 128 (or one of 128 x 64):
//   0. the diagonal tiles yield g_ii -> per-token normalisation factors, published token by token
//   1. density epilogue of every tile (when the factors of its row and column block are there) -> rho partials;
//      grid-wide barrier
//   2. delta epilogue of every tile, re-reading the accumulators; rho of the tile's rows and columns is summed
//      from the partials on the way (the diagonal tiles publish it)
// The grid (at most one CTA per SM) is launched cooperatively, so all CTAs are resident together; factors and barrier
// are words in global memory, cleared by clear_kernel (filter.cu) in front, with bounded waits.  No wait can form a cycle: a factor
// is published by a CTA that has waited for nothing but its own tensor-core work and that kernel.
// The load warp and the MMA warp are idle once the CTA's last MMA is issued, and so are, a little later, the
// operand buffers and -- for the rest of the kernel, which is arithmetic on the accumulators -- the memory system:
// if the caller has a K-norm (Eq. 4) to compute, these two warps and two more stream K through the operand buffers with tensor
// copies and reduce it there (resident_knorm).
constexpr int kResidentUnits = 2;
constexpr int kResidentBN = 2 * BM;                       // columns of a unit
constexpr int kResidentEpiThreads = 512;
constexpr int kResidentThreads = 64 + kResidentEpiThreads + 64;
constexpr int kKnThreads = 128;                           // of the four warps in front of and behind the epilogue's

__device__ __forceinline__ unsigned int ld_acquire_u32(const unsigned int* p) {
    unsigned int v;
    asm volatile("ld.acquire.gpu.global.u32 %0, [%1];" : "=r"(v) : "l"(p) : "memory");
    return v;
}

// Barrier over all CTAs of the grid, called by the epilogue threads.  Returns true when the grid must give up.
// One thread speaks for the CTA: the CTA barrier orders every epilogue thread's writes before that thread's release
// (and its acquire before their later reads), so the other threads need none of their own.
__device__ __forceinline__ bool resident_grid_barrier(unsigned int* counter, volatile int* abort_flag, bool aborted,
                                                      unsigned long long limit_ns) {
    epi_bar_sync<kResidentEpiThreads>();
    if (threadIdx.x == 64 && !aborted) {
        asm volatile("red.release.gpu.global.add.u32 [%0], 1;" ::"l"(counter) : "memory");
        const unsigned long long t0 = global_ns();
        while (ld_acquire_u32(counter) < gridDim.x) {
            if (limit_ns == 0ull || global_ns() - t0 > limit_ns) { *abort_flag = 1; break; }
        }
    }
    return epi_bar_or<kResidentEpiThreads>(aborted || *abort_flag != 0);
}

// Unit t of the resident sweep: the B * TI units that start with a diagonal tile first, then the others, sample
// by sample and row block by row block.
struct ResidentUnit {
    int b, ti, tj0;        // sample, row block, first column block
    int width;             // column blocks inside the tensor: unit_w, or fewer for the last unit of a row
};
__host__ __device__ inline int resident_extra_units(int TI, int unit_w) {
    int e = 0;
    for (int ti = 0; ti < TI; ++ti) e += (TI - ti + unit_w - 1) / unit_w - 1;
    return e;
}
// Units of 64 columns (tj0 counts blocks of 64): block ti owns the column blocks from 2 ti on.
__host__ __device__ inline int resident_half_units(int TI, int TJ) {
    int e = 0;
    for (int ti = 0; ti < TI; ++ti) e += TJ - 2 * ti;
    return e;
}
__device__ __forceinline__ ResidentUnit decode_half_unit(const KernelArgs& k, long long t) {
    const int TJ = (k.g.n + 63) / 64;
    const long long n_diag = (long long)k.g.B * TJ;
    ResidentUnit u;
    u.width = 1;
    if (t < n_diag) {
        u.b = (int)(t / TJ);
        u.tj0 = (int)(t - (long long)u.b * TJ);
        u.ti = u.tj0 / 2;
    } else {
        const long long x = t - n_diag;
        u.b = (int)(x / k.extra_units_per_b);
        int r = (int)(x - (long long)u.b * k.extra_units_per_b);
        int ti = 0;
        for (int m = TJ - 2; r >= m; ++ti, m -= 2) r -= m;     // units of row block ti behind its diagonal ones
        u.ti = ti;
        u.tj0 = 2 * ti + 2 + r;
    }
    return u;
}
__device__ __forceinline__ ResidentUnit decode_resident_unit(const KernelArgs& k, long long t) {
    const int TI = k.t.TI;
    const long long n_diag = (long long)k.g.B * TI;
    ResidentUnit u;
    if (t < n_diag) {
        u.b = (int)(t / TI);
        u.ti = (int)(t - (long long)u.b * TI);
        u.tj0 = u.ti;
    } else {
        const long long x = t - n_diag;                    // extra_units_per_b > 0 here
        u.b = (int)(x / k.extra_units_per_b);
        int r = (int)(x - (long long)u.b * k.extra_units_per_b);
        int ti = 0;
        for (; ti < TI; ++ti) {
            const int m = (TI - ti + k.unit_w - 1) / k.unit_w - 1;             // units of row block ti beyond its first
            if (r < m) break;
            r -= m;
        }
        u.ti = ti;
        u.tj0 = ti + k.unit_w * (r + 1);
    }
    u.width = min(k.unit_w, TI - u.tj0);
    return u;
}

constexpr int kKnChunkTokens = 8;                          // tokens per chunk: 16 threads each
constexpr int kKnBuffers = 3;
__host__ __device__ constexpr int knorm_buffers(int H, int d) {         // 0: a chunk does not fit
    const long long fit = (long long)GemmSmem<kResidentBN>::kTileBytes / ((long long)H * kKnChunkTokens * d * 2);
    return fit < kKnBuffers ? (int)fit : kKnBuffers;
}

// K-norm (Eq. 4) by the warps beside the epilogue's, after the CTA's last MMA has completed.  Chunks of eight consecutive
// tokens of one sample, all heads, are copied into the operand buffers, up to three chunks in flight; sixteen threads
// reduce one token as in the stand-alone kernel, so that both give the same bits.  One tensor copy per chunk: as bulk copies, one
// per head, they took a warp 1.3 us to issue where the arithmetic takes 1.0 (32 heads).
__device__ __forceinline__ void resident_knorm(const GramArgs& g, const CUtensorMap* map_k, const uint8_t* buf_gen, uint32_t buf_smem,
                                               uint32_t bar_kn, uint32_t bar_last_mma,
                                               volatile int* abort_flag, unsigned long long limit_ns) {
    const int tid = threadIdx.x < 64 ? threadIdx.x : threadIdx.x - kResidentEpiThreads;        // 0 .. 127
    auto all_ok = [](bool ok) {
        uint32_t out;
        asm volatile(
            "{\n\t.reg .pred p, q;\n\t"
            "setp.eq.b32 p, %1, 0;\n\t"
            "bar.red.or.pred q, 2, %2, p;\n\t"
            "selp.u32 %0, 0, 1, q;\n\t}"
            : "=r"(out) : "r"((uint32_t)ok), "n"(kKnThreads) : "memory");
        return out != 0;
    };
    // the tensor cores read the operand buffers until the last MMA completes
    if (!all_ok(mbar_wait(bar_last_mma, 0, abort_flag, limit_ns))) return;

    const int H = g.kn_H, d8 = g.kn_d / 8, Nv = g.kn_Nv;
    const uint32_t chunk_bytes = (uint32_t)(H * kKnChunkTokens * d8) * 16u;
    const int nbuf = knorm_buffers(H, g.kn_d);             // >= 1 (gram_resident_takes_knorm)
    const int chunks_per_b = (Nv + kKnChunkTokens - 1) / kKnChunkTokens;
    const long long total = (long long)g.kn_B * chunks_per_b;
    auto issue = [&](long long c, int buf) {               // thread 0
        const int b = (int)(c / chunks_per_b), i0 = (int)(c - (long long)b * chunks_per_b) * kKnChunkTokens;
        mbar_expect_tx(bar_kn + 8 * buf, chunk_bytes);     // (rows past the sequence arrive as zeros)
        tma_load_4d(buf_smem + (uint32_t)buf * chunk_bytes, map_k, bar_kn + 8 * buf, 0, g.kn_vis_start + i0, 0, b);
    };
    long long issued = 0;                                  // chunks this CTA has requested (thread 0)
    if (tid == 0)
        for (; issued < nbuf && blockIdx.x + issued * gridDim.x < total; ++issued)
            issue(blockIdx.x + issued * gridDim.x, (int)issued);

    const int tk = tid >> 4, s = tid & 15;
    long long it = 0;
    bool ok = true;
    for (long long c = blockIdx.x; c < total; c += gridDim.x, ++it) {
        const int buf = (int)(it % nbuf);
        ok = all_ok(mbar_wait(bar_kn + 8 * buf, (uint32_t)((it / nbuf) & 1), abort_flag, limit_ns));
        if (!ok) break;
        const int b = (int)(c / chunks_per_b);
        const int i0 = (int)(c - (long long)b * chunks_per_b) * kKnChunkTokens;
        const int cnt = min(kKnChunkTokens, Nv - i0);
        const uint4* rows = reinterpret_cast<const uint4*>(buf_gen + (size_t)buf * chunk_bytes) + (size_t)tk * d8;
        const int head16 = kKnChunkTokens * d8;            // uint4 per head of a chunk
        float a0 = 0.f, a1 = 0.f;
        if (tk < cnt) {
            for (int piece = s; piece < d8; piece += 16) {
#pragma unroll 8
                for (int h = 0; h < H; ++h) knorm_sq_acc(rows[(size_t)h * head16 + piece], a0, a1);
            }
        }
        float part = a0 + a1;
#pragma unroll
        for (int off = 8; off > 0; off >>= 1) part += __shfl_xor_sync(0xffffffffu, part, off);
        if (tk < cnt && s == 0) g.kn_score[(size_t)b * Nv + i0 + tk] = sqrtf(part);
        asm volatile("bar.sync 2, %0;" ::"n"(kKnThreads) : "memory");      // the buffer has been read by everyone
        if (tid == 0) {
            const long long cn = blockIdx.x + issued * gridDim.x;
            if (cn < total) {
                asm volatile("fence.proxy.async.shared::cta;" ::: "memory");
                issue(cn, buf);
                ++issued;
            }
        }
    }
    if (!ok && tid == 0) {
        // giving up: wait (bounded) for the copies still in flight before the CTA's shared memory goes away
        for (long long j = it; j < issued; ++j) mbar_drain(bar_kn + 8 * (int)(j % nbuf), (uint32_t)((j / nbuf) & 1));
    }
}

// BN: columns of the epilogue's tiles: 128, or 64 for units of half a tile.
template <int METRIC, bool SPATIAL, int BN>
__global__ void __launch_bounds__(kResidentThreads, 1)
gram_resident_kernel(const __grid_constant__ CUtensorMap map_a, const __grid_constant__ CUtensorMap map_b,
                     const __grid_constant__ CUtensorMap map_k, const KernelArgs k) {
    constexpr bool HALF = BN == 64;
    constexpr int NS = 4;
    using S = GemmSmem<kResidentBN>;                       // stages of 128 + 256 operand rows
    constexpr uint32_t kStages = HALF ? HalfUnitSmem::kStages : S::kStages;
    constexpr uint32_t kStageBytes = HALF ? HalfUnitSmem::kStageBytes : S::kStageBytes;
    constexpr int kEpiBytes = HALF ? HalfUnitSmem::kEpiBytes : S::kEpiBytes;
    auto unit_of = [&](long long t) { return HALF ? decode_half_unit(k, t) : decode_resident_unit(k, t); };
    auto on_diagonal = [](const ResidentUnit& u) { return u.ti == (HALF ? u.tj0 / 2 : u.tj0); };
    const GramArgs& g = k.g;
    extern __shared__ uint8_t smem_raw[];
    const uint32_t raw = smem_u32(smem_raw);
    const uint32_t tiles = (raw + 1023u) & ~1023u;
    uint8_t* gen = smem_raw + (tiles - raw);
    EpiSmem sm;
    sm.template carve<BN>(gen + S::kTileBytes);
    uint64_t* bars = reinterpret_cast<uint64_t*>(gen + S::kTileBytes + kEpiBytes);
    // barriers: full[kStages], empty[kStages], tmem_full[kResidentUnits], drain, knorm[kKnBuffers]
    const uint32_t bar_full = smem_u32(bars);
    const uint32_t bar_empty = bar_full + 8 * kStages;
    const uint32_t bar_tfull = bar_empty + 8 * kStages;
    const uint32_t bar_drain = bar_tfull + 8 * kResidentUnits;
    const uint32_t bar_kn = bar_drain + 8;
    uint32_t* tmem_slot = reinterpret_cast<uint32_t*>(bars + 2 * kStages + kResidentUnits + 1 + kKnBuffers);
    static_assert((2 * kStages + kResidentUnits + 1 + kKnBuffers) * 8 + 8 <= S::kBarBytes, "barrier block too small");
    volatile int* abort_flag = reinterpret_cast<volatile int*>(tmem_slot + 1);

    const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
    constexpr uint32_t kTmemCols = kResidentUnits * kResidentBN;   // 512: the whole tensor memory of the SM

    if (threadIdx.x == 0) {
        for (uint32_t s = 0; s < kStages; ++s) {
            mbar_init(bar_full + 8 * s, 1);
            mbar_init(bar_empty + 8 * s, 1);
        }
        for (int a = 0; a < kResidentUnits; ++a) mbar_init(bar_tfull + 8 * a, 1);
        mbar_init(bar_drain, 1);
        for (int a = 0; a < kKnBuffers; ++a) mbar_init(bar_kn + 8 * a, 1);
        *abort_flag = 0;
        asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
        asm volatile("prefetch.tensormap [%0];" ::"l"(reinterpret_cast<uint64_t>(&map_a)) : "memory");
        asm volatile("prefetch.tensormap [%0];" ::"l"(reinterpret_cast<uint64_t>(&map_b)) : "memory");
    }
    if (warp == 1) tmem_alloc(smem_u32(tmem_slot), kTmemCols);
    tc_fence_before();
    __syncthreads();
    tc_fence_after();
    const uint32_t tmem_base = *tmem_slot;

    const long long total_units = k.total_tiles;          // <= kResidentUnits * gridDim.x (checked by the launcher)
    const int KB = g.D / BK;
    uint32_t issued = 0, issued_parity = 0;               // thread 0, per stage: a load was issued / parity of its phase

    if (warp == 0) {
        // ------------------------------------------------------------------ TMA producer
        if (lane == 0) {
            const unsigned long long lim = k.limit_of(kRoleLoad);
            uint32_t stage = 0, phase = 0;
            bool ok = true;
            for (long long t = blockIdx.x; ok && t < total_units; t += gridDim.x) {
                const ResidentUnit u = unit_of(t);
                const int I0 = u.ti * BM, J0 = u.tj0 * BN;
                for (int kb = 0; kb < KB; ++kb) {
                    if (!mbar_wait(bar_empty + 8 * stage, phase ^ 1u, abort_flag, lim)) { ok = false; break; }
                    const uint32_t sa = tiles + stage * kStageBytes;
                    // rows of the box past the sample's last token are zero-filled and still count as received
                    mbar_expect_tx(bar_full + 8 * stage, HALF ? kStageBytes : S::kABytes + (uint32_t)k.unit_w * S::kABytes);
                    tma_load_3d(sa, &map_a, bar_full + 8 * stage, kb * BK, I0, u.b);
                    tma_load_3d(sa + S::kABytes, &map_b, bar_full + 8 * stage, kb * BK, J0, u.b);
                    issued |= 1u << stage;
                    issued_parity = (issued_parity & ~(1u << stage)) | (phase << stage);
                    if (++stage == kStages) { stage = 0; phase ^= 1u; }
                }
            }
        }
    } else if (warp == 1) {
        // ------------------------------------------------------------------ MMA issuer: unit s of this CTA -> columns 256 s ..
        if (lane == 0) {
            const uint32_t idesc = !HALF && k.unit_w == 2 ? umma_idesc_bf16(BM, kResidentBN) : umma_idesc_bf16(BM, BN);
            const unsigned long long lim = k.limit_of(kRoleMma);
            uint32_t stage = 0, phase = 0;
            uint32_t slot = 0;
            bool ok = true;
            for (long long t = blockIdx.x; ok && t < total_units; t += gridDim.x, ++slot) {
                const uint32_t d_tmem = tmem_base + slot * kResidentBN;
                for (int kb = 0; kb < KB; ++kb) {
                    if (!mbar_wait(bar_full + 8 * stage, phase, abort_flag, lim)) { ok = false; break; }
                    tc_fence_after();
                    const uint32_t sa = tiles + stage * kStageBytes;
                    const uint64_t da = umma_desc_k128(sa), db = umma_desc_k128(sa + S::kABytes);
#pragma unroll
                    for (int kk = 0; kk < BK / UMMA_K; ++kk)
                        tc_mma_bf16(d_tmem, da + (uint64_t)(2 * kk), db + (uint64_t)(2 * kk), idesc,
                                    (kb > 0 || kk > 0) ? 1u : 0u);
                    tc_commit(bar_empty + 8 * stage);
                    if (++stage == kStages) { stage = 0; phase ^= 1u; }
                }
                if (!ok) break;
                tc_commit(bar_tfull + 8 * slot);
            }
            tc_commit(bar_drain);                          // (as in gram_tc_kernel)
            mbar_drain(bar_drain, 0);
        }
    }
    if (warp < 2 || warp >= 2 + kResidentEpiThreads / 32) {
        __syncwarp();
        if (g.kn_K) {
            const long long my_units = (total_units - blockIdx.x + gridDim.x - 1) / gridDim.x;   // >= 1
            resident_knorm(g, &map_k, gen, tiles, bar_kn, bar_tfull + 8 * (uint32_t)(my_units - 1),
                           abort_flag, k.limit_of(kRoleLoad | kRoleMma));
        }
    } else {
        // ------------------------------------------------------------------ epilogue (warps 2..17)
        bool ok = true, stop = false;
        const unsigned long long lim = k.limit_of(kRoleEpi);
        grid_dependency_wait();                            // clear_kernel has cleared status word, factors and barrier counter
        // tile s (0 or 1) of this CTA's unit number `slot`
        auto tile_call = [&](const ResidentUnit& u, uint32_t slot, int s, bool wait_mma) {
            EpiCall c;
            c.b = u.b;
            c.ti = u.ti;
            c.tj = u.tj0 + s;
            c.tmem_tile = tmem_base + slot * kResidentBN + (uint32_t)s * BN;
            c.wait_bar = wait_mma ? bar_tfull + 8 * slot : 0;
            c.wait_parity = 0;
            c.arrive_bar = 0;
            c.abort_flag = abort_flag;
            c.limit_ns = lim;
            return c;
        };

        // ---- phase 0: the diagonal tiles give g_ii, hence the per-token factors every other epilogue needs
        uint32_t slot = 0;
        for (long long t = blockIdx.x; t < total_units && !stop; t += gridDim.x, ++slot) {
            const ResidentUnit u = unit_of(t);
            if (!on_diagonal(u)) continue;                  // uniform over the CTA
            const EpiCall c = tile_call(u, slot, 0, true);
            stop = epi_tile<BN, GRAM_DIAG, METRIC, false, NS, 8>(k, sm, c, ok);
        }
        // ---- phase 1: density partials, tile by tile as soon as the factors of its row and column block exist
        slot = 0;
        for (long long t = blockIdx.x; t < total_units && !stop; t += gridDim.x, ++slot) {
            const ResidentUnit u = unit_of(t);
            for (int s = 0; s < u.width && !stop; ++s) {
                const EpiCall c = tile_call(u, slot, s, true);
                stop = epi_tile<BN, GRAM_RHO, METRIC, false, NS, 8>(k, sm, c, ok);
            }
        }
        stop = resident_grid_barrier(g.grid_sync, abort_flag, stop, lim);
        // The kernels that follow cannot share an SM with a CTA of this grid (registers, shared memory); from here
        // on they may at least be set up.
        grid_dependency_launch_dependents();
        // ---- phase 2: delta and parents from the same accumulators; every tile sums the rho of its own rows and
        //      columns from the partials (fixed order: the same bits everywhere)
        slot = 0;
        for (long long t = blockIdx.x; t < total_units && !stop; t += gridDim.x, ++slot) {
            const ResidentUnit u = unit_of(t);
            for (int s = 0; s < u.width && !stop; ++s) {
                const EpiCall c = tile_call(u, slot, s, false);
                stop = epi_tile<BN, GRAM_DELTA, METRIC, SPATIAL, NS, 8>(k, sm, c, ok);
            }
        }
    }

    tc_fence_before();
    __syncthreads();
    if (warp == 1) {
        tc_fence_after();
        tmem_dealloc(tmem_base, kTmemCols);
    }
    if (threadIdx.x == 0 && *abort_flag) {
        // (see gram_tc_kernel: unconsumed operand loads must have landed before the CTA goes away)
        for (uint32_t s = 0; s < kStages; ++s)
            if (issued >> s & 1u) mbar_drain(bar_full + 8 * s, issued_parity >> s & 1u);
        atomicMax(g.status, VITCOP_ERR_TIMEOUT);
    }
    grid_dependency_launch_dependents();
}

// ------------------------------------------------------------------------------------------------
// host side
// ------------------------------------------------------------------------------------------------
typedef CUresult (*EncodeTiledFn)(CUtensorMap*, CUtensorMapDataType, cuuint32_t, void*, const cuuint64_t*,
                                  const cuuint64_t*, const cuuint32_t*, const cuuint32_t*, CUtensorMapInterleave,
                                  CUtensorMapSwizzle, CUtensorMapL2promotion, CUtensorMapFloatOOBfill);

EncodeTiledFn encode_tiled_fn() {
    static const EncodeTiledFn fn = []() -> EncodeTiledFn {            // (threads that come first together wait for one another)
        void* p = nullptr;
        cudaDriverEntryPointQueryResult q;
        if (cudaGetDriverEntryPoint("cuTensorMapEncodeTiled", &p, cudaEnableDefault, &q) == cudaSuccess &&
            q == cudaDriverEntryPointSuccess)
            return reinterpret_cast<EncodeTiledFn>(p);
        return nullptr;
    }();
    return fn;
}

// 3-D view (D, n, B) of the bf16 feature tensor with a (64, box_rows, 1) box and the 128-byte swizzle.
bool make_feat_map(CUtensorMap* map, const void* feat, int B, int n, int D, int box_rows) {
    EncodeTiledFn fn = encode_tiled_fn();
    if (!fn) return false;
    cuuint64_t dims[3] = {(cuuint64_t)D, (cuuint64_t)n, (cuuint64_t)B};
    cuuint64_t strides[2] = {(cuuint64_t)D * 2, (cuuint64_t)n * D * 2};
    cuuint32_t box[3] = {(cuuint32_t)BK, (cuuint32_t)box_rows, 1};
    cuuint32_t estr[3] = {1, 1, 1};
    return fn(map, CU_TENSOR_MAP_DATA_TYPE_BFLOAT16, 3, const_cast<void*>(feat), dims, strides, box, estr,
              CU_TENSOR_MAP_INTERLEAVE_NONE, CU_TENSOR_MAP_SWIZZLE_128B, CU_TENSOR_MAP_L2_PROMOTION_L2_256B,
              CU_TENSOR_MAP_FLOAT_OOB_FILL_NONE) == CUDA_SUCCESS;
}

// Time limit of the kernels' bounded waits and, for failure-handling tests, the roles whose waits give up at once.
std::atomic<unsigned long long> g_wait_ns{kWaitLimitNs};
std::atomic<int> g_expire_roles{0};

int num_sms() {
    static std::atomic<int> sms[kMaxDevices];
    const int dev = current_device();
    int v = sms[dev].load(std::memory_order_relaxed);
    if (v <= 0) {
        if (cudaDeviceGetAttribute(&v, cudaDevAttrMultiProcessorCount, dev) != cudaSuccess || v <= 0) v = 148;
        sms[dev].store(v, std::memory_order_relaxed);
    }
    return v;
}

template <int BN, int MODE, int METRIC>
int launch_one(const CUtensorMap& ma, const CUtensorMap& mb, const KernelArgs& k, cudaStream_t stream, bool pdl) {
    using S = GemmSmem<BN>;
    static DoneOnDevice attr_done;
    auto kern = gram_tc_kernel<BN, MODE, METRIC>;
    const int arc = allow_dynamic_smem(kern, S::kTotal, attr_done);
    if (arc != VITCOP_OK) return arc;
    cudaLaunchConfig_t cfg = {};
    cfg.gridDim = dim3((unsigned)(k.total_tiles < num_sms() ? k.total_tiles : num_sms()));
    cfg.blockDim = dim3(kGemmThreads);
    cfg.dynamicSmemBytes = S::kTotal;
    cfg.stream = stream;
    cudaLaunchAttribute attr[1];
    attr[0].id = cudaLaunchAttributeProgrammaticStreamSerialization;
    attr[0].val.programmaticStreamSerializationAllowed = 1;
    cfg.attrs = attr;
    cfg.numAttrs = pdl_allowed(pdl) ? 1 : 0;
    KernelTimeScope timed(MODE == GRAM_DIAG ? "gram_tc_kernel<diag>" : "gram_tc_kernel<sim>", stream);
    return record_cuda(cudaLaunchKernelEx(&cfg, kern, ma, mb, k));
}

// As many CTAs as there are SMs (never fewer than the units need): the shortest chain of units per CTA.
long long resident_ctas(long long units) {
    const long long least = (units + kResidentUnits - 1) / kResidentUnits, sms = num_sms();
    return units < sms ? units : least > sms ? least : sms;
}

template <int METRIC, bool SPATIAL, int BN>
int launch_resident_one(const CUtensorMap& ma, const CUtensorMap& mb, const CUtensorMap& mk, const KernelArgs& k, cudaStream_t stream) {
    using S = GemmSmem<kResidentBN>;
    static DoneOnDevice attr_done;
    auto kern = gram_resident_kernel<METRIC, SPATIAL, BN>;
    constexpr int kSmem = S::kTotal + (BN == 64 ? HalfUnitSmem::kEpiBytes - S::kEpiBytes : 0);
    const int arc = allow_dynamic_smem(kern, kSmem, attr_done);
    if (arc != VITCOP_OK) return arc;
    cudaLaunchConfig_t cfg = {};
    cfg.gridDim = dim3((unsigned)resident_ctas(k.total_tiles));
    cfg.blockDim = dim3(kResidentThreads);
    cfg.dynamicSmemBytes = kSmem;
    cfg.stream = stream;
    cudaLaunchAttribute attr[2];
    attr[0].id = cudaLaunchAttributeCooperative;          // all CTAs resident together: they wait for one another
    attr[0].val.cooperative = 1;
    // (Of its own stream only clear_kernel can still be running when the grid starts, and that waits for nothing any more.)
    attr[1].id = cudaLaunchAttributeProgrammaticStreamSerialization;
    attr[1].val.programmaticStreamSerializationAllowed = 1;
    cfg.attrs = attr;
    cfg.numAttrs = pdl_allowed(true) ? 2 : 1;
    KernelTimeScope timed("gram_resident_kernel", stream);
    return record_cuda(cudaLaunchKernelEx(&cfg, kern, ma, mb, mk, k));
}

}  // namespace

int gram_num_sms() { return num_sms(); }

bool make_rowmajor_bf16_map(CUtensorMap* map, const void* base, int batches, int rows, int cols, int box_rows) {
    return make_feat_map(map, base, batches, rows, cols, box_rows);
}

bool make_keys_map(CUtensorMap* map, const void* K, int B, int H, int N, int d, int box_tokens, int box_heads) {
    EncodeTiledFn fn = encode_tiled_fn();
    if (!fn) return false;
    const cuuint64_t row = (cuuint64_t)d * 2;
    cuuint64_t dims[4] = {(cuuint64_t)d, (cuuint64_t)N, (cuuint64_t)H, (cuuint64_t)B};
    cuuint64_t strides[3] = {row, row * N, row * N * H};
    cuuint32_t box[4] = {(cuuint32_t)d, (cuuint32_t)box_tokens, (cuuint32_t)box_heads, 1};
    cuuint32_t estr[4] = {1, 1, 1, 1};
    return fn(map, CU_TENSOR_MAP_DATA_TYPE_BFLOAT16, 4, const_cast<void*>(K), dims, strides, box, estr, CU_TENSOR_MAP_INTERLEAVE_NONE,
              CU_TENSOR_MAP_SWIZZLE_NONE, CU_TENSOR_MAP_L2_PROMOTION_NONE, CU_TENSOR_MAP_FLOAT_OOB_FILL_NONE) == CUDA_SUCCESS;
}

unsigned long long gram_wait_limit_ns() { return g_wait_ns.load(); }
int pair_expire_roles() {
    const int r = g_expire_roles.load();
    return (r | r >> 3) & 7;
}

void gram_set_wait_debug(unsigned long long limit_ns, int expire_roles) {
    g_wait_ns.store(limit_ns ? limit_ns : kWaitLimitNs);
    g_expire_roles.store(expire_roles & 63);
}

int launch_gram_sweep(int mode, const void* feat, const GramArgs& args, cudaStream_t stream, bool pdl) {
    if (mode != GRAM_DIAG && mode != GRAM_SIM) return VITCOP_ERR_INVALID_ARG;
    KernelArgs k;
    k.g = args;
    k.t = make_gram_tiling(args.n);
    if (mode == GRAM_SIM) {
        // plain rectangle: rows [row0, row_end) x all columns
        k.t.TI = (args.row_end - args.row0 + BM - 1) / BM;
        k.t.tiles_per_b = k.t.TI * k.t.TJ;
    } else {
        k.g.row0 = 0;
        k.g.row_end = args.n;
        k.t.tiles_per_b = k.t.TI;                              // one tile per 128-row block
    }
    k.total_tiles = (long long)args.B * k.t.tiles_per_b;
    k.extra_units_per_b = 0;
    k.unit_w = 0;
    k.wait_ns = g_wait_ns.load();
    k.expire_roles = g_expire_roles.load() & 7;
    k.reports = args.reports;
    if (k.total_tiles <= 0) return VITCOP_OK;
    CUtensorMap ma, mb;
    if (!make_feat_map(&ma, feat, args.B, args.n, args.D, BM) || !make_feat_map(&mb, feat, args.B, args.n, args.D, BM))
        return VITCOP_ERR_CUDA;
    const bool euclid = args.metric == 1;
    if (mode == GRAM_DIAG)
        return euclid ? launch_one<BM, GRAM_DIAG, 1>(ma, mb, k, stream, pdl)
                      : launch_one<BM, GRAM_DIAG, 0>(ma, mb, k, stream, pdl);
    return euclid ? launch_one<BM, GRAM_SIM, 1>(ma, mb, k, stream, pdl)
                  : launch_one<BM, GRAM_SIM, 0>(ma, mb, k, stream, pdl);
}

bool gram_fits_resident(int B, int n) {
    static std::atomic<int> cooperative[kMaxDevices];     // the resident kernel needs a cooperative launch: 1 yes, 2 no
    const int dev = current_device();
    int c = cooperative[dev].load(std::memory_order_relaxed);
    if (c == 0) {
        int v = 0;
        c = (cudaDeviceGetAttribute(&v, cudaDevAttrCooperativeLaunch, dev) == cudaSuccess && v) ? 1 : 2;
        cooperative[dev].store(c, std::memory_order_relaxed);
    }
    if (c != 1) return false;
    const int ti = (n + BM - 1) / BM;
    const long long units = (long long)B * (ti + resident_extra_units(ti, 2));
    return units > 0 && units <= (long long)kResidentUnits * num_sms();
}

// Units of 64 columns where that still leaves one unit per SM at most: with more, a CTA's second unit would cost what the
// shorter units save (a unit's epilogue is most of the kernel's time).  One sample of 576 tokens: 25 CTAs instead of 15,
// the call 35.9 -> 33.8 us; beyond the line the units of 128 or 256 columns use every SM as well.
bool gram_resident_halves(int B, int n) {
    const long long units = resident_half_units((n + BM - 1) / BM, (n + 63) / 64);
    return (long long)B * units <= num_sms();
}

// How a problem is cut into units.
struct ResidentCut {
    bool halves;                                           // units of 64 columns
    int unit_w, extra_per_b;                               // column blocks of a unit; units of a sample that hold no diagonal tile
    long long total;
    ResidentCut(int B, int n) {
        const int TI = (n + BM - 1) / BM, TJ = (n + 63) / 64;
        halves = gram_resident_halves(B, n);
        unit_w = (long long)B * TI * (TI + 1) / 2 <= num_sms() ? 1 : 2;
        const int units = halves ? resident_half_units(TI, TJ) : TI + resident_extra_units(TI, unit_w);
        extra_per_b = units - (halves ? TJ : TI);
        total = (long long)B * units;
    }
};

bool gram_resident_takes_knorm(int H, int d) {
    // eight 16-byte pieces per row, or sixteen and more (the lane layouts of the stand-alone kernel that sixteen lanes a token
    // reproduce), a copy's box of at most 256 elements a side, and at least one chunk of eight tokens must fit the operand buffers
    if (H <= 0 || H > 256 || d % 8 || d > 256 || (d != 64 && d < 128)) return false;
    return knorm_buffers(H, d) > 0;
}

// All of them where the copies are double buffered, for samples of more than one row tile: one kernel less, and with all of them the
// selection follows within the labels' kernel.  Two and a half chunks of eight tokens to a CTA in the sweep and the other samples
// beside vic_finalize_kernel / all in the sweep, us: 1 x 300 tokens x 32 heads of 128 28.7 / 26.8, 7 x 700 x 32 of 128 47.1 / 44.0, 16 x 576 x
// 32 of 128 66.9 / 57.5 (8 chunks), 16 x 576 x 4 of 64 50.1 / 47.4, 32 x 576 x 32 of 128 119.1 / 101.8 (16 chunks), 148 x 256 x 32 of 128
// 226.2 / 208.9 (32).  Short chunks are held up by their waits: above 24 of them rows of 2 KB at least (140 x 256 x 4 of 64 91.6 / 94.8
// with 30, 120 x 256 x 8 of 128 101.3 / 92.2 with 26).
// Not where a CTA has many keys and all of them together are few: short samples have few CTAs for them (129 to 192 tokens four), and below
// 16 MB the other kernel ends beside vic_finalize_kernel.  A chunk takes a time of its own and one for each piece of 16 lanes, so
// pieces are counted: beyond 170 to a CTA calls one behind the other are 1.5 % faster in two parts (112 of 520 problems of 129 to 640 tokens,
// B 1 to 16; 1 x 182 x 32 of 128 with 768 features 27.9 / 28.9, 8 x 182 x 32 of 128 29.6 / 31.0, 1 x 256 x 48 of 128 27.6 / 30.6), the others
// 4.4 % less with all.  (With the L2 flushed in front all of them is the faster form on either side, by 5 %: the line is drawn for calls that
// follow the layer that wrote their keys.)
// Samples of one row tile have one CTA each, whose sweep ends when its keys do: three chunks (1 x 64 x 32 of 128 26.8 / 30.8 with all
// 8, 64 x 64 x 16 of 128 43.5 / 44.9; more only pays where they fill the chip, 100 x 128 x 32 of 128 108.6 / 100.3).  With a single buffer
// each chunk waits for the one before (48 heads of 256: 2 x 576 35.0 / 36.0, 16 x 200 63.6 / 70.8): two and a half chunks to a CTA.
int gram_resident_knorm_samples(int B, int n, int H, int d, int Nv) {
    const long long ctas = resident_ctas(ResidentCut(B, n).total), chunks = (Nv + kKnChunkTokens - 1) / kKnChunkTokens;
    const long long share = 5 * ctas / (2 * chunks);
    const bool few = 2.0 * B * Nv * H * d < 16e6 && chunks * B * H * ((d + 127) / 128) > 170 * ctas;
    const bool all = n > BM && !few ? chunks * B <= 24 * ctas || H * d >= 1024 : chunks * B <= 3 * ctas;
    return share >= B || (knorm_buffers(H, d) > 1 && all) ? B : (int)share;
}

int launch_gram_resident(const void* feat, const GramArgs& args, const GramTiling& tiling, cudaStream_t stream) {
    KernelArgs k;
    k.g = args;
    k.t = tiling;
    k.g.row0 = 0;
    k.g.row_end = args.n;
    const ResidentCut cut(args.B, args.n);
    const bool halves = cut.halves;
    k.unit_w = cut.unit_w;
    k.extra_units_per_b = cut.extra_per_b;
    k.total_tiles = cut.total;
    k.wait_ns = g_wait_ns.load();
    k.expire_roles = g_expire_roles.load() & 7;
    k.reports = 0;
    if (k.total_tiles <= 0) return VITCOP_OK;
    if (k.total_tiles > (long long)kResidentUnits * num_sms()) return VITCOP_ERR_INVALID_ARG;
    CUtensorMap ma, mb, mk = {};
    if (!make_feat_map(&ma, feat, args.B, args.n, args.D, BM) ||
        !make_feat_map(&mb, feat, args.B, args.n, args.D, halves ? 64 : BM * k.unit_w))
        return VITCOP_ERR_CUDA;
    if (args.kn_K && !make_keys_map(&mk, args.kn_K, args.kn_B, args.kn_H, args.kn_N, args.kn_d, kKnChunkTokens, args.kn_H)) return VITCOP_ERR_CUDA;
    const bool euclid = args.metric == 1;
    const bool spatial = args.tau2 >= 0.f && args.pos != nullptr;
    if (halves) {
        if (spatial)
            return euclid ? launch_resident_one<1, true, 64>(ma, mb, mk, k, stream) : launch_resident_one<0, true, 64>(ma, mb, mk, k, stream);
        return euclid ? launch_resident_one<1, false, 64>(ma, mb, mk, k, stream) : launch_resident_one<0, false, 64>(ma, mb, mk, k, stream);
    }
    if (spatial)
        return euclid ? launch_resident_one<1, true, BM>(ma, mb, mk, k, stream) : launch_resident_one<0, true, BM>(ma, mb, mk, k, stream);
    return euclid ? launch_resident_one<1, false, BM>(ma, mb, mk, k, stream) : launch_resident_one<0, false, BM>(ma, mb, mk, k, stream);
}

}  // namespace vitcop
