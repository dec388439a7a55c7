// Interface between the tensor-core kernels on the Gram matrix (gram.cu) and the rest of the redundancy filter (filter.cu).
#pragma once

#include "internal.cuh"

namespace vitcop {

constexpr int kGramBM = 128;   // rows of an output tile (UMMA M)

// GRAM_DIAG visits only the diagonal tiles and turns g_ii into the per-token factors w and a; GRAM_SIM writes rows of
// similarities.  GRAM_RHO and GRAM_DELTA are phases of the one-kernel sweep.
enum GramMode { GRAM_RHO = 0, GRAM_DELTA = 1, GRAM_SIM = 2, GRAM_DIAG = 3 };

// Tiling in row and column blocks of 128 tokens.
struct GramTiling {
    int TI, TJ;        // row blocks, column blocks per sample
    int tiles_per_b;   // tiles gram_tc_kernel visits per sample
    int n_pad;         // padded token count of one partial-sum slot
    __host__ __device__ int slots() const { return TJ + TI; }   // rho partial slots per sample: TJ row-side + TI column-side
};

inline GramTiling make_gram_tiling(int n) {
    GramTiling t;
    t.TI = t.TJ = (n + kGramBM - 1) / kGramBM;
    t.tiles_per_b = t.TI * t.TJ;
    t.n_pad = t.TI * kGramBM;
    return t;
}

// Bounded device waits of the Gram kernels: the time after which a wait gives up (0 = the default of 2 s) and, for
// failure-handling tests, the roles whose waits give up at once (1 load warp, 2 MMA warp, 4 epilogue warps; times 8: in the
// kernels on pairs of SMs alone).
// Applies to launches made after the call.
void gram_set_wait_debug(unsigned long long limit_ns, int expire_roles);
unsigned long long gram_wait_limit_ns();
int pair_expire_roles();                               // as the kernels on pairs of SMs take them

struct GramArgs {
    int B, n, D;
    int row0, row_end;          // GRAM_SIM: rows [row0, row_end) are produced
    int metric;                 // 0 cosine, 1 euclid
    float c2;                   // -(log2 e) / d_c^2
    float tau2;                 // tau^2; < 0: no spatial test
    const float* w;             // [B, n] factor multiplying the Gram value (cosine 1/|f|, euclid 1)
    const float* a;             // [B, n] additive term (cosine 1, euclid |f|^2):  d^2 = a_i + a_j - 2 g w_i w_j
    const float* rho;           // [B, n]                          (GRAM_DELTA)
    const float* pos;           // [B, n, 2] or nullptr            (GRAM_DELTA)
    float* part;                // [B, slots, n_pad] rho partials  (GRAM_RHO)
    unsigned long long* best;   // [B, n] packed (d2 bits << 32 | index), ~0 = none   (GRAM_DELTA)
    float* sim_out;             // [B, row_end - row0, n]          (GRAM_SIM)
    float* w_out;               // [B, n] factors written by GRAM_DIAG (best, if given, is reset to ~0 as well)
    float* a_out;               // [B, n]
    float* rho_out;             // [B, n] written by the resident sweep (same memory as rho)
    float* rho_user;            // [B, n] optional copy of rho for the caller
    unsigned int* grid_sync;    // counter of the resident sweep's grid-wide barrier (a word of the status block)
    uint32_t* ready;            // resident sweep [B, n]: a token's factor (w, or for euclid a) once it is known, as its bits + 1
                                // (both cleared by the kernel in front)
    // Optional K-norm (Eq. 4) for the resident sweep's warps beside the epilogue's to stream once the MMAs are done:
    // K bf16 [kn_B, kn_H, kn_N, kn_d] dense, span [kn_vis_start, kn_vis_start + kn_Nv), score [kn_B, kn_Nv].
    // Only shapes gram_resident_takes_knorm accepts.
    const void* kn_K;
    float* kn_score;
    int kn_B, kn_H, kn_N, kn_d, kn_vis_start, kn_Nv;
    float4* bbox;               // [B, ceil(n / 128)] bounding box (min x, min y, max x, max y) of every row block's
                                // positions, or nullptr: written by GRAM_DIAG
    int* status;                // device status word
    int reports;                // GRAM_DIAG: clear the status word; CTAs that give up report it (internal.cuh) to rho_reduce_kernel
};

// rho of token i of one sample from the partial sums of the tiles that hold it, in a fixed order (reproducible
// bits): the row-side slots ti .. TJ - 1 of the column blocks that pair its row block ti with later tokens, then the
// column-side slots TJ .. TJ + ti of the row blocks that pair it with earlier ones.  One contiguous walk, as long for every
// token, loaded sixteen at a time (independent loads: up to 1920 tokens one trip to L2).  `p` points at the sample's slot 0,
// token i.
__device__ __forceinline__ float rho_from_partials(const float* p, const GramTiling& t, int i) {
    const float* const q = p + (size_t)(i / kGramBM) * t.n_pad;
    const int entries = t.TJ + 1;
    float s = 0.f;
    for (int c = 0; c < entries; c += 16) {
        float v[16];
#pragma unroll
        for (int u = 0; u < 16; ++u) v[u] = c + u < entries ? q[(c + u) * t.n_pad] : 0.f;
#pragma unroll
        for (int u = 0; u < 16; ++u) s += v[u];            // (nothing is negative: adding 0 changes no bit)
    }
    return s;
}

// The same sum in the same order where the one-kernel sweep works on units of 64 columns (gram_resident_halves): per sample
// TI row-side slots of float4 {32-column sums of the tile}, then TI column-side slots.
__device__ inline float rho_from_half_partials(const float* part_b, const GramTiling& t, int n, int i) {
    const int ti = i / kGramBM;
    const float4* const row = reinterpret_cast<const float4*>(part_b) + i;
    const float* const col = part_b + (size_t)4 * t.TI * t.n_pad + i;
    constexpr int kCols = 8, kRows = 6;
    float cv[kCols];                                       // (travels with the first row-side entries)
#pragma unroll
    for (int u = 0; u < kCols; ++u) cv[u] = u <= ti ? col[(size_t)u * t.n_pad] : 0.f;
    float s = 0.f;
    for (int c = ti; c < t.TI; c += kRows) {
        float4 v[kRows];
#pragma unroll
        for (int u = 0; u < kRows; ++u) v[u] = c + u < t.TI ? row[(size_t)(c + u) * t.n_pad] : make_float4(0.f, 0.f, 0.f, 0.f);
#pragma unroll
        for (int u = 0; u < kRows; ++u) {
            if (c + u >= t.TI) continue;
            float x = v[u].x + v[u].y;
            if ((c + u) * kGramBM + kGramBM / 2 < n) x = (x + v[u].z) + v[u].w;        // (else there is no second unit)
            s += x;
        }
    }
#pragma unroll
    for (int u = 0; u < kCols; ++u)
        if (u <= ti) s += cv[u];
    for (int u = kCols; u <= ti; ++u) s += col[(size_t)u * t.n_pad];
    return s;
}

// True when the one-kernel sweep cuts the problem into units of 64 columns instead of 128 or 256 (gram.cu).
bool gram_resident_halves(int B, int n);

// True when the whole symmetric sweep of the problem fits the tensor memory of one wave of CTAs (at most two units
// of one row block against two column blocks per SM): density and delta can then share one pass over the Gram tiles
// (launch_gram_resident).
bool gram_fits_resident(int B, int n);

// True when the resident sweep can compute the K-norm of keys with H heads of d elements on the side.
bool gram_resident_takes_knorm(int H, int d);

// How many leading samples' K-norm (H heads of d elements, spans of Nv tokens) the resident sweep of [B, n] finishes without being
// held up.
int gram_resident_knorm_samples(int B, int n, int H, int d, int Nv);

// One kernel for the norms, Eq. 2 and Eq. 3 on small problems, behind one that has cleared grid_sync, ready and the status word: every CTA keeps the accumulators of its tiles in
// tensor memory; the diagonal tiles publish the per-token factors, which the density epilogues of the other tiles wait for
// value by value, the grid synchronises once (bounded waits) after the density
// partials; the delta epilogue sums the partials it needs itself and re-reads the same accumulators.
// `tiling` = make_gram_tiling(n).
int launch_gram_resident(const void* feat, const GramArgs& args, const GramTiling& tiling, cudaStream_t stream);

// Multiprocessors of the current device.
int gram_num_sms();

// Enqueues GRAM_DIAG or GRAM_SIM.
int launch_gram_sweep(int mode, const void* feat, const GramArgs& args, cudaStream_t stream, bool pdl);

}  // namespace vitcop
