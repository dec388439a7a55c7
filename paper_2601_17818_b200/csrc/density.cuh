// What the density sweep (density.cu) leaves for the search of Eq. 3 (nearest.cu), and how it is laid out.
#pragma once

#include "gram.cuh"

namespace vitcop {

// The symmetric half of a sample's Gram matrix is cut into tiles of 256 x 256, numbered column-tile major: column tile tj
// holds the row tiles 0 .. tj and starts at tj (tj + 1) / 2.  The sweep keeps every Gram value it computes, in blocks of
// 32 x 32 pairs: block (rb, cb), rb <= cb, of a sample sits at gram_block_offset floats, its element (r, c) at
// gram_elem_offset inside it.
//
// Beside the values it leaves a summary of every block: for each of the block's 64 tokens the smallest squared distance to a
// token of the other side (blk_min).  Eq. 3 asks for the nearest DENSER token, and densities are known only when the sweep is
// over; but a block whose minimum is not below what a token has already found cannot hold its answer, so the search
// reads the minima and, of the Gram values, only the handful of blocks per token that it has to look into.
constexpr int kBlk = 32;                                   // tokens per side of a summarised block
constexpr int kSweepTile = 256;
constexpr int kSweepBlks = kSweepTile / kBlk;
struct SweepTiling {
    int T;             // 256-token tiles per sample
    int tiles_per_b;   // tiles of the symmetric half
    int TI;            // 128-token blocks
    int n_pad;         // TI * 128: tokens of one partial-sum slot
    __host__ __device__ int n_blk() const { return n_pad / kBlk; }     // blocks of 32 tokens
    // rho partial slots of a token: slot k holds the sum over the tokens of 128-token block k (later blocks from the row side of
    // the tiles, earlier ones from the column side), slot TI the column side of the token's own block
    __host__ __device__ int slots() const { return TI + 1; }
};
inline SweepTiling make_sweep_tiling(int n) {
    SweepTiling t;
    t.T = (n + kSweepTile - 1) / kSweepTile;
    t.tiles_per_b = t.T * (t.T + 1) / 2;
    t.TI = (n + kGramBM - 1) / kGramBM;
    t.n_pad = t.TI * kGramBM;
    return t;
}
constexpr size_t kSweepTileFloats = (size_t)kSweepTile * kSweepTile;
__host__ __device__ inline size_t gram_block_offset(int rb, int cb) {
    const int tp = rb / kSweepBlks, tj = cb / kSweepBlks;
    return (size_t)(tj * (tj + 1) / 2 + tp) * kSweepTileFloats +
           (size_t)((rb % kSweepBlks) * kSweepBlks + cb % kSweepBlks) * (kBlk * kBlk);
}
// Groups of four columns, inside a group row by row: the 32 threads of a warp, one row each, store 512 contiguous bytes per
// instruction.
__host__ __device__ inline int gram_elem_offset(int r, int c) { return ((c >> 2) * kBlk + r) * 4 + (c & 3); }

// What the sweep and the search keep of a group of samples: count and list of the search's leftovers, the tokens as the search
// reads them, block densities, block minima, Gram values (4 bytes per pair of the symmetric half, tile padding included).  They
// run group by group, so that the workspace stays bounded whatever the batch.
struct SweepGroupWs {
    size_t off_left, off_tok, off_blk_rho, off_blk_min, off_gram, total;
    SweepGroupWs(size_t samples, int n) {
        const SweepTiling s = make_sweep_tiling(n);
        size_t o = 0;
        off_left = o;    o += align_up((samples * n + 1) * 4, 256);
        off_tok = o;     o += align_up(samples * s.n_pad * sizeof(float4), 256);
        off_blk_rho = o; o += align_up(samples * s.n_blk() * 4, 256);
        off_blk_min = o; o += align_up(samples * s.n_blk() * s.n_pad * 4, 256);
        off_gram = o;    o += align_up(samples * s.tiles_per_b * kSweepTileFloats * 4, 256);
        total = o;
    }
};
constexpr size_t kSweepGroupBytes = (size_t)3 << 29;      // 1.5 GB: two samples of 16384 tokens take 1.2 GB
// Samples of a group where it may take `bytes`; 0 if one is too much.
inline int sweep_group_samples(int B, int n, size_t bytes) {
    const size_t per = SweepGroupWs(1, n).total;           // (never less than a sample adds)
    size_t g = bytes / per < (size_t)B ? bytes / per : (size_t)B;
    while (g < (size_t)B && SweepGroupWs(g + 1, n).total <= bytes) ++g;
    return (int)g;
}

struct SweepArgs {
    int B, n, D;
    float c2;                   // -(log2 e) / d_c^2
    float tau2;                 // tau^2; < 0: no spatial test
    const float* w;             // [B, n] per-token factors of the distance, as in GramArgs
    const float* a;
    float* rho;                 // [B, n]
    const float* pos;           // [B, n, 2] or nullptr
    const float4* bbox;         // [B, TI] bounding boxes of the 128-token blocks' positions, or nullptr
    float* part;                // [B, slots, n_pad] rho partials
    float* gram;                // [B, tiles_per_b, 256 x 256] Gram values
    float* blk_min;             // [B, n_pad, n_blk]: entry (t, k) = smallest d^2 between token t and the other tokens of
                                // block k (32 k ..), +inf where the blocks lie beyond the spatial radius
    float4* tok;                // [B, n_pad] what a pair needs of a token: (w or, for euclid, a; rho; position).  Tokens past
                                // the sample's last one, to the end of its block of 32, have density 0
    uint32_t* blk_rho;          // [B, n_blk] bits of the largest density in a block of 32 tokens
    int32_t* left;              // tokens (b n + i) that one warp's share of the search did not settle, and their number
    int32_t* n_left;
    unsigned long long* best;   // [B, n] packed (d^2 bits << 32 | index) of the nearest denser token, ~0 = none
    int* status;                // device status word
    int diag_reports;           // CTAs of the diagonal in front that reported whether they gave up, 0: they set the word themselves
    SweepTiling t;
    KnormJob kn;                // K-norm that the sweep computes on the side (kn.K null: none); d = 64 or 128
};

// Eq. 3 only pairs tokens within the spatial radius, so blocks of 128 x 128 pairs whose row tokens all lie farther than the
// radius from the column tokens cannot contribute: the density sweep need not keep them and the search never looks into
// them.  The distance between the bounding boxes is taken with the operations of the per-pair test (fp32 differences,
// squares joined by one fma), all of them monotone, so it never exceeds the distance of any pair: what is skipped is
// exactly what the per-pair test would have rejected.
__device__ __forceinline__ bool blocks_outside_radius(const float4& r, const float4& c, float tau2) {
    const float dx = fmaxf(0.f, fmaxf(r.x - c.z, c.x - r.z));
    const float dy = fmaxf(0.f, fmaxf(r.y - c.w, c.y - r.w));
    return fmaf(dx, dx, dy * dy) > tau2;
}

// How many leading samples' K-norm a sweep over `samples` samples of n tokens should compute on the side.
int sweep_knorm_samples(const KnormJob& job, int samples, int n, int D, int metric);

// Eq. 2: rho partials, Gram values and block minima (metric: 0 cosine, 1 euclid).
int launch_density_sweep(const void* feat, const SweepArgs& args, int metric, cudaStream_t stream, bool pdl);

// Eq. 3 from what the sweep left and the densities: args.best of every token.
int launch_nearest_denser(const SweepArgs& args, int metric, cudaStream_t stream, bool pdl);

}  // namespace vitcop
