// Centres, forest roots and labels of one sample (Algorithm 2, steps 3-4) by a group of R CTAs (group.cuh): the device routine of
// vic_finalize_kernel and of the kernel that goes on with the selection (filter.cu).
//
// The CTAs have their SMs to themselves, so what counts is the number of dependent steps, not throughput: every thread holds its
// tokens' keys in registers, all global loads are in flight together, the cut among the keys is found with one or two histogram passes
// of 10 or 11 bits that start at the highest bit in which two keys differ (each CTA counts its own tokens, all add up all counts), and
// what is left in the cut's bin is ranked by counting.  Every CTA then has the whole table of parents (two bytes a token) and follows
// its own tokens' chains to the root in it; after kChase steps the CTAs tell one another how far they came.
#pragma once

#include "group.cuh"

namespace vitcop {

// One CTA takes 11 bits a pass; of several each reads all counts, 4 KB a CTA at 10 bits (1.8 us of a pass with eight CTAs at 11, 0.9 so).
template <int R>
constexpr int kVicBits = R == 1 ? 11 : 10;
template <int R>
constexpr int kVicBinsPer = (1 << kVicBits<R>) / kGroupThreads;              // of a thread
constexpr int kVicRank = 256;                              // bins of up to this many keys are ranked by counting
constexpr uint32_t kVicIndex = VITCOP_MAX_VISUAL_TOKENS - 1, kVicCentre = 0x8000u;         // an entry of the table: parent; the token is a centre
// Steps of a round and rounds of the chase.  Tokens d steps from their root need one round below 64, two below 4033, four at the 16383 of the
// longest sample.  The rest is the limit: parents are denser than their children and form no cycle, but behind a sweep that gave up they
// are whatever the workspace held (two negative densities one step apart are each other's), and then too the kernel has to end.
constexpr int kChase = 64, kChaseRounds = 8;
static_assert((kVicIndex & (kVicIndex + 1)) == 0 && kVicIndex < kVicCentre, "indices and the mark of a centre share 16 bits");

struct VicArgs {
    const uint16_t* feat;
    int n, D, nc;
    const float* rho;
    const unsigned long long* best;
    const float *w, *a;
    int32_t *label, *n_clusters;
    float* delta2_user;
    int32_t* parent_user;
};

// Dynamic shared memory: table uint16 [R * share], won uint8 [share], centre list uint16 [nc] (surplus orphans).
template <int R>
__host__ __device__ constexpr size_t vic_smem(int n, int nc) {
    return (size_t)R * share_capacity<R>(n) * 2 + (size_t)share_capacity<R>(n) + (size_t)(nc > 0 ? nc : 1) * 2 + 16;
}

template <int R>
struct VicShared {
    uint32_t hist[2][kVicBinsPer<R> * kGroupThreads];      // by turns
    unsigned long long orph_best[kGroupThreads];           // surplus orphans: what they have found, and their list
    int orph_list[kGroupThreads];
    unsigned long long cand_key[kVicRank], all_key[R == 1 ? 1 : kVicRank];
    uint16_t cand_idx[kVicRank], all_idx[R == 1 ? 1 : kVicRank];
    uint32_t warp_sums[32];
    uint32_t lo, hi, digit, krem, count, cands;
    uint32_t flags[kChaseRounds];                          // per round of the chase: 1 a chain goes on, 2 a root is no centre
    int orph_cnt, centre_cnt;

    // All CTAs, before any of them calls vic_labels.
    __device__ __forceinline__ void init() {
        const int tid = threadIdx.x;
        for (int k = tid; k < 2 * kVicBinsPer<R> * kGroupThreads; k += kGroupThreads) hist[0][k] = 0u;
        if (tid < kChaseRounds) flags[tid] = 0u;
        if (tid == 0) { lo = 0xFFFFFFFFu; hi = 0u; cands = 0u; centre_cnt = 0; }
        group_sync<R>();
    }
};

// The labels of this thread's tokens, written to v.label too.
template <int R, int E>
__device__ __forceinline__ void vic_labels(const VicArgs& v, int b, VicShared<R>& sh, uint8_t* dyn, int (&lab)[E]) {
    const int tid = threadIdx.x, lane = tid & 31, n = v.n, nc = v.nc;
    const Share<R> s(n);
    const int own = s.own();
    uint16_t* const table = reinterpret_cast<uint16_t*>(dyn);
    uint8_t* const won = dyn + (size_t)R * s.share * 2;
    const size_t bo = (size_t)b * n;
    const float* const rho = v.rho + bo;
    const unsigned long long* const best = v.best + bo;

    // (Loads of what the preceding kernels wrote: pointers without __restrict__, so that nothing lets the compiler move one in
    // front of the wait.)
    // rank key, ascending = better centre candidate: ( ~( orphan ? 0xFFFFFFFF : gamma ), ~rho, index )
    uint32_t hi[E];
    uint16_t entry[E];                                     // of the table, but for the mark
    constexpr bool kHold = E <= 4;
    float r[kHold ? E : 1];
    auto rho_key = [&](int e) {
        if constexpr (kHold) return ~__float_as_uint(r[e]);
        else return ~__float_as_uint(__ldcg(rho + s.base + e * kGroupThreads + tid));
    };
    uint32_t in = 0, sel = 0, ranked = 0;                  // in: tokens (bit e) on the cut; sel: chosen ones
    {
        unsigned long long p[E];
        float x[E];
#pragma unroll
        for (int e = 0; e < E; ++e) {
            const int l = e * kGroupThreads + tid;
            p[e] = l < own ? __ldcg(best + s.base + l) : 0ull;
            x[e] = l < own ? __ldcg(rho + s.base + l) : 0.f;
        }
        uint32_t lo_k = 0xFFFFFFFFu, hi_k = 0u;
#pragma unroll
        for (int e = 0; e < E; ++e) {
            const int l = e * kGroupThreads + tid, i = s.base + l;
            if constexpr (kHold) r[e] = x[e];
            hi[e] = 0u;
            entry[e] = 0;
            if (l < own) {
                in |= 1u << e;
                const bool orphan = p[e] == ~0ull;
                const float d2 = orphan ? __int_as_float(0x7f800000) : __uint_as_float((uint32_t)(p[e] >> 32));
                const int par = orphan ? -1 : (int)(uint32_t)(p[e] & 0xFFFFFFFFull);
                if (v.delta2_user) v.delta2_user[bo + i] = d2;
                if (v.parent_user) v.parent_user[bo + i] = par;
                entry[e] = (uint16_t)((par < 0 || par >= n) ? i : par);
                hi[e] = ~(orphan ? 0xFFFFFFFFu : __float_as_uint(x[e] * sqrtf(d2)));
                lo_k = min(lo_k, hi[e]);
                hi_k = max(hi_k, hi[e]);
            }
        }
        lo_k = __reduce_min_sync(0xffffffffu, lo_k);
        hi_k = __reduce_max_sync(0xffffffffu, hi_k);
        if (lane < R && lo_k <= hi_k) {
            min_cluster(at_cta<R>(&sh.lo, lane), lo_k);
            max_cluster(at_cta<R>(&sh.hi, lane), hi_k);
        }
    }
    group_sync<R>();

    // ---- the nc smallest keys
    if (nc >= n) {
        sel = in;
    } else if (nc > 0) {
        uint32_t krem = (uint32_t)nc;
        int word = 0, top = 32 - __clz(sh.lo ^ sh.hi);     // word of the key, bits of it not yet looked at
        for (int pass = 0;; ++pass) {
            while (top == 0) top = ++word == 2 ? 14 : 32;  // (indices differ: the last word settles everything)
            const int shift = top > kVicBits<R> ? top - kVicBits<R> : 0;
            auto digit = [&](int e) {
                const uint32_t k = word == 0 ? hi[e] : word == 1 ? rho_key(e) : (uint32_t)(s.base + e * kGroupThreads + tid);
                return (k >> shift) & ((1u << (top - shift)) - 1u);
            };
            uint32_t* const hist = sh.hist[pass & 1];
#pragma unroll
            for (int e = 0; e < E; ++e)
                if (in >> e & 1u) atomicAdd(&hist[digit(e)], 1u);
            group_sync<R>();
            uint32_t h = 0, h1 = 0;
            uint32_t* const other = sh.hist[(pass & 1) ^ 1];               // (read by everyone: all CTAs have come here since)
            if constexpr (R == 1) {
                h = hist[2 * tid];
                h1 = hist[2 * tid + 1];
                other[2 * tid] = other[2 * tid + 1] = 0;
            } else {
#pragma unroll
                for (int u = 0; u < R; ++u) h += ld_cluster(at_cta<R>(hist + tid, u));
                other[tid] = 0;
            }
            uint32_t total;
            const uint32_t before = block_exclusive_sum(h + h1, sh.warp_sums, total);
            if (before < krem && krem <= before + h + h1) {
                const bool second = krem > before + h;
                sh.digit = kVicBinsPer<R> * tid + (second ? 1 : 0);
                sh.krem = krem - before - (second ? h : 0u);
                sh.count = second ? h1 : h;
            }
            __syncthreads();
            const uint32_t cut = sh.digit, count = sh.count;
            krem = sh.krem;
#pragma unroll
            for (int e = 0; e < E; ++e) {
                if (in >> e & 1u) {
                    const uint32_t d = digit(e);
                    if (d < cut) sel |= 1u << e;
                    if (d != cut) in &= ~(1u << e);
                }
            }
            top = shift;
            if (count == krem) {                           // the whole bin is wanted
                sel |= in;
                break;
            }
            if (count <= (uint32_t)kVicRank) {
                // few left: listed, and ranked below
#pragma unroll
                for (int e = 0; e < E; ++e) {
                    if (in >> e & 1u) {
                        const int l = e * kGroupThreads + tid;
                        const uint32_t at = atomicAdd(&sh.cands, 1u);
                        sh.cand_key[at] = ((unsigned long long)hi[e] << 32) | (unsigned long long)rho_key(e);
                        sh.cand_idx[at] = (uint16_t)(s.base + l);
                        won[l] = 0;
                    }
                }
                ranked = krem;
                break;
            }
            __syncthreads();                               // (digit .. are rewritten)
        }
    }
    if (ranked > 0) {                                      // (uniform over the CTAs)
        group_sync<R>();
        const unsigned long long* key = sh.cand_key;
        const uint16_t* idx_of = sh.cand_idx;
        int cands = (int)sh.cands;
        if (R > 1) {
            uint32_t c[R];
            cands = 0;
#pragma unroll
            for (int u = 0; u < R; ++u) c[u] = ld_cluster(at_cta<R>(&sh.cands, u));
            int from = 0, at = tid;
#pragma unroll
            for (int u = 0; u < R; ++u) {
                if (tid >= cands && tid < cands + (int)c[u]) {
                    from = u;
                    at = tid - cands;
                }
                cands += (int)c[u];
            }
            if (tid < cands) {
                sh.all_key[R == 1 ? 0 : tid] = ld_cluster64(at_cta<R>(sh.cand_key + at, from));
                sh.all_idx[R == 1 ? 0 : tid] = (uint16_t)ld_cluster16(at_cta<R>(sh.cand_idx + at, from));
            }
            key = sh.all_key;
            idx_of = sh.all_idx;
            __syncthreads();
        }
        // all candidates of this CTA at once, on a warp each or on as many lanes as there are for them (at least four)
        static_assert(kVicRank * 4 <= kGroupThreads, "four lanes a candidate");
        const int mine = (int)sh.cands;
        int log_lanes = 5;
        while (mine << log_lanes > kGroupThreads) --log_lanes;
        const int lanes = 1 << log_lanes, c = tid >> log_lanes, sub = tid & (lanes - 1);
        uint32_t better = 0;
        int idx = 0;
        if (c < mine) {
            const unsigned long long k = sh.cand_key[c];
            idx = sh.cand_idx[c];
            for (int o = sub; o < cands; o += lanes) {
                const unsigned long long x = key[o];
                better += (uint32_t)(x < k) | ((uint32_t)(x == k) & (uint32_t)(idx_of[o] < idx));
            }
        }
        for (int off = 1; off < lanes; off <<= 1) better += __shfl_xor_sync(0xffffffffu, better, off);
        if (c < mine && sub == 0 && better < ranked) won[idx - s.base] = 1;
        __syncthreads();
#pragma unroll
        for (int e = 0; e < E; ++e)
            if ((in >> e & 1u) && won[e * kGroupThreads + tid]) sel |= 1u << e;
    }
    // ---- the table: centres are roots, an orphan is one already
    auto tell_others = [&]() {                             // this CTA's part of the table (complete) to the others
        if constexpr (R > 1) {
#pragma unroll
            for (int u = 1; u < R; ++u) {
                const int to = (s.part + u) % R;
                for (int x = tid; x < s.share / 8; x += kGroupThreads)
                    st_cluster4(at_cta<R>(table + s.base + 8 * x, to), *reinterpret_cast<const uint4*>(table + s.base + 8 * x));
            }
        }
    };
#pragma unroll
    for (int e = 0; e < E; ++e) {
        const int l = e * kGroupThreads + tid, i = s.base + l;
        if (l < own) table[i] = (sel >> e & 1u) ? (uint16_t)(i | kVicCentre) : entry[e];
    }
    if (R > 1) __syncthreads();
    tell_others();
    group_sync<R>();
    // ---- roots: any value read is an ancestor, roots are fixed points
    uint32_t at[E];                                        // the root's entry
    uint32_t flags;
    if constexpr (R == 1) {                                // pointer jumping
        for (int round = 0; round < 16; ++round) {
            int changed = 0;
#pragma unroll
            for (int e = 0; e < E; ++e) {
                const int i = e * kGroupThreads + tid;
                if (i < n) {
                    uint32_t p = table[i] & kVicIndex;
                    const uint32_t q = table[p] & kVicIndex;
                    if (q != p) {
                        p = table[q] & kVicIndex;
                        table[i] = (uint16_t)(table[p] & kVicIndex);
                        changed = 1;
                    }
                }
            }
            if (!__syncthreads_or(changed)) break;
        }
        int surplus = 0;
#pragma unroll
        for (int e = 0; e < E; ++e) {
            const int i = e * kGroupThreads + tid;
            at[e] = i < n ? table[table[i] & kVicIndex] : 0u;
            if (i < n && !(at[e] & kVicCentre)) surplus = 1;
        }
        flags = __syncthreads_or(surplus) ? 2u : 0u;
    } else {
        // (the token's ancestor; at the end the root's entry)
#pragma unroll
        for (int e = 0; e < E; ++e) at[e] = (uint32_t)(s.base + e * kGroupThreads + tid);
        uint32_t open = 0, found = 0;
#pragma unroll
        for (int e = 0; e < E; ++e)
            if (e * kGroupThreads + tid < own) open |= 1u << e;
        for (int round = 0; round < kChaseRounds; ++round) {
#pragma unroll
            for (int e = 0; e < E; ++e) {
                if (!(open >> e & 1u)) continue;
                // (a warp goes on to the end of its longest chain: bound by instruction issue)
                uint32_t p = at[e], q = table[p];
                for (int step = 1; step < kChase && (q & kVicIndex) != p; ++step) {
                    p = q & kVicIndex;
                    q = table[p];
                }
                if ((q & kVicIndex) == p) {
                    open &= ~(1u << e);
                    found |= q & kVicCentre ? 0u : 2u;
                    p = q;
                }
                at[e] = p;
            }
            // (bits of the warp, to every CTA)
            const uint32_t say = __reduce_or_sync(0xffffffffu, (open ? 1u : 0u) | found);
            if (say && lane < R) or_cluster(at_cta<R>(&sh.flags[round], lane), say);
            group_sync<R>();
            flags = sh.flags[round];
            if (!(flags & 1u)) break;
            // chains go on: what was found so far goes into the tables (an ancestor in the place of another)
#pragma unroll
            for (int e = 0; e < E; ++e)
                if (open >> e & 1u) table[s.base + e * kGroupThreads + tid] = (uint16_t)at[e];
            __syncthreads();
            tell_others();
            group_sync<R>();
        }
        // (the limit: an ancestor stands in for the root, as above)
#pragma unroll
        for (int e = 0; e < E; ++e)
            if (open >> e & 1u) at[e] = table[at[e]];
    }
    // ---- a root that is an orphan but not a centre joins the nearest centre (feature distance)
    if ((flags & 2u) && nc > 0) {
        // Surplus orphans are rare but each needs its distance to every centre: every CTA lists its own, kGroupThreads tokens at a time,
        // and the (orphan, centre) pairs are spread over its warps; the nearest centre wins through a packed minimum
        // (distance bits, then the lower centre).
        uint16_t* const centres = reinterpret_cast<uint16_t*>(won + ((s.share + 1) & ~1));
        unsigned long long* const orph_best = sh.orph_best;
        int* const orph_list = sh.orph_list;
        const uint16_t* const feat = v.feat + (size_t)b * n * v.D;
        const float *const w = v.w + bo, *const a = v.a + bo;
        for (int i = tid; i < n; i += kGroupThreads)
            if (table[i] == (i | kVicCentre)) centres[atomicAdd(&sh.centre_cnt, 1)] = (uint16_t)i;
        for (int l0 = 0; l0 < own; l0 += kGroupThreads) {
            __syncthreads();                               // the previous round's list has been consumed
            if (tid == 0) sh.orph_cnt = 0;
            __syncthreads();
            const int o = s.base + l0 + tid;
            if (l0 + tid < own && table[o] == o) {
                const int k = atomicAdd(&sh.orph_cnt, 1);
                orph_list[k] = o;
                orph_best[k] = ~0ull;
            }
            __syncthreads();
            const int pairs = sh.orph_cnt * nc;
            for (int pr = tid >> 5; pr < pairs; pr += kGroupThreads / 32) {
                const int k = pr / nc, oo = orph_list[k], c = centres[pr - k * nc];
                const uint16_t* fo = feat + (size_t)oo * v.D;
                const uint16_t* fc = feat + (size_t)c * v.D;
                float dot = 0.f;
                for (int x = lane * 2; x < v.D; x += 64) {
                    const uint32_t f = *reinterpret_cast<const uint32_t*>(fo + x);
                    const uint32_t g = *reinterpret_cast<const uint32_t*>(fc + x);
                    dot = fmaf(bf16lo(f), bf16lo(g), dot);
                    dot = fmaf(bf16hi(f), bf16hi(g), dot);
                }
#pragma unroll
                for (int off = 16; off > 0; off >>= 1) dot += __shfl_xor_sync(0xffffffffu, dot, off);
                const float d2 = fmaxf(0.f, fmaf(-2.f, (dot * w[oo]) * w[c], a[oo] + a[c]));
                if (lane == 0) atomicMin(&orph_best[k], ((unsigned long long)__float_as_uint(d2) << 32) | (unsigned long long)(uint32_t)c);
            }
            __syncthreads();
            // the adopted centre, in every CTA's table (an entry that is not the token's own: another CTA may still be listing centres)
            if (tid < sh.orph_cnt) {
                const int o2 = orph_list[tid];
                const uint32_t c = (uint32_t)(orph_best[tid] & 0xFFFFFFFFull) | kVicCentre;
#pragma unroll
                for (int u = 0; u < R; ++u) st_cluster16(at_cta<R>(table + o2, u), c);
            }
        }
        group_sync<R>();
#pragma unroll
        for (int e = 0; e < E; ++e)
            if (e * kGroupThreads + tid < own && !(at[e] & kVicCentre)) at[e] = table[at[e]];
    }
    // ---- labels
#pragma unroll
    for (int e = 0; e < E; ++e) {
        lab[e] = (int)(at[e] & kVicIndex);
        if (e * kGroupThreads + tid < own) v.label[bo + s.base + e * kGroupThreads + tid] = lab[e];
    }
    if (s.part == 0 && tid == 0) v.n_clusters[b] = nc;
}

}  // namespace vitcop
