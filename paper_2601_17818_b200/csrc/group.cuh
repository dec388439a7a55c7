// One sample worked on by R CTAs of 1024 threads, a thread-block cluster (R = 1: an ordinary CTA): which tokens are whose, and the
// way into the other CTAs' shared memory.
#pragma once

#include "async_copy.cuh"
#include "internal.cuh"

namespace vitcop {

constexpr int kGroupThreads = 1024;

// CTA `part` owns the tokens [part * share, (part + 1) * share) of n, thread t of it the tokens e * 1024 + t of these, e < E; shares
// are multiples of eight, so that 16-bit tables indexed by token split at 16-byte boundaries.
template <int R>
struct Share {
    int n, share, part, base;
    __device__ __forceinline__ explicit Share(int n_) : n(n_) {
        share = R == 1 ? (n + 7) & ~7 : ((n + R - 1) / R + 7) & ~7;
        part = R == 1 ? 0 : (int)cluster_ctarank();
        base = part * share;
    }
    __device__ __forceinline__ int own() const { return max(0, min(share, n - base)); }       // tokens of this CTA
};
// Tokens of a CTA, at most.
template <int R>
__host__ __device__ constexpr int share_capacity(int Nv_cap) { return R == 1 ? (Nv_cap + 7) & ~7 : ((Nv_cap + R - 1) / R + 7) & ~7; }

template <int R>
__device__ __forceinline__ void group_sync() {
    if (R == 1) __syncthreads();
    else cluster_sync_all();
}
// Shared memory of CTA `to`, by the address that it has in this CTA.
template <int R>
__device__ __forceinline__ uint32_t at_cta(const void* p, int to) {
    return R == 1 ? smem_u32(p) : cluster_map(smem_u32(p), (uint32_t)to);
}
__device__ __forceinline__ uint32_t ld_cluster(uint32_t a) {
    uint32_t v;
    asm volatile("ld.shared::cluster.u32 %0, [%1];" : "=r"(v) : "r"(a) : "memory");
    return v;
}
__device__ __forceinline__ unsigned long long ld_cluster64(uint32_t a) {
    unsigned long long v;
    asm volatile("ld.shared::cluster.u64 %0, [%1];" : "=l"(v) : "r"(a) : "memory");
    return v;
}
__device__ __forceinline__ uint32_t ld_cluster16(uint32_t a) {
    uint16_t v;
    asm volatile("ld.shared::cluster.u16 %0, [%1];" : "=h"(v) : "r"(a) : "memory");
    return v;
}
__device__ __forceinline__ void st_cluster16(uint32_t a, uint32_t v) {
    asm volatile("st.shared::cluster.u16 [%0], %1;" ::"r"(a), "h"((uint16_t)v) : "memory");
}
__device__ __forceinline__ void st_cluster4(uint32_t a, const uint4& v) {
    asm volatile("st.shared::cluster.v4.u32 [%0], {%1, %2, %3, %4};" ::"r"(a), "r"(v.x), "r"(v.y), "r"(v.z), "r"(v.w) : "memory");
}
__device__ __forceinline__ void min_cluster(uint32_t a, uint32_t v) { asm volatile("red.shared::cluster.min.u32 [%0], %1;" ::"r"(a), "r"(v) : "memory"); }
__device__ __forceinline__ void max_cluster(uint32_t a, uint32_t v) { asm volatile("red.shared::cluster.max.u32 [%0], %1;" ::"r"(a), "r"(v) : "memory"); }
__device__ __forceinline__ void or_cluster(uint32_t a, uint32_t v) { asm volatile("red.shared::cluster.or.b32 [%0], %1;" ::"r"(a), "r"(v) : "memory"); }

}  // namespace vitcop
