// Internal declarations shared by the translation units of libvitcop (not part of the public ABI).
#pragma once

#include <cuda_runtime.h>
#include <stdint.h>

#include <atomic>

#include "vitcop.h"

namespace vitcop {

// Device status word lives in the first 256 bytes of every workspace.
constexpr size_t kStatusBytes = 256;
// A kernel that nothing of its call precedes finds the status word as the last call left it, and none of its CTAs can clear it for
// the others.  Its CTAs report in a byte each whether they gave up, and a later kernel of the call sets the word.  (A memset
// in front of the first kernel is 1.2 us of its own and another 1.5 until the kernel behind it starts.)
constexpr int kReportsAt = 64, kMaxReports = (int)kStatusBytes - kReportsAt;

inline size_t align_up(size_t x, size_t a) { return (x + a - 1) / a * a; }

// Records the first failing CUDA runtime error of the calling thread.
int record_cuda(cudaError_t e);

// What the launchers remember is remembered per device: one process may drive several.
constexpr int kMaxDevices = 64;
inline int current_device() {
    int dev = 0;
    return (cudaGetDevice(&dev) == cudaSuccess && dev >= 0 && dev < kMaxDevices) ? dev : 0;
}

// Raises a kernel's dynamic shared-memory limit once per device: to the most the kernel is ever launched with, because another
// thread may launch it between this call and the launch behind it.
typedef std::atomic<unsigned long long> DoneOnDevice;      // a bit per device
template <typename Kernel>
inline int allow_dynamic_smem(Kernel kern, size_t most_bytes, DoneOnDevice& done) {
    const unsigned long long bit = 1ull << current_device();
    if (done.load(std::memory_order_relaxed) & bit) return VITCOP_OK;
    const cudaError_t e = cudaFuncSetAttribute(kern, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)most_bytes);
    if (e != cudaSuccess) return record_cuda(e);
    done.fetch_or(bit, std::memory_order_relaxed);
    return VITCOP_OK;
}

// How many clusters of R CTAs (an SM each) the device runs of a kernel at a time: not SMs / R, because a cluster stays inside a group of
// SMs.  0 if it cannot be told.  `known`: number + 1, per device; `allow` raises the kernel's limit of dynamic shared memory.
typedef std::atomic<int> KnownOnDevice[kMaxDevices];
template <typename Kernel, typename Allow>
inline int clusters_at_once(Kernel kern, int R, int threads, size_t smem, Allow allow, KnownOnDevice& known) {
    std::atomic<int>& k = known[current_device()];
    int v = k.load(std::memory_order_relaxed);
    if (v == 0) {
        cudaLaunchConfig_t cfg = {};
        cfg.gridDim = dim3((unsigned)R);
        cfg.blockDim = dim3((unsigned)threads);
        cfg.dynamicSmemBytes = smem;
        cudaLaunchAttribute attr[1];
        attr[0].id = cudaLaunchAttributeClusterDimension;
        attr[0].val.clusterDim.x = (unsigned)R;
        attr[0].val.clusterDim.y = attr[0].val.clusterDim.z = 1;
        cfg.attrs = attr;
        cfg.numAttrs = 1;
        int n = 0;
        if (allow() != VITCOP_OK || cudaOccupancyMaxActiveClusters(&n, kern, &cfg) != cudaSuccess || n < 0) {
            cudaGetLastError();
            n = 0;
        }
        v = n + 1;
        k.store(v, std::memory_order_relaxed);
    }
    return v - 1;
}

// Diagnostic per-kernel timing (vitcop_kernel_timing_begin / _end).  While it is on, a KernelTimeScope
// around a launch records one CUDA event before and one after the kernel on its stream, and launchers
// drop the programmatic-dependent-launch attribute so that consecutive kernels do not overlap.
bool kernel_timing_on();
struct KernelTimeScope {
    KernelTimeScope(const char* name, cudaStream_t stream);
    ~KernelTimeScope();
    KernelTimeScope(const KernelTimeScope&) = delete;
    KernelTimeScope& operator=(const KernelTimeScope&) = delete;
private:
    int slot_;
    cudaStream_t stream_;
};
inline bool pdl_allowed(bool requested) { return requested && !kernel_timing_on(); }

// ---- launchers (enqueue on `stream`, return VITCOP_OK or VITCOP_ERR_CUDA) -------------------------
int launch_knorm(const void* K, int B, int H, int d, int64_t stride_b, int64_t stride_h, int64_t stride_n,
                 int vis_start, const int32_t* vis_len, int vis_len_uniform, float* score, int Nv_cap,
                 cudaStream_t stream, bool late_wait = false, bool* launched = nullptr, int* clear_status = nullptr);
// (`launched`, when given, tells whether a kernel was enqueued at all: an empty span needs none.  `clear_status`: a status
// word that the kernel sets to VITCOP_OK.)

// K-norm to be enqueued in the middle of the filter's kernel chain (vitcop_collaborative_step): it does not depend
// on the filter, so it runs beside the filter's sweep.
struct KnormJob {
    const void* K;
    int B, H, N, d, vis_start, Nv;
    float* score;
};

// Cluster-quota selection to follow the labels in the same kernel where the scores are there by then (`taken`).
struct QuotaJob {
    const float* score;                                    // [B, Nv]
    int budget;
    int32_t *keep, *n_keep;                                // [B, Nv], [B]
    bool taken;
};

int launch_select(const float* score, const int32_t* label, int B, const int32_t* vis_len, int vis_len_uniform,
                  int Nv_cap, int mode, int largest, int budget, int32_t* keep_idx, int keep_stride,
                  int32_t* n_keep, uint8_t* keep_mask, int* status_word, cudaStream_t stream, bool pdl,
                  int* clear_status = nullptr);
// (`clear_status`: plain mode sets this status word to VITCOP_OK on the way, in place of a memset in front of the kernel.)

// Plain selection (smallest scores) inside the copy, in place of a list; where compact_selects says that this is the faster way.
struct SmallestJob {
    const float* score;                                    // [B, keep_stride]
    int budget;
    int32_t *keep, *n_keep;                                // the list, written: [B, keep_stride], [B]
};
bool compact_selects(bool hidden, bool V, int B, int H, int d, int Dh, int Nv_cap, int Ncap);

int launch_compact(const void* hidden, const void* K, const void* V, int B, int H, int N, int d, int Dh,
                   const int32_t* seq_len, int vis_start, const int32_t* vis_len, int vis_len_uniform,
                   const int32_t* keep_idx, int keep_stride, const int32_t* n_keep, void* hidden_out, void* K_out,
                   void* V_out, int Ncap, int32_t* kept_pos, int32_t* out_len, cudaStream_t stream, bool early,
                   const SmallestJob* smallest = nullptr);
// (`early`: the tensors are inputs of a whole call whose first kernel has waited for everything queued before it, so rows that
// do not depend on the selection may be copied while the kernels in front are still running.)

size_t filter_workspace_bytes(int B, int n, int D);
// The least that launch_filter takes: with less than filter_workspace_bytes the samples go through in smaller groups.
size_t filter_workspace_least_bytes(int B, int n);
size_t similarity_workspace_bytes(int B, int n, int D);
int launch_filter(const void* feat, const float* pos, int B, int n, int D, const vitcop_filter_params& p,
                  int n_centers, int32_t* label, int32_t* n_clusters, float* rho, float* delta2, int32_t* parent,
                  void* workspace, size_t workspace_bytes, cudaStream_t stream, const KnormJob* knorm = nullptr,
                  QuotaJob* quota = nullptr);
int launch_similarity_rows(const void* feat, int B, int n, int D, int metric, int row_begin, int row_end,
                           float* out, void* workspace, cudaStream_t stream);

int launch_merge(const void* hidden, int B, int N, int Dh, int vis_start, const int32_t* vis_len, int vis_len_uniform,
                 int Nv_cap, const int32_t* label, const uint8_t* keep_mask, void* merged_bf16, float* merged_f32,
                 int32_t* merged_label, int32_t* merged_count, int32_t* n_merged, int Mcap, void* workspace,
                 cudaStream_t stream);
size_t merge_workspace_bytes(int B, int Nv_cap, int Mcap);

size_t kproj_workspace_bytes(int B, int N, int H, int d);
int launch_kproj_knorm(const void* hidden, const void* W, int B, int N, int Dh, int H, int d, const float* cos_tab,
                       const float* sin_tab, const int32_t* position, int n_pos, void* K_out, int vis_start, int Nv,
                       float* score, void* workspace, cudaStream_t stream);

size_t saliency_workspace_bytes(int B, int H, int M);
int launch_cls_saliency(const void* q, const void* K, int B, int H, int M, int d, float scale, float* saliency,
                        float* cls_self, void* workspace, cudaStream_t stream);

// ---- small device helpers ---------------------------------------------------------------------------
#ifdef __CUDACC__
__device__ __forceinline__ float bf16lo(uint32_t u) { return __uint_as_float(u << 16); }
__device__ __forceinline__ float bf16hi(uint32_t u) { return __uint_as_float(u & 0xFFFF0000u); }

// Programmatic dependent launch: wait until the preceding kernel on the stream has completed
// (no-op when the kernel was not launched with the PDL attribute).
__device__ __forceinline__ void grid_dependency_wait() { asm volatile("griddepcontrol.wait;" ::: "memory"); }
__device__ __forceinline__ void grid_dependency_launch_dependents() {
    asm volatile("griddepcontrol.launch_dependents;" ::: "memory");
}

__device__ __forceinline__ void report_gave_up(int* status, bool gave_up) {
    reinterpret_cast<volatile uint8_t*>(status)[kReportsAt + blockIdx.x] = gave_up ? 1 : 0;
}
// Called by a warp, behind the kernel whose `ctas` CTAs reported.
__device__ __forceinline__ bool any_gave_up(const int* status, int ctas) {
    bool any = false;
    for (int c = threadIdx.x & 31; c < ctas; c += 32)
        any |= reinterpret_cast<const volatile uint8_t*>(status)[kReportsAt + c] != 0;
    return __any_sync(0xffffffffu, any);
}

// Exclusive prefix count of `flag` over a CTA of 1024 threads, in thread order; `total` receives the CTA-wide
// count.  Must be called by all threads.  warp_sums: shared uint32_t[32].
__device__ __forceinline__ uint32_t block_prefix_count(bool flag, uint32_t* warp_sums, uint32_t& total) {
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    const uint32_t bal = __ballot_sync(0xffffffffu, flag);
    const uint32_t before = __popc(bal & ((1u << lane) - 1u));
    if (lane == 0) warp_sums[warp] = __popc(bal);
    __syncthreads();
    uint32_t v = warp_sums[lane];
#pragma unroll
    for (int off = 1; off < 32; off <<= 1) {
        const uint32_t t = __shfl_up_sync(0xffffffffu, v, off);
        if (lane >= off) v += t;
    }
    total = __shfl_sync(0xffffffffu, v, 31);
    const uint32_t base = __shfl_sync(0xffffffffu, v, (warp + 31) & 31);
    __syncthreads();
    return (warp == 0 ? 0u : base) + before;
}

// Exclusive prefix sum of one value per thread over a CTA of 1024 threads, in thread order; `total` receives the CTA-wide sum.
__device__ __forceinline__ uint32_t block_exclusive_sum(uint32_t v, uint32_t* warp_sums, uint32_t& total) {
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    uint32_t incl = v;
#pragma unroll
    for (int off = 1; off < 32; off <<= 1) {
        const uint32_t t = __shfl_up_sync(0xffffffffu, incl, off);
        if (lane >= off) incl += t;
    }
    if (lane == 31) warp_sums[warp] = incl;
    __syncthreads();
    uint32_t w = warp_sums[lane];
#pragma unroll
    for (int off = 1; off < 32; off <<= 1) {
        const uint32_t t = __shfl_up_sync(0xffffffffu, w, off);
        if (lane >= off) w += t;
    }
    total = __shfl_sync(0xffffffffu, w, 31);
    const uint32_t base = warp == 0 ? 0u : __shfl_sync(0xffffffffu, w, warp - 1);
    __syncthreads();
    return base + incl - v;
}

// Exclusive prefix of one value per warp (uniform inside the warp) over the 32 warps of a CTA of 1024 threads; `total` = the sum.
__device__ __forceinline__ uint32_t warp_totals_scan(uint32_t warp_total, uint32_t* warp_sums, uint32_t& total) {
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    if (lane == 0) warp_sums[warp] = warp_total;
    __syncthreads();
    uint32_t v = warp_sums[lane];
#pragma unroll
    for (int off = 1; off < 32; off <<= 1) {
        const uint32_t t = __shfl_up_sync(0xffffffffu, v, off);
        if (lane >= off) v += t;
    }
    total = __shfl_sync(0xffffffffu, v, 31);
    const uint32_t base = __shfl_sync(0xffffffffu, v, (warp + 31) & 31);
    __syncthreads();
    return warp == 0 ? 0u : base;
}

#endif

}  // namespace vitcop
