// Shared host/device helpers of the HSD library: status handling, integer types, launch checks.
#pragma once
#include <cuda_runtime.h>
#include <cuda_bf16.h>
#include <stdint.h>
#include <atomic>
#include "../../include/hsd.h"

typedef unsigned long long u64;
typedef unsigned int u32;

#define HSD_CUDA_OK(expr)                         \
  do {                                            \
    cudaError_t e__ = (expr);                     \
    if (e__ != cudaSuccess) return HSD_E_CUDA;    \
  } while (0)

// Kernel launches issued by this library (reported by hsd_kernel_launches()).
extern unsigned long long g_hsd_launches;
static inline void hsd_count_launches(int n) { g_hsd_launches += (unsigned long long)n; }

static inline int hsd_launch_status() {
  return cudaGetLastError() == cudaSuccess ? HSD_OK : HSD_E_CUDA;
}

// Raises a kernel's dynamic shared memory limit, once per device (the limit belongs to the current device; `done`: a bit
// per device, one word per kernel).
static inline int hsd_smem_limit(const void *kernel, int bytes, std::atomic<u64> &done) {
  int dev = 0;
  HSD_CUDA_OK(cudaGetDevice(&dev));
  const u64 bit = 1ull << (dev & 63);
  if (dev < 64 && (done.load(std::memory_order_relaxed) & bit)) return HSD_OK;
  HSD_CUDA_OK(cudaFuncSetAttribute(kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, bytes));
  if (dev < 64) done.fetch_or(bit, std::memory_order_relaxed);
  return HSD_OK;
}

// A chain of kernels on one stream, each of which may start (and prepare: barriers, tensor memory, the first weights) while
// the one before it still runs.  Every CTA of such a kernel calls chain_wait() before it touches anything the kernels
// before it read or wrote: it returns when the one before is complete, which had waited in the same way.  chain_next()
// lets the next kernel's CTAs come as SMs become free.  The first kernel of a public call may itself start early, behind
// whatever is on the stream; after a launch of the ordinary kind both do nothing.  A kernel whose successor reads inputs of the
// call ahead of its own wait calls chain_next() behind its chain_wait().
__device__ __forceinline__ void chain_wait() { asm volatile("griddepcontrol.wait;" ::: "memory"); }
__device__ __forceinline__ void chain_next() { asm volatile("griddepcontrol.launch_dependents;" ::: "memory"); }
template <class... KA, class... A>
static inline cudaError_t hsd_launch(void (*kernel)(KA...), dim3 grid, int threads, size_t smem, cudaStream_t s, int cluster, bool chained, A &&...args) {
  cudaLaunchConfig_t cfg = {};
  cfg.gridDim = grid; cfg.blockDim = dim3(threads); cfg.dynamicSmemBytes = smem; cfg.stream = s;
  cudaLaunchAttribute at[2];
  int n = 0;
  if (cluster > 0) {
    at[n].id = cudaLaunchAttributeClusterDimension;
    at[n].val.clusterDim.x = cluster; at[n].val.clusterDim.y = 1; at[n].val.clusterDim.z = 1;
    ++n;
  }
  if (chained) {
    at[n].id = cudaLaunchAttributeProgrammaticStreamSerialization;
    at[n].val.programmaticStreamSerializationAllowed = 1;
    ++n;
  }
  cfg.attrs = at; cfg.numAttrs = n;
  return cudaLaunchKernelEx(&cfg, kernel, static_cast<KA>(args)...);
}

// SMs of the GPU that measured lines (path choices, unit sizes) refer to; launches ask the device.
constexpr int kMeasuredSMs = 148;

__host__ __device__ static inline int ceil_div(int a, int b) { return (a + b - 1) / b; }

// Stored value -> fp32 (bf16 widens exactly).
__device__ __forceinline__ float to_f32(float v) { return v; }
__device__ __forceinline__ float to_f32(__nv_bfloat16 v) { return __bfloat162float(v); }

// Row lists of one forward pass: in device memory, or (few rows) in the kernel's own parameters, which saves a small pass
// the upload in front of it (1.5 us, and 5 us until the kernel behind it starts).
constexpr int kRowBlob = 1536;
struct PassRows {
  const int *row_seq, *row_pos, *lrow_src;   // sequence and position of each row; packed row of each logits row
  const int4 *attn;                          // work items: (first packed row, rows, sequence, position of first row)
  const long long *lrow_dst;                 // destination row in the level's logits buffer
  int in_blob, o_pos, o_attn, o_src, o_dst;  // 1: the lists lie in `blob` (row_seq in front), not at the pointers
  __align__(16) unsigned char blob[kRowBlob];
  __device__ __forceinline__ const int *seq() const { return in_blob ? reinterpret_cast<const int *>(blob) : row_seq; }
  __device__ __forceinline__ const int *pos() const { return in_blob ? reinterpret_cast<const int *>(blob + o_pos) : row_pos; }
  __device__ __forceinline__ const int *src() const { return in_blob ? reinterpret_cast<const int *>(blob + o_src) : lrow_src; }
  __device__ __forceinline__ int4 item(int i) const { return in_blob ? reinterpret_cast<const int4 *>(blob + o_attn)[i] : attn[i]; }
  __device__ __forceinline__ long long dst(int r) const { return in_blob ? reinterpret_cast<const long long *>(blob + o_dst)[r] : lrow_dst[r]; }
};
