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

// SMs of the GPU that measured lines (path choices, unit sizes) refer to; launches ask the device.
constexpr int kMeasuredSMs = 148;

__host__ __device__ static inline int ceil_div(int a, int b) { return (a + b - 1) / b; }

// Stored value -> fp32 (bf16 widens exactly).
__device__ __forceinline__ float to_f32(float v) { return v; }
__device__ __forceinline__ float to_f32(__nv_bfloat16 v) { return __bfloat162float(v); }
