// Dynamic shared-memory limit of a kernel, raised once per device: the attribute belongs to the device's context, so
// a process that works on several devices has to set it on each of them.
#pragma once

#include <cuda_runtime.h>

#include <atomic>

namespace coarse {

// The devices on which a kernel's limit is raised (one static object per kernel and launcher).
struct SmemLimit {
  std::atomic<unsigned long long> done{0};
};

// Raises `kernel`'s limit to `bytes` on the current device unless that was done before.  Safe from several threads:
// at worst two of them set the same value.
inline cudaError_t raise_smem_limit(SmemLimit& limit, const void* kernel, size_t bytes) {
  int dev = 0;
  const cudaError_t e = cudaGetDevice(&dev);
  if (e != cudaSuccess) return e;
  const unsigned long long bit = dev < 64 ? 1ull << dev : 0ull;  // device 64 on: set at every launch
  if (limit.done.load(std::memory_order_acquire) & bit) return cudaSuccess;
  const cudaError_t r = cudaFuncSetAttribute(kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)bytes);
  if (r == cudaSuccess) limit.done.fetch_or(bit, std::memory_order_release);
  return r;
}

}  // namespace coarse
