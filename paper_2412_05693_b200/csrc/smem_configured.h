// The largest dynamic shared-memory size a kernel has been configured for, per device: cudaFuncSetAttribute applies to the
// current device only, and a process may hold handles on several GPUs.  Threads with handles of their own share a kernel's
// entry; the attribute only ever grows, so that none takes back what another is about to launch with.
#pragma once
#include <cuda_runtime.h>

#include <atomic>
#include <cstddef>
#include <mutex>

namespace bm {

struct SmemConfigured {
  std::atomic<size_t> bytes[64] = {};
  std::mutex growing;
  template <typename Kernel>
  cudaError_t ensure(Kernel kernel, size_t smem) {
    int dev = 0;
    cudaError_t e = cudaGetDevice(&dev);
    if (e != cudaSuccess) return e;
    if (dev < 0 || dev >= 64) return cudaErrorInvalidDevice;
    if (smem <= bytes[dev].load(std::memory_order_acquire)) return cudaSuccess;
    std::lock_guard<std::mutex> lock(growing);
    if (smem <= bytes[dev].load(std::memory_order_relaxed)) return cudaSuccess;
    e = cudaFuncSetAttribute(reinterpret_cast<const void*>(kernel), cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem);
    if (e != cudaSuccess) return e;
    bytes[dev].store(smem, std::memory_order_release);
    return cudaSuccess;
  }
};

}  // namespace bm
