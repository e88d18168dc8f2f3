// A kernel's dynamic shared memory limit above the default 48 KB.
#pragma once

#include <cuda_runtime_api.h>

#include <atomic>
#include <cstdint>

namespace ddflb {

// One static object per kernel: raises its limit on the current device.  The
// attribute belongs to a device and a process may use several, so it is set once
// on each; a launch after that costs one cudaGetDevice.
class SharedLimit {
 public:
  cudaError_t raise(const void* kernel, int bytes) {
    int dev = 0;
    cudaError_t e = cudaGetDevice(&dev);
    if (e != cudaSuccess) return e;
    // (beyond 64 devices: set at every launch)
    const uint64_t bit = dev >= 0 && dev < 64 ? uint64_t(1) << dev : 0;
    if (raised_.load(std::memory_order_relaxed) & bit) return cudaSuccess;
    e = cudaFuncSetAttribute(kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, bytes);
    if (e == cudaSuccess) raised_.fetch_or(bit, std::memory_order_relaxed);
    return e;
  }

 private:
  std::atomic<uint64_t> raised_{0};
};

}  // namespace ddflb
