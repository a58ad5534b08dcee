// A kernel's opt-in to more than 48 KB of dynamic shared memory, once per device.
//
// The attribute belongs to the device that is current when it is set, so a
// process that uses several devices sets it on each; one that failed is tried
// again by the next launch.  One object per kernel instantiation (a
// function-local static); safe from several threads.
#pragma once
#include <cuda_runtime.h>
#include <stddef.h>

#include <atomic>

namespace nlse {

class SmemLimit {
 public:
  template <class Kernel>
  cudaError_t allow(Kernel kern, size_t bytes) {
    int dev = 0;
    cudaError_t e = cudaGetDevice(&dev);
    if (e != cudaSuccess) return e;
    const unsigned long long bit = dev < 64 ? 1ull << dev : 0ull;   // beyond: set at every launch
    if (set_.load(std::memory_order_acquire) & bit) return cudaSuccess;
    e = cudaFuncSetAttribute(kern, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)bytes);
    if (e == cudaSuccess) set_.fetch_or(bit, std::memory_order_release);
    return e;
  }

 private:
  std::atomic<unsigned long long> set_{0};
};

}  // namespace nlse
