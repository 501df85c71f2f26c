// The limit of a kernel's dynamic shared memory above 48 KB belongs to a device:
// it is raised once on each that launches the kernel, from whichever thread is
// first (two at once set the same value).
#pragma once

#include <cuda_runtime_api.h>

#include <atomic>
#include <cstdint>

namespace tlda {

class SmemLimit {
 public:
  // On the current device; the launch that follows reports what fails here.
  cudaError_t raise(const void *kernel, int bytes) {
    int dev = 0;
    if (cudaError_t e = cudaGetDevice(&dev)) return e;
    const uint64_t bit = dev < 64 ? uint64_t(1) << dev : 0;  // devices past the mask are set each time
    if (done_.load(std::memory_order_acquire) & bit) return cudaSuccess;
    if (cudaError_t e = cudaFuncSetAttribute(kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, bytes)) return e;
    done_.fetch_or(bit, std::memory_order_release);
    return cudaSuccess;
  }

 private:
  std::atomic<uint64_t> done_{0};
};

}  // namespace tlda
