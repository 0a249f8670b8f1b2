// Kernels whose dynamic shared memory exceeds 48 KB need an attribute raised first.  It is a setting of
// each device, so a launcher keeps one SharedLimit per set of kernels and raises it on the first launch on
// every device (the current device's ordinal is a thread-local read of the runtime; raising it on every
// launch instead would be a driver call a step).  Safe with several threads: the attribute is set before
// its device is noted, and setting it twice changes nothing.
#pragma once

#include <cuda_runtime.h>
#include <stdint.h>

#include <atomic>

namespace gks {

class SharedLimit {
 public:
  template <class... K>
  cudaError_t raise(int bytes, K *...kernels) {
    int dev = 0;
    cudaError_t e = cudaGetDevice(&dev);
    if (e != cudaSuccess) return e;
    const uint64_t bit = dev < 64 ? uint64_t(1) << dev : 0;   // past 63: raised on every launch
    if (done_.load(std::memory_order_acquire) & bit) return cudaSuccess;
    for (const void *k : {reinterpret_cast<const void *>(kernels)...}) {
      e = cudaFuncSetAttribute(k, cudaFuncAttributeMaxDynamicSharedMemorySize, bytes);
      if (e != cudaSuccess) return e;
    }
    done_.fetch_or(bit, std::memory_order_release);
    return cudaSuccess;
  }

 private:
  std::atomic<uint64_t> done_{0};
};

}  // namespace gks
