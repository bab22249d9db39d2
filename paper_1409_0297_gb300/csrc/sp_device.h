// State kept once per device of the process.
#pragma once
#include <cuda_runtime_api.h>

#include <atomic>

namespace sp {

// Function attributes (shared-memory limit, cluster size) belong to the device that is current
// when they are set.  run(set) calls set() for each device once; a failed call is tried again.
// Contexts of several threads and devices may call it side by side: the worst is a second set().
class PerDevice {
 public:
  template <class F>
  cudaError_t run(F set) {
    int dev = 0;
    cudaError_t e = cudaGetDevice(&dev);
    if (e != cudaSuccess) return e;
    if (dev < 0 || dev >= 64) return set();
    const unsigned long long bit = 1ull << dev;
    if (done_.load(std::memory_order_acquire) & bit) return cudaSuccess;
    e = set();
    if (e == cudaSuccess) done_.fetch_or(bit, std::memory_order_release);
    return e;
  }

 private:
  std::atomic<unsigned long long> done_{0};
};

}  // namespace sp
