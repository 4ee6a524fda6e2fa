// A kernel's attributes (its dynamic shared-memory limit, its preferred
// shared-memory split) are those of one device: each device that a process
// uses needs them set, whichever thread comes first.
#pragma once

#include <cuda_runtime.h>

#include <atomic>

class PerDevice {
 public:
  // calls set() (a cudaError_t) on a device's first use, and again while it fails
  template <class F>
  cudaError_t once(F set) {
    int dev = 0;
    cudaError_t e = cudaGetDevice(&dev);
    if (e != cudaSuccess) return e;
    const unsigned long long bit = dev < 64 ? 1ull << dev : 0;  // further devices: every time
    if (done_.load(std::memory_order_acquire) & bit) return cudaSuccess;
    e = set();
    if (e == cudaSuccess) done_.fetch_or(bit, std::memory_order_release);
    return e;
  }

 private:
  std::atomic<unsigned long long> done_{0};
};
