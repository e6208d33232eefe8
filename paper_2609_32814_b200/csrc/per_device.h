// Attributes of a kernel (its shared-memory limit, cluster sizes) belong to a device, not to the process.
#pragma once

#include <cuda_runtime_api.h>

#include <atomic>
#include <cstdint>

namespace algproj {

// once(set) runs `set` the first time it is called with a device current, and again while `set` fails; one per kernel,
// called by any thread.
class OncePerDevice {
  std::atomic<uint64_t> done_{0};   // a bit each

 public:
  template <typename Set>
  cudaError_t operator()(Set set) {
    int dev = 0;
    cudaError_t e = cudaGetDevice(&dev);
    if (e != cudaSuccess) return e;
    const bool tracked = dev >= 0 && dev < 64;   // (a device past the bits: set every time)
    if (tracked && (done_.load(std::memory_order_acquire) >> dev & 1)) return cudaSuccess;
    e = set();
    if (e == cudaSuccess && tracked) done_.fetch_or(1ull << dev, std::memory_order_release);
    return e;
  }
};

}  // namespace algproj
