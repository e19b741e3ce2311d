// What is done once on each device, such as a kernel's shared-memory limit.
#pragma once
#include <atomic>
#include <cstdint>

#include <cuda_runtime_api.h>

namespace stf {

// Runs `set` on the current device unless an earlier call there succeeded.  A process may use
// several devices, each from several threads (which may both run it: it sets the same again).
class OncePerDevice {
  std::atomic<uint64_t> done{0};      // devices 0..63; others run it each time

 public:
  template <class Set>
  cudaError_t operator()(Set set) {
    int device = 0;
    cudaError_t e = cudaGetDevice(&device);
    if (e != cudaSuccess) return e;
    const uint64_t bit = device < 64 ? uint64_t(1) << device : 0;
    if (done.load(std::memory_order_acquire) & bit) return cudaSuccess;
    e = set();
    if (e == cudaSuccess) done.fetch_or(bit, std::memory_order_release);
    return e;
  }
};

}  // namespace stf
