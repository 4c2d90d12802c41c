// A preparation that runs once per device (kernel attributes belong to the
// device that is current when they are set); safe with several host threads:
// two that meet run it twice, which attributes allow.
#pragma once
#include <cuda_runtime.h>
#include <stdint.h>

#include <atomic>

namespace tg {

class DeviceOnce {
 public:
  // f() on the first call with the current device (on every call beyond
  // device 63), again after a failure
  template <class F>
  cudaError_t operator()(F f) {
    int dev = 0;
    cudaError_t e = cudaGetDevice(&dev);
    if (e != cudaSuccess) return e;
    const uint64_t bit = (dev >= 0 && dev < 64) ? 1ull << dev : 0;
    if (done_.load(std::memory_order_acquire) & bit) return cudaSuccess;
    e = f();
    if (e == cudaSuccess) done_.fetch_or(bit, std::memory_order_release);
    return e;
  }

 private:
  std::atomic<uint64_t> done_{0};
};

}  // namespace tg
