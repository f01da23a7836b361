// Settings that belong to a device, not to the process (a kernel's dynamic
// shared-memory limit): made by the first caller on each device.
#pragma once

#include <cuda_runtime.h>

#include <atomic>
#include <mutex>

namespace ltgw {

class OncePerDevice {
 public:
  // set() once on the current device (again after a failure); its status.
  template <class F>
  cudaError_t operator()(F &&set) {
    int dev = 0;
    cudaError_t e = cudaGetDevice(&dev);
    if (e != cudaSuccess) return e;
    if (dev < 0 || dev >= kDevices) return set();
    if (done_[dev].load(std::memory_order_acquire)) return cudaSuccess;
    std::lock_guard<std::mutex> lock(mu_);
    if (done_[dev].load(std::memory_order_relaxed)) return cudaSuccess;
    e = set();
    if (e == cudaSuccess) done_[dev].store(true, std::memory_order_release);
    return e;
  }

 private:
  static constexpr int kDevices = 64;
  std::atomic<bool> done_[kDevices] = {};
  std::mutex mu_;
};

}  // namespace ltgw
