// Set-up that each device of the process needs once, such as a kernel's
// attributes, from any thread.
#pragma once

#include <cuda_runtime_api.h>

#include <atomic>

namespace tn {

// Runs `setup` on the current device unless it has succeeded there before.  Two
// threads may both run it, so it must be safe to repeat; a failure is returned
// and tried again by the next call.
class PerDevice {
 public:
  template <class F>
  cudaError_t operator()(F&& setup) {
    int dev = 0;
    cudaError_t e = cudaGetDevice(&dev);
    if (e != cudaSuccess) return e;
    const bool known = dev >= 0 && dev < kDevices;  // (beyond: set up by every call)
    if (known && done_[dev].load(std::memory_order_acquire)) return cudaSuccess;
    e = setup();
    if (e == cudaSuccess && known) done_[dev].store(true, std::memory_order_release);
    return e;
  }

 private:
  static constexpr int kDevices = 64;
  std::atomic<bool> done_[kDevices] = {};
};

// Lets `kernel` use `bytes` of dynamic shared memory on the current device.
template <class K>
cudaError_t allow_smem(PerDevice& once, K* kernel, int bytes) {
  return once([&] {
    return cudaFuncSetAttribute(reinterpret_cast<const void*>(kernel), cudaFuncAttributeMaxDynamicSharedMemorySize, bytes);
  });
}

}  // namespace tn
