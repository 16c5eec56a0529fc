// What the host asks or sets once per device: kernel attributes hold for the device that is current when they are set,
// and what is resident at once is a device's own.
#pragma once
#include <mutex>

#include <cuda_runtime.h>

namespace cat {

// get(f): f()'s result on the current device, from f's first call there.  f itself runs every time on a device with a
// number past the table's (the library's entry points refuse those anyway).
template <typename R>
class PerDevice {
 public:
  template <typename F>
  R get(F&& f) {
    int dev = -1;
    if (cudaGetDevice(&dev) != cudaSuccess || dev < 0 || dev >= kMax) return f();
    std::lock_guard<std::mutex> lock(mu_);
    if (!have_[dev]) {
      value_[dev] = f();
      have_[dev] = true;
    }
    return value_[dev];
  }

 private:
  static constexpr int kMax = 64;
  std::mutex mu_;
  bool have_[kMax] = {};
  R value_[kMax] = {};
};

// Allows `kernel` the given dynamic shared memory on the current device.
template <typename Kernel>
cudaError_t allow_smem(Kernel kernel, size_t bytes) {
  return cudaFuncSetAttribute(kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)bytes);
}

}  // namespace cat
