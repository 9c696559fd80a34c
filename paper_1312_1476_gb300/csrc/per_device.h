// per_device.h -- a number formed once per device.
//
// What a launcher finds out or sets once before its first launch (a kernel's
// dynamic shared memory, permission for clusters of 16, resident blocks) holds for
// the kernel on one device; a problem of another device in the same process needs
// its own.
#pragma once

#include <cuda_runtime.h>

#include <atomic>

namespace gmrf {

class PerDevice {
 public:
  // The current device's number, from form(&v) (v > 0 where it returns cudaSuccess)
  // unless an earlier call formed it.  Several host threads may form it at once.
  template <typename F>
  cudaError_t get(F&& form, int* out = nullptr) {
    int dev = -1;
    cudaError_t e = cudaGetDevice(&dev);
    if (e != cudaSuccess) return e;
    const bool kept = dev >= 0 && dev < kDevices;
    int v = kept ? v_[dev].load(std::memory_order_acquire) : 0;
    if (v == 0) {
      e = form(&v);
      if (e != cudaSuccess) return e;
      if (kept) v_[dev].store(v, std::memory_order_release);
    }
    if (out) *out = v;
    return cudaSuccess;
  }

 private:
  static constexpr int kDevices = 64;
  std::atomic<int> v_[kDevices] = {};
};

// A function attribute, on the current device.
template <typename K>
cudaError_t set_attribute(PerDevice& done, K* kernel, cudaFuncAttribute attr, int value) {
  return done.get([&](int* v) {
    *v = 1;
    return cudaFuncSetAttribute(reinterpret_cast<const void*>(kernel), attr, value);
  });
}

}  // namespace gmrf
