// State that belongs to a device, such as a kernel's function attributes: set or
// found on the first use on every device of the process.
#pragma once

#include <atomic>

#include <cuda_runtime.h>

namespace hyteg {

struct PerDevice {
  static constexpr int kDevices = 64;  // on further devices: found by every call
  std::atomic<int> found[kDevices] = {};  // value + 1; 0: not yet found

  // *value: what find(value) gave on the current device.  Threads that come
  // first together may all call find, which gives them the same.
  template <class F>
  cudaError_t get(int* value, F find) {
    int d = 0;
    cudaError_t e = cudaGetDevice(&d);
    if (e != cudaSuccess) return e;
    const bool kept = d >= 0 && d < kDevices;
    if (const int v = kept ? found[d].load(std::memory_order_acquire) : 0) {
      *value = v - 1;
      return cudaSuccess;
    }
    e = find(value);
    if (e == cudaSuccess && kept) found[d].store(*value + 1, std::memory_order_release);
    return e;
  }
};

}  // namespace hyteg
