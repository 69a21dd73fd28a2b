// Host-side facts and settings that belong to a device, asked or made once for each: a kernel's
// attributes and its occupancy are the device's, and a process may use several.
#pragma once

#include <cuda_runtime.h>

#include <atomic>
#include <mutex>

namespace glide {

// A value per device.  Safe from several threads; what failed is not kept.
template <class T>
class PerDevice {
 public:
  // The current device's value, made by make(T&) the first time.
  template <class F>
  cudaError_t get(T& out, F make) {
    int dev = 0;
    const cudaError_t e = cudaGetDevice(&dev);
    if (e != cudaSuccess) return e;
    if (dev < 0 || dev >= kMost) return make(out);  // more devices than are kept: made on every call
    Slot& s = slots_[dev];
    if (!s.ready.load(std::memory_order_acquire)) {
      std::lock_guard<std::mutex> lock(mutex_);
      if (!s.ready.load(std::memory_order_relaxed)) {
        const cudaError_t made = make(s.value);
        if (made != cudaSuccess) return made;
        s.ready.store(true, std::memory_order_release);
      }
    }
    out = s.value;
    return cudaSuccess;
  }

 private:
  static constexpr int kMost = 32;
  struct Slot {
    std::atomic<bool> ready{false};
    T value{};
  };
  Slot slots_[kMost];
  std::mutex mutex_;
};

// An attribute of the current device, `otherwise` if it cannot be asked.
inline int device_attribute(PerDevice<int>& kept, cudaDeviceAttr attr, int otherwise) {
  int v = otherwise;
  const cudaError_t e = kept.get(v, [&](int& x) {
    int dev = 0;
    const cudaError_t at = cudaGetDevice(&dev);
    return at == cudaSuccess ? cudaDeviceGetAttribute(&x, attr, dev) : at;
  });
  return e == cudaSuccess && v > 0 ? v : otherwise;
}

// Multiprocessors of the current device.
inline int sm_count() {
  static PerDevice<int> kept;
  return device_attribute(kept, cudaDevAttrMultiProcessorCount, 1);
}

// Largest dynamic shared memory a block of the current device may opt in to.
inline int smem_optin_bytes() {
  static PerDevice<int> kept;
  return device_attribute(kept, cudaDevAttrMaxSharedMemoryPerBlockOptin, 227 * 1024);
}

// Lets `kernel` take `bytes` of dynamic shared memory on the current device; `done` is the kernel's own.
template <class K>
cudaError_t allow_smem(PerDevice<int>& done, K kernel, int bytes) {
  int unused = 0;
  return done.get(unused, [&](int&) {
    return cudaFuncSetAttribute(kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, bytes);
  });
}

}  // namespace glide
