// What belongs to a device and not to the process.  A kernel's attributes
// (its dynamic shared memory limit, non-portable cluster sizes) and its
// occupancy are those of the calling thread's current device, and a process
// may use several.
#pragma once

#include <cuda_runtime_api.h>

#include <atomic>
#include <mutex>

namespace dp {

// A value >= 0 found out once on each device: f() runs on the first call with
// a device current, on its thread (others wait for it); a negative result (a
// failure) is returned but not kept.
class PerDevice {
 public:
  template <typename F>
  int operator()(F f) {
    int dev = 0;
    if (cudaGetDevice(&dev) != cudaSuccess || dev < 0 || dev >= kMax) return f();
    int v = have_[dev].load(std::memory_order_acquire);
    if (v > 0) return v - 1;
    std::lock_guard<std::mutex> hold(m_);
    v = have_[dev].load(std::memory_order_relaxed);
    if (v > 0) return v - 1;
    v = f();
    if (v >= 0) have_[dev].store(v + 1, std::memory_order_release);
    return v;
  }

 private:
  static constexpr int kMax = 64;
  std::atomic<int> have_[kMax] = {};   // value + 1
  std::mutex m_;
};

// Sets one attribute of kernel K to `value` on the calling thread's current
// device, once on each.
template <auto K, cudaFuncAttribute A>
cudaError_t kernel_attribute(int value) {
  static PerDevice set;
  return (cudaError_t)-set([&] {
    return -(int)cudaFuncSetAttribute(reinterpret_cast<const void *>(K), A, value);
  });
}

}  // namespace dp
