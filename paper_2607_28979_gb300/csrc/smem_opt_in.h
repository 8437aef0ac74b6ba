// A kernel's opt-in to more than 48 KB of dynamic shared memory, remembered per device.
#pragma once

#include <cuda_runtime_api.h>

#include <atomic>
#include <mutex>

namespace mot {

// One static object per kernel at its launch site. CUDA keeps the attribute per device, a process may
// hold handles on several, and every call makes its handle's device current; threads may launch at
// the same time. The size only grows, so that a smaller launch does not lower it under another
// thread's larger one.
class SmemOptIn {
 public:
  template <class... P>
  cudaError_t operator()(void (*kernel)(P...), int bytes) {
    return set(reinterpret_cast<const void*>(kernel), bytes);
  }

 private:
  static constexpr int kDefault = 48 * 1024, kDevices = 64;

  cudaError_t set(const void* kernel, int bytes) {
    if (bytes <= kDefault) return cudaSuccess;
    int dev = 0;
    cudaError_t e = cudaGetDevice(&dev);
    if (e != cudaSuccess) return e;
    if (dev >= kDevices)   // not remembered
      return cudaFuncSetAttribute(kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, bytes);
    if (have_[dev].load(std::memory_order_acquire) >= bytes) return cudaSuccess;
    std::lock_guard<std::mutex> lock(m_);
    if (have_[dev].load(std::memory_order_relaxed) >= bytes) return cudaSuccess;
    e = cudaFuncSetAttribute(kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, bytes);
    if (e == cudaSuccess) have_[dev].store(bytes, std::memory_order_release);
    return e;
  }

  std::mutex m_;
  std::atomic<int> have_[kDevices] = {};
};

}  // namespace mot
