// Dynamic shared memory of a kernel above the 48 KB that every launch may ask for.
#pragma once

#include <cuda_runtime_api.h>

#include <atomic>
#include <cstddef>
#include <mutex>

namespace lps {

// The limit of one kernel (a static of its launcher). cudaFuncSetAttribute acts on the current device only,
// so what has been allowed is kept per device; it only grows, so that a launch of another thread or plan
// with more shared memory stays within it. A launch that is within the limit takes one device query.
class SmemLimit {
 public:
  cudaError_t raise(const void* kernel, size_t bytes) {
    if (bytes <= kDefault) return cudaSuccess;
    int dev = 0;
    cudaError_t e = cudaGetDevice(&dev);
    if (e != cudaSuccess) return e;
    if (dev >= kDevices) return cudaFuncSetAttribute(kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)bytes);
    if (allowed_[dev].load(std::memory_order_acquire) >= bytes) return cudaSuccess;
    std::lock_guard<std::mutex> lock(mutex_);
    if (allowed_[dev].load(std::memory_order_relaxed) >= bytes) return cudaSuccess;
    e = cudaFuncSetAttribute(kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)bytes);
    if (e == cudaSuccess) allowed_[dev].store(bytes, std::memory_order_release);
    return e;
  }

 private:
  static constexpr size_t kDefault = 48 * 1024;
  static constexpr int kDevices = 64;
  std::mutex mutex_;
  std::atomic<size_t> allowed_[kDevices] = {};
};

}  // namespace lps
