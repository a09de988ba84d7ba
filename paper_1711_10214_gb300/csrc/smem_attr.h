// More than 48 KB of shared memory (static and dynamic) needs an attribute of the kernel,
// which holds on the device it was set on.  A SmemAttr (one static object per kernel) remembers the largest
// size set on each device, so that any device and any thread of the process may launch:
// the size only grows, under a lock, and a launch finds at least its own.
#pragma once
#include <cuda_runtime.h>

#include <atomic>
#include <cstddef>
#include <mutex>

namespace ashrt {

struct SmemAttr {
  static constexpr int kDevices = 16;   // further ones set the attribute on every call
  std::atomic<size_t> set[kDevices] = {};
  std::mutex mu;
};

inline cudaError_t set_smem_ptr(const void* kern, size_t bytes, SmemAttr& a) {
  if (bytes <= 40 * 1024) return cudaSuccess;   // with up to 8 KB of static shared memory
  int dev = 0;
  cudaError_t e = cudaGetDevice(&dev);
  if (e != cudaSuccess) return e;
  const bool known = dev >= 0 && dev < SmemAttr::kDevices;
  if (known && a.set[dev].load(std::memory_order_acquire) >= bytes) return cudaSuccess;
  std::lock_guard<std::mutex> lock(a.mu);
  if (known && a.set[dev].load(std::memory_order_relaxed) >= bytes) return cudaSuccess;
  e = cudaFuncSetAttribute(kern, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)bytes);
  if (e == cudaSuccess && known) a.set[dev].store(bytes, std::memory_order_release);
  return e;
}

template <typename K>
inline cudaError_t set_smem(K kern, size_t bytes, SmemAttr& a) {
  return set_smem_ptr((const void*)kern, bytes, a);
}

}  // namespace ashrt
