// Settings that belong to one device. A context may be made on any device of the process, so
// nothing about a device is kept for the process as a whole.
#pragma once
#include <cuda_runtime.h>

#include <atomic>
#include <mutex>

namespace tmk {

constexpr int kMaxDevices = 64;  // devices beyond these ask the runtime every time

// SMs of the current device
inline int sm_count() {
  static std::atomic<int> known[kMaxDevices];
  int dev = 0, n = 0;
  if (cudaGetDevice(&dev) != cudaSuccess) return 148;
  const bool kept = dev >= 0 && dev < kMaxDevices;
  if (kept && (n = known[dev].load(std::memory_order_relaxed)) > 0) return n;
  if (cudaDeviceGetAttribute(&n, cudaDevAttrMultiProcessorCount, dev) != cudaSuccess || n <= 0) return 148;
  if (kept) known[dev].store(n, std::memory_order_relaxed);
  return n;
}

// Lets Kernel be launched with `bytes` of dynamic shared memory on the current device: the limit is
// an attribute of the kernel on one device, raised once for each (and again for more bytes).
template <auto Kernel>
bool allow_smem(size_t bytes) {
  static std::atomic<size_t> raised[kMaxDevices];
  static std::mutex raising;  // two threads with different sizes must not lower each other's limit
  int dev = 0;
  if (cudaGetDevice(&dev) != cudaSuccess) return false;
  const bool kept = dev >= 0 && dev < kMaxDevices;
  if (kept && raised[dev].load(std::memory_order_relaxed) >= bytes) return true;
  std::lock_guard<std::mutex> lock(raising);
  if (kept && raised[dev].load(std::memory_order_relaxed) >= bytes) return true;
  if (cudaFuncSetAttribute(Kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)bytes) != cudaSuccess) return false;
  if (kept) raised[dev].store(bytes, std::memory_order_relaxed);
  return true;
}

}  // namespace tmk
