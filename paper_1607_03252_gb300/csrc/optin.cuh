// The dynamic shared-memory opt-in of a kernel (more than 48 KB per block). The limit belongs to the
// device that is current when it is raised, so it is kept per kernel and device; a call that
// fails is not remembered: the next one tries again and reports it again.
#pragma once
#include <cuda_runtime.h>

#include <atomic>

namespace mlmc {

constexpr int kMaxDevices = 64;

// Allows `bytes` of dynamic shared memory (the same on every call) for launches of Kernel on the
// device current on the calling thread. Cheap once done for the device; safe from several threads.
template <auto Kernel>
[[nodiscard]] inline cudaError_t allow_dynamic_smem(size_t bytes) {
  static std::atomic<bool> done[kMaxDevices]{};
  int dev = 0;
  cudaError_t e = cudaGetDevice(&dev);
  if (e != cudaSuccess) return e;
  const bool known = dev >= 0 && dev < kMaxDevices;
  if (known && done[dev].load(std::memory_order_relaxed)) return cudaSuccess;
  e = cudaFuncSetAttribute(Kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)bytes);
  if (e == cudaSuccess && known) done[dev].store(true, std::memory_order_relaxed);
  return e;
}

}  // namespace mlmc
