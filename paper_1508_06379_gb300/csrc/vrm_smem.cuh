// Dynamic shared memory beyond the 48 KB a launch may ask for by itself.
#pragma once

#include <cuda_runtime_api.h>

#include <atomic>
#include <cstddef>

namespace vrm {

// Lets KERNEL ask for up to `bytes` (the largest that any launch of it takes) on
// the current device.  The limit is a property of kernel and device, so it is
// set once on each device (a launch on another one would be refused), and to one
// value only: set to each launch's own size, a thread could lower it between
// another's setting and launch.
template <auto KERNEL>
inline cudaError_t allow_smem(size_t bytes) {
  static std::atomic<unsigned long long> done{0};  // a bit per device
  int dev = 0;
  cudaError_t e = cudaGetDevice(&dev);
  if (e != cudaSuccess) return e;
  const unsigned long long bit = dev < 64 ? 1ull << dev : 0ull;  // (beyond: set on every call)
  if (done.load(std::memory_order_acquire) & bit) return cudaSuccess;
  e = cudaFuncSetAttribute(reinterpret_cast<const void*>(KERNEL), cudaFuncAttributeMaxDynamicSharedMemorySize,
                           (int)bytes);
  if (e == cudaSuccess) done.fetch_or(bit, std::memory_order_release);
  return e;
}

}  // namespace vrm
