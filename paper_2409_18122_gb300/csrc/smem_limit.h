// smem_limit.h -- the opt-in to more than 48 KB of dynamic shared memory, which belongs to one
// kernel on one device.
#pragma once

#include <cuda_runtime_api.h>
#include <stddef.h>
#include <stdint.h>

#include <atomic>

namespace gs {

// Lets `kKernel` be launched on the current device with `bytes` of dynamic shared memory.  Always
// called with the same size for a kernel; the runtime is asked once per kernel and device (a flag
// each for the first 64 devices, every time beyond them), from whichever thread comes first.
template <auto kKernel>
cudaError_t allow_smem(size_t bytes) {
  static std::atomic<uint64_t> done{0};
  int dev = 0;
  cudaError_t e = cudaGetDevice(&dev);
  if (e != cudaSuccess) return e;
  const uint64_t bit = dev >= 0 && dev < 64 ? (uint64_t)1 << dev : 0;
  if (done.load(std::memory_order_acquire) & bit) return cudaSuccess;
  e = cudaFuncSetAttribute(reinterpret_cast<const void*>(kKernel), cudaFuncAttributeMaxDynamicSharedMemorySize,
                           (int)bytes);
  if (e == cudaSuccess) done.fetch_or(bit, std::memory_order_release);
  return e;
}

}  // namespace gs
