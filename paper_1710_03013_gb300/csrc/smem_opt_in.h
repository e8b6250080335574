// A kernel's opt-in to more than 48 KB of dynamic shared memory, an attribute of
// the kernel on one device.  Asking costs 0.19 us; the launchers of an inner
// iteration (20 of them and more in a fit of 0.6 ms) ask once a device.
#pragma once

#include <cuda_runtime_api.h>
#include <stdint.h>

#include <atomic>

namespace kkm {

// done: a bit for each of the first 64 devices on which the kernel has it.  An
// error is not kept.
inline cudaError_t smem_opt_in(std::atomic<uint64_t>& done, const void* kernel, int bytes) {
  int dev = 0;
  cudaError_t e = cudaGetDevice(&dev);
  if (e != cudaSuccess) return e;
  const uint64_t bit = dev >= 0 && dev < 64 ? (uint64_t)1 << dev : 0;
  if (done.load(std::memory_order_relaxed) & bit) return cudaSuccess;
  e = cudaFuncSetAttribute(kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, bytes);
  if (e == cudaSuccess) done.fetch_or(bit, std::memory_order_relaxed);
  return e;
}

}  // namespace kkm
