// Dynamic shared memory of a kernel.
#pragma once

#include <cuda_runtime.h>

#include <atomic>

namespace td {

// Lets launches of Kernel use all the shared memory that a block may have on the current device.  The limit is
// one per kernel, device and process, while a launch's size depends on its network and batch: a limit set to
// each launch's own size is lowered by another thread's launch between this one's setting and launching, which
// then fails (measured: four threads with a network each, batches of 1 to 700, fail within a second).  Every
// caller sets the same value, so there is nothing to lower.  It reserves nothing: a launch takes what it asks for.
template <auto Kernel>
cudaError_t allow_shared_memory() {
  static std::atomic<int> fixed{-1};   // the kernel's static shared memory, a property of its code
  int dev = 0, most = 0, own = fixed.load(std::memory_order_relaxed);
  cudaError_t e = cudaGetDevice(&dev);
  if (e == cudaSuccess) e = cudaDeviceGetAttribute(&most, cudaDevAttrMaxSharedMemoryPerBlockOptin, dev);
  if (e == cudaSuccess && own < 0) {
    cudaFuncAttributes at;
    e = cudaFuncGetAttributes(&at, Kernel);
    if (e == cudaSuccess) fixed.store(own = (int)at.sharedSizeBytes, std::memory_order_relaxed);
  }
  if (e != cudaSuccess) return e;
  return cudaFuncSetAttribute(Kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, most - own);
}

}  // namespace td
