// Dynamic shared memory that, with a kernel's static arrays (up to 14 KB here),
// may exceed the 48 KB every launch may use.  The limit belongs to the kernel, not to a launch,
// so it is always set to all an SM has: a value fitted to one grid would fail
// the launch of another grid's solve, by another thread or between a solve's
// begin and its iterations.
#pragma once

#include <cuda_runtime.h>

namespace dpf {

// Before a launch with `bytes` of dynamic shared memory (any number of times).
template <class F>
inline cudaError_t allow_smem(F* kernel, size_t bytes) {
  if (bytes <= 32 * 1024) return cudaSuccess;
  int dev = 0, most = 0;
  cudaFuncAttributes at;
  cudaError_t e = cudaGetDevice(&dev);
  if (e == cudaSuccess) e = cudaDeviceGetAttribute(&most, cudaDevAttrMaxSharedMemoryPerBlockOptin, dev);
  if (e == cudaSuccess) e = cudaFuncGetAttributes(&at, (const void*)kernel);
  if (e == cudaSuccess)
    e = cudaFuncSetAttribute((const void*)kernel, cudaFuncAttributeMaxDynamicSharedMemorySize,
                             most - (int)at.sharedSizeBytes);
  return e;
}

}  // namespace dpf
