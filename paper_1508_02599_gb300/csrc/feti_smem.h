// Shared memory that a kernel may be launched with.
//
// The limit (cudaFuncAttributeMaxDynamicSharedMemorySize) belongs to the function
// on its device, not to a launch: contexts in several threads share it.  Set to a
// launch's own size it can be lowered by one thread between another's setting it
// and launching, and that launch is refused.  So it is only ever set to one value,
// all that a block may have on the device beside the kernel's static arrays, and
// nothing is remembered here: a device reset takes the limit with it.
#pragma once
#include <cuda_runtime.h>

#include <cstddef>

namespace feti {

// Before a launch of `kernel` with `bytes` of dynamic shared memory on the
// current device; 48 KB in all need no permission.
template <typename Kernel>
cudaError_t allow_smem(Kernel* kernel, size_t bytes) {
  if (bytes <= 16 * 1024) return cudaSuccess;  // no kernel here has more than 32 KB of static arrays
  const void* fn = reinterpret_cast<const void*>(kernel);
  cudaFuncAttributes a{};
  int dev = 0, most = 0;
  cudaError_t e = cudaFuncGetAttributes(&a, fn);
  if (e == cudaSuccess) e = cudaGetDevice(&dev);
  if (e == cudaSuccess) e = cudaDeviceGetAttribute(&most, cudaDevAttrMaxSharedMemoryPerBlockOptin, dev);
  if (e != cudaSuccess) return e;
  const int full = most - (int)a.sharedSizeBytes;
  if (a.maxDynamicSharedSizeBytes >= full) return cudaSuccess;
  return cudaFuncSetAttribute(fn, cudaFuncAttributeMaxDynamicSharedMemorySize, full);
}

}  // namespace feti
