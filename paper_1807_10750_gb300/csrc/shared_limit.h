// How much dynamic shared memory a kernel may be launched with.
#pragma once

#include <cuda_runtime.h>

namespace isingx {

// Lets `kernel` be launched with all the shared memory the device gives a
// block; cudaErrorInvalidValue if a launch with `bytes` would not fit even so.
// The limit belongs to the kernel, not to the handle that sets it: set to a
// handle's own size, it would refuse the larger launch of another thread's handle
// between that thread's set and its launch. With one value there is no order
// to get wrong.
inline cudaError_t allow_shared(const void* kernel, int device, size_t bytes) {
  int optin = 0;
  cudaFuncAttributes attr{};
  cudaError_t e = cudaDeviceGetAttribute(&optin, cudaDevAttrMaxSharedMemoryPerBlockOptin, device);
  if (e == cudaSuccess) e = cudaFuncGetAttributes(&attr, kernel);
  if (e != cudaSuccess) return e;
  const int limit = optin - static_cast<int>(attr.sharedSizeBytes);
  if (limit < 0 || bytes > static_cast<size_t>(limit)) return cudaErrorInvalidValue;
  return attr.maxDynamicSharedSizeBytes == limit
             ? cudaSuccess
             : cudaFuncSetAttribute(kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, limit);
}

}  // namespace isingx
