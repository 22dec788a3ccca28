// Opt-in to the largest dynamic shared memory, once per kernel and device.
#pragma once
#include <cuda_runtime.h>

#include <mutex>

namespace mpsvqe {
namespace gate {

// The dynamic shared-memory limit of a kernel is process-wide state: handles of
// different chi launch the same instantiation from several threads, so the limit is
// raised once to the device's opt-in maximum and never lowered.
template <auto Kernel>
inline cudaError_t raise_smem_limit() {
  static std::once_flag once[64];
  static cudaError_t status[64];
  int dev = 0;
  cudaError_t e = cudaGetDevice(&dev);
  if (e != cudaSuccess) return e;
  if (dev < 0 || dev >= 64) return cudaErrorInvalidDevice;
  std::call_once(once[dev], [dev] {
    int optin = 0;
    status[dev] = cudaDeviceGetAttribute(&optin, cudaDevAttrMaxSharedMemoryPerBlockOptin, dev);
    if (status[dev] == cudaSuccess)
      status[dev] = cudaFuncSetAttribute(Kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, optin);
  });
  return status[dev];
}

}  // namespace gate
}  // namespace mpsvqe
