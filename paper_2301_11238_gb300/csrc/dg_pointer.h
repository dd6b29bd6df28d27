// Where a caller's "device" pointer may be dereferenced.
#pragma once
#include <cuda_runtime_api.h>

namespace dgswe {

// Whether kernels on device `dev` may use memory with these attributes without peer
// access or host mapping; anything else goes through copies, which take every
// address the driver knows.
inline bool kernel_addressable(const cudaPointerAttributes& a, int dev) {
  return a.type == cudaMemoryTypeDevice && a.device == dev;
}

// The same for a pointer and the current device (false if CUDA cannot tell).
inline bool kernel_addressable(const void* p) {
  cudaPointerAttributes a{};
  int dev = -1;
  if (cudaGetDevice(&dev) != cudaSuccess || cudaPointerGetAttributes(&a, p) != cudaSuccess) {
    cudaGetLastError();
    return false;
  }
  return kernel_addressable(a, dev);
}

}  // namespace dgswe
