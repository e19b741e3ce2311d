// Where a caller's array lies.
#pragma once
#include <cuda_runtime_api.h>

namespace stf {

// Memory allocated on `device` itself: not managed or page-locked, and not another device's,
// which kernels here cannot write without peer access.
inline bool local_attributes(const cudaPointerAttributes& at, int device) {
  return at.type == cudaMemoryTypeDevice && at.device == device;
}

// Whether p lies in memory of the current device (false for NULL).
inline bool local_memory(const void* p) {
  cudaPointerAttributes at;
  int device = 0;
  if (!p) return false;
  if (cudaPointerGetAttributes(&at, p) != cudaSuccess || cudaGetDevice(&device) != cudaSuccess) {
    cudaGetLastError();
    return false;
  }
  return local_attributes(at, device);
}

}  // namespace stf
