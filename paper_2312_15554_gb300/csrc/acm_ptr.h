// acm_ptr.h -- where a caller's buffer lies (host code, plain C++).
#pragma once
#include <cuda_runtime_api.h>

namespace acm {

// Device memory of the current device `dev` (the kernels run there and read and
// write the buffer directly), or managed memory. Memory of another GPU is not: a
// kernel reaches it only with peer access, a copy always does.
inline bool on_device(const void* p, int dev) {
  cudaPointerAttributes a;
  if (cudaPointerGetAttributes(&a, p) != cudaSuccess) {
    cudaGetLastError();
    return false;
  }
  return (a.type == cudaMemoryTypeDevice && a.device == dev) || a.type == cudaMemoryTypeManaged;
}

}  // namespace acm
