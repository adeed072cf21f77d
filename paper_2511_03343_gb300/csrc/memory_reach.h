// Which of a caller's arrays a plan's kernels may use where they lie.
#pragma once
#include <cuda_runtime_api.h>

namespace sssp {

// The plan's device's own memory and managed memory.  Another device's is not reachable without peer access, and
// host memory not on every system: a copy reaches both, or reports that it cannot, where a kernel would fault.
inline bool reached_in_place(cudaMemoryType type, int owner, int device) {
  return type == cudaMemoryTypeManaged || (type == cudaMemoryTypeDevice && owner == device);
}

inline bool reached_in_place(const void* p, int device) {
  cudaPointerAttributes a{};
  if (cudaPointerGetAttributes(&a, p) != cudaSuccess) {
    cudaGetLastError();
    return false;
  }
  return reached_in_place(a.type, a.device, device);
}

}  // namespace sssp
