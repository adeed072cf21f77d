// Internal interface of the one-CTA march kernel whose warps split the modes by parity
// (march_eo.cuh): the default shape's kernel on Dirichlet grids with L = N + 1 in [512, 4096].
#pragma once
#include <cuda_runtime.h>

namespace sssp {
struct SolveDesc;
}

namespace sssp_eo {

constexpr int kMinLog2 = 9;
constexpr int kMaxLog2 = 12;

inline bool supported(int log2L) { return log2L >= kMinLog2 && log2L <= kMaxLog2; }
// build the current device's tables of a size (kept for the process; plan creation calls it so that a
// march allocates nothing)
cudaError_t prepare(int log2L);
cudaError_t launch_march(int log2L, const sssp::SolveDesc* d, int count, cudaStream_t st, bool cplx);

}  // namespace sssp_eo
