// Internal interface of the march on periodic grids of 512, 1024 and 2048 points (march_dft.cuh).
#pragma once
#include <cuda_runtime.h>

namespace sssp {
struct SolveDesc;
}

namespace sssp_dft {

constexpr bool supported(int log2M) { return log2M >= 9 && log2M <= 11; }
// build the current device's table of a size (kept for the process; plan creation calls it)
cudaError_t prepare(int log2M);
// split: CTAs per solve that share the TL rows of a march without Neumann terms (march_kernel.cuh)
cudaError_t launch_march(int log2M, const sssp::SolveDesc* d, int count, cudaStream_t st, bool cplx, int split);

}  // namespace sssp_dft
