// Internal interface of the one-CTA kernels whose warps split the modes by parity (march_eo.cuh), on
// Dirichlet grids: the transform for L = N + 1 in [512, 4096], and the default shape's march for
// L = 2048 and 4096.
#pragma once
#include <cuda_runtime.h>

namespace sssp {
struct SolveDesc;
struct StartArgs;
}

namespace sssp_eo {

constexpr int kMinLog2 = 9;        // the transform
constexpr int kMinMarchLog2 = 11;  // the march
constexpr int kMaxLog2 = 12;

constexpr bool supported(int log2L) { return log2L >= kMinLog2 && log2L <= kMaxLog2; }
constexpr bool march_supported(int log2L) { return log2L >= kMinMarchLog2 && log2L <= kMaxLog2; }
// build the current device's tables of a size (kept for the process; plan creation calls it so that a
// march allocates nothing)
cudaError_t prepare(int log2L);
cudaError_t launch_march(int log2L, const sssp::SolveDesc* d, int count, cudaStream_t st, bool cplx);

// DST-I of `count` fields (sssp_dst_eo_kernel); off = 1: L-long result rows from mode 0, off = 0: N-long
cudaError_t launch_dst(int log2L, const float2* in, float2* out, float scale, int count, long long in_stride,
                       long long out_stride, int off, cudaStream_t st, const sssp::StartArgs& sa);

}  // namespace sssp_eo
