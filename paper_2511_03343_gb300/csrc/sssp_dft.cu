// Tables, instantiations and launches of the march on periodic grids of 512 .. 2048 points (march_dft.cuh).
#include <cuda_runtime.h>

#include <cmath>
#include <map>
#include <mutex>
#include <utility>
#include <vector>

#include "dft_launch.h"
#include "march_dft.cuh"

namespace sssp_dft {

namespace {

std::mutex g_mu;
std::map<std::pair<int, int>, const float2*> g_tabs;  // (device, log2M): the roots of DTw

template <int LOG2M>
cudaError_t set_attrs() {
  const cudaFuncAttribute a = cudaFuncAttributeMaxDynamicSharedMemorySize;
  const int sm = int(sssp::DCfg<LOG2M>::SMEM);
  const cudaError_t e = cudaFuncSetAttribute(sssp::sssp_march_dft_kernel<LOG2M, false>, a, sm);
  return e != cudaSuccess ? e : cudaFuncSetAttribute(sssp::sssp_march_dft_kernel<LOG2M, true>, a, sm);
}

cudaError_t tabs_for(int log2M, const float2** out) {
  int dev = 0;
  cudaError_t e = cudaGetDevice(&dev);
  if (e != cudaSuccess) return e;
  std::lock_guard<std::mutex> lk(g_mu);
  auto it = g_tabs.find({dev, log2M});
  if (it != g_tabs.end()) {
    *out = it->second;
    return cudaSuccess;
  }
  e = log2M == 9 ? set_attrs<9>() : (log2M == 10 ? set_attrs<10>() : set_attrs<11>());
  if (e != cudaSuccess) return e;
  const int M = 1 << log2M, Q = M / 64;
  std::vector<float2> h(M + Q);
  for (int i = 0; i < M; ++i) h[i] = make_float2(float(std::cos(2.0 * M_PI * i / M)), float(-std::sin(2.0 * M_PI * i / M)));
  for (int j = 0; j < Q; ++j)
    h[M + j] = make_float2(float(std::cos(2.0 * M_PI * j / Q) - double(h[64 * j].x)), float(-std::sin(2.0 * M_PI * j / Q) - double(h[64 * j].y)));
  float2* d = nullptr;
  if ((e = cudaMalloc(&d, sizeof(float2) * h.size())) != cudaSuccess) return e;
  if ((e = cudaMemcpy(d, h.data(), sizeof(float2) * h.size(), cudaMemcpyHostToDevice)) != cudaSuccess) {
    cudaFree(d);
    return e;
  }
  *out = g_tabs[{dev, log2M}] = d;
  return cudaSuccess;
}

template <int LOG2M>
cudaError_t launch_t(const sssp::SolveDesc* d, int count, const float2* wM, cudaStream_t st, bool cplx, int split) {
  using K = sssp::DCfg<LOG2M>;
  if (cplx) sssp::sssp_march_dft_kernel<LOG2M, true><<<dim3(count, split), K::NT, K::SMEM, st>>>(d, wM);
  else sssp::sssp_march_dft_kernel<LOG2M, false><<<dim3(count, split), K::NT, K::SMEM, st>>>(d, wM);
  return cudaGetLastError();
}

}  // namespace

cudaError_t prepare(int log2M) {
  const float2* t = nullptr;
  return supported(log2M) ? tabs_for(log2M, &t) : cudaErrorInvalidValue;
}

cudaError_t launch_march(int log2M, const sssp::SolveDesc* d, int count, cudaStream_t st, bool cplx, int split) {
  const float2* t = nullptr;
  const cudaError_t e = supported(log2M) ? tabs_for(log2M, &t) : cudaErrorInvalidValue;
  if (e != cudaSuccess) return e;
  switch (log2M) {
    case 9: return launch_t<9>(d, count, t, st, cplx, split);
    case 10: return launch_t<10>(d, count, t, st, cplx, split);
    default: return launch_t<11>(d, count, t, st, cplx, split);
  }
}

}  // namespace sssp_dft
