// Tables, instantiations and launches of the parity-split one-CTA march kernel (march_eo.cuh).
#include <cuda_runtime.h>

#include <algorithm>
#include <cmath>
#include <map>
#include <mutex>
#include <utility>
#include <vector>

#include "eo_launch.h"
#include "march_eo.cuh"

namespace sssp_eo {

namespace {

std::mutex g_mu;
std::map<std::pair<int, int>, sssp::EoTabs> g_tabs;  // (device, log2L)
std::map<int, int> g_sms;                             // device -> SMs

template <int LOG2L>
cudaError_t set_attrs() {
  const cudaFuncAttribute a = cudaFuncAttributeMaxDynamicSharedMemorySize;
  cudaError_t e = cudaFuncSetAttribute(sssp::sssp_dst_eo_kernel<LOG2L>, a, int(sssp::EDst<LOG2L>::SMEM));
  if constexpr (LOG2L >= kMinMarchLog2) {
    if (e == cudaSuccess)
      e = cudaFuncSetAttribute(sssp::sssp_march_eo_kernel<LOG2L, false>, a, int(sssp::ECfg<LOG2L>::SMEM));
    if (e == cudaSuccess)
      e = cudaFuncSetAttribute(sssp::sssp_march_eo_kernel<LOG2L, true>, a, int(sssp::ECfg<LOG2L>::SMEM_CPLX));
  }
  return e;
}

// tables in FP64, rounded once to FP32, and the kernels' shared-memory attributes
cudaError_t tabs_for(int log2L, sssp::EoTabs* out) {
  int dev = 0;
  cudaError_t e = cudaGetDevice(&dev);
  if (e != cudaSuccess) return e;
  std::lock_guard<std::mutex> lk(g_mu);
  auto it = g_tabs.find({dev, log2L});
  if (it != g_tabs.end()) {
    *out = it->second;
    return cudaSuccess;
  }
  e = log2L == 9 ? set_attrs<9>() : (log2L == 10 ? set_attrs<10>() : (log2L == 11 ? set_attrs<11>() : set_attrs<12>()));
  if (e != cudaSuccess) return e;
  const int L = 1 << log2L, M = L / 2;
  std::vector<float2> h(2 * size_t(M) + 1 + size_t(M) / 2);  // wM (M), cL (M + 1), beta (M floats)
  for (int i = 0; i < M; ++i) h[i] = make_float2(float(std::cos(2.0 * M_PI * i / M)), float(-std::sin(2.0 * M_PI * i / M)));
  for (int i = 0; i <= M; ++i) h[M + i] = make_float2(float(std::cos(M_PI * i / L)), float(-std::sin(M_PI * i / L)));
  float* beta = reinterpret_cast<float*>(&h[2 * M + 1]);
  beta[0] = 0.f;
  for (int i = 1; i < M; ++i) beta[i] = float(0.5 / std::sin(M_PI * i / M));
  float2* d = nullptr;
  if ((e = cudaMalloc(&d, sizeof(float2) * h.size())) != cudaSuccess) return e;
  if ((e = cudaMemcpy(d, h.data(), sizeof(float2) * h.size(), cudaMemcpyHostToDevice)) != cudaSuccess) {
    cudaFree(d);
    return e;
  }
  if (!g_sms.count(dev) && (e = cudaDeviceGetAttribute(&g_sms[dev], cudaDevAttrMultiProcessorCount, dev)) != cudaSuccess) return e;
  const sssp::EoTabs t{d, d + M, reinterpret_cast<const float*>(d + 2 * M + 1)};
  g_tabs[{dev, log2L}] = t;
  *out = t;
  return cudaSuccess;
}

template <int LOG2L>
cudaError_t launch_t(const sssp::SolveDesc* d, int count, const sssp::EoTabs& tb, cudaStream_t st, bool cplx) {
  using K = sssp::ECfg<LOG2L>;
  if (cplx) sssp::sssp_march_eo_kernel<LOG2L, true><<<count, K::NT, K::SMEM_CPLX, st>>>(d, tb);
  else sssp::sssp_march_eo_kernel<LOG2L, false><<<count, K::NT, K::SMEM, st>>>(d, tb);
  return cudaGetLastError();
}

template <int LOG2L>
cudaError_t dst_t(const float2* in, float2* out, float scale, int count, long long is, long long os, int off,
                  const sssp::EoTabs& tb, cudaStream_t st, const sssp::StartArgs& sa, int sms) {
  using D = sssp::EDst<LOG2L>;
  sssp::sssp_dst_eo_kernel<LOG2L><<<std::min(count, sms * D::MIN_BLOCKS), D::K::NT, D::SMEM, st>>>(in, out, scale, tb, count, is,
                                                                                                   os, off, sa);
  return cudaGetLastError();
}

}  // namespace

cudaError_t launch_dst(int log2L, const float2* in, float2* out, float scale, int count, long long in_stride,
                       long long out_stride, int off, cudaStream_t st, const sssp::StartArgs& sa) {
  if (!supported(log2L)) return cudaErrorInvalidValue;
  sssp::EoTabs t;
  const cudaError_t e = tabs_for(log2L, &t);
  if (e != cudaSuccess) return e;
  int dev = 0, sms = 0;
  cudaGetDevice(&dev);
  {
    std::lock_guard<std::mutex> lk(g_mu);
    sms = g_sms[dev];
  }
  switch (log2L) {
    case 9: return dst_t<9>(in, out, scale, count, in_stride, out_stride, off, t, st, sa, sms);
    case 10: return dst_t<10>(in, out, scale, count, in_stride, out_stride, off, t, st, sa, sms);
    case 11: return dst_t<11>(in, out, scale, count, in_stride, out_stride, off, t, st, sa, sms);
    default: return dst_t<12>(in, out, scale, count, in_stride, out_stride, off, t, st, sa, sms);
  }
}

cudaError_t prepare(int log2L) {
  if (!supported(log2L)) return cudaErrorInvalidValue;
  sssp::EoTabs t;
  return tabs_for(log2L, &t);
}

cudaError_t launch_march(int log2L, const sssp::SolveDesc* d, int count, cudaStream_t st, bool cplx) {
  if (!march_supported(log2L)) return cudaErrorInvalidValue;
  sssp::EoTabs t;
  const cudaError_t e = tabs_for(log2L, &t);
  if (e != cudaSuccess) return e;
  switch (log2L) {
    case 11: return launch_t<11>(d, count, t, st, cplx);
    default: return launch_t<12>(d, count, t, st, cplx);
  }
}

}  // namespace sssp_eo
