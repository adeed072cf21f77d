// Launch of the FD-SSP march kernel (march_fd.cuh), L = N + 1 = 8 .. 4096, and the host FP64
// factorisation of its tridiagonal stage matrices.
#include <cuda_runtime.h>

#include <complex>
#include <map>
#include <mutex>
#include <vector>

#include "fd_launch.h"
#include "march_fd.cuh"

namespace sssp_fd {

namespace {

struct Room {
  int sms = 0, solves = 0;  // SMs of a device, staged solves resident on one
};

// the staged form's shared-memory attribute and residency on the current device (once a device and size)
template <int LOG2L>
cudaError_t room_for(Room* out) {
  using C = sssp::FdCfg<LOG2L>;
  static std::mutex mu;
  static std::map<int, Room> cache;
  int dev = 0;
  cudaError_t e = cudaGetDevice(&dev);
  if (e != cudaSuccess) return e;
  std::lock_guard<std::mutex> lk(mu);
  auto it = cache.find(dev);
  if (it == cache.end()) {
    const auto k = sssp::sssp_fd_march_kernel<LOG2L, true>;
    Room r;
    if ((e = cudaFuncSetAttribute(k, cudaFuncAttributeMaxDynamicSharedMemorySize, int(C::SMEM))) != cudaSuccess) return e;
    if ((e = cudaDeviceGetAttribute(&r.sms, cudaDevAttrMultiProcessorCount, dev)) != cudaSuccess) return e;
    if ((e = cudaOccupancyMaxActiveBlocksPerMultiprocessor(&r.solves, k, C::NT, C::SMEM)) != cudaSuccess) return e;
    it = cache.emplace(dev, r).first;
  }
  *out = it->second;
  return cudaSuccess;
}

// Staged tables leave room for S = 4, 2 and 1 solves an SM at L = 512, 1024 and 2048 (read in place: 13, 6 and 3), so
// more of them march in waves.  With k solves an SM, marches in place take about k times, staged ones about
// 0.9 S ceil(k / S) times as long as one more solve in place does: L = 1024, [8/8], 40 steps, in place /
// staged ms: 304 solves 2.11 / 1.66, 400 2.89 / 3.19, 608 3.71 / 3.27, 700 4.48 / 4.84, 912 5.41 / 4.87;
// L = 512: 608 solves 2.09 / 1.65, 640 2.46 / 2.89, 912 2.93 / 3.06, 1216 3.78 / 3.22; L = 2048 staged at every
// count (160 solves 3.66 / 3.20, 456 5.32 / 4.91).  One wave gains at every count.
bool staged(const Room& r, int count) {
  if (r.sms < 1 || r.solves < 1) return false;
  const int k = (count + r.sms - 1) / r.sms, waves = (k + r.solves - 1) / r.solves;
  return waves == 1 || 9LL * r.solves * waves <= 10LL * k;
}

template <int LOG2L>
cudaError_t launch_t(const sssp::SolveDesc* d, int count, cudaStream_t st) {
  using C = sssp::FdCfg<LOG2L>;
  if constexpr (C::STAGEABLE) {
    Room r;
    const cudaError_t e = room_for<LOG2L>(&r);
    if (e != cudaSuccess) return e;
    if (staged(r, count)) {
      sssp::sssp_fd_march_kernel<LOG2L, true><<<count, C::NT, C::SMEM, st>>>(d);
      return cudaGetLastError();
    }
  }
  sssp::sssp_fd_march_kernel<LOG2L, false><<<count, C::NT, 0, st>>>(d);
  return cudaGetLastError();
}

float4 split_ff(std::complex<double> v) {
  const float hr = float(v.real()), hi = float(v.imag());
  return make_float4(hr, hi, float(v.real() - double(hr)), float(v.imag() - double(hi)));
}

}  // namespace

bool supported(int log2L) { return log2L >= sssp::kFdMinLog2 && log2L <= sssp::kFdMaxLog2; }

cudaError_t launch_march(int log2L, const sssp::SolveDesc* d, int count, cudaStream_t st) {
  switch (log2L) {
    case 3: return launch_t<3>(d, count, st);
    case 4: return launch_t<4>(d, count, st);
    case 5: return launch_t<5>(d, count, st);
    case 6: return launch_t<6>(d, count, st);
    case 7: return launch_t<7>(d, count, st);
    case 8: return launch_t<8>(d, count, st);
    case 9: return launch_t<9>(d, count, st);
    case 10: return launch_t<10>(d, count, st);
    case 11: return launch_t<11>(d, count, st);
    case 12: return launch_t<12>(d, count, st);
  }
  return cudaErrorInvalidValue;
}

void factor_node(const double* V, int N, int L, double H, double k0, const std::complex<double>* b, int p,
                 float4* out) {
  using cd = std::complex<double>;
  const double dz = H / double(N + 1), s = 1.0 / ((k0 * dz) * (k0 * dz));
  for (int j = 0; j < p; ++j) {
    float4* tab = out + size_t(j) * L * 3;  // FdEntry = 3 float4 per point
    const cd e = b[j] * s;
    for (int q = 0; q < 3; ++q) tab[q] = make_float4(0.f, 0.f, 0.f, 0.f);  // index 0: the boundary
    cd cprev(0.0, 0.0);
    for (int n = 1; n <= N; ++n) {
      const cd dn = 1.0 + b[j] * (V[n - 1] - 2.0 * s);
      const cd den = (n == 1) ? dn : dn - e * cprev;
      const cd inv = 1.0 / den;
      const cd cp = (n < N) ? e * inv : cd(0.0, 0.0);
      float4* ent = tab + size_t(n) * 3;
      ent[0] = split_ff(inv);
      ent[1] = split_ff(-e * inv);
      ent[2] = split_ff(-cp);
      cprev = cp;
    }
  }
}

}  // namespace sssp_fd
