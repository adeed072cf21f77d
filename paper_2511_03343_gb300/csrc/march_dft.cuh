// SSSP range march on periodic grids (and rigid boundaries, which march their even extension) of M = 512, 1024
// or 2048 points: one solve per CTA of M/8 threads, one complex DFT of M points each way per Neumann term,
// everything else on the thread's own points.
//
// M = 8 Q 8.  Thread (g, i) -- group g < 8 of Q threads, i < Q -- holds the column c = g + 8 i: points and modes
// c + C r, r < 8, C = M/8, of depth and spectral values alike.  A transform is
//   a radix-8 pass over r (output k1, twiddle w_M^{c k1}),
//   an exchange over the block, which gathers row (k1, m2 = c mod 8), m1 = i, in group k1,
//   the Q-point transform of every row as H x 8 (H = Q/8 threads a row), and, once more within the group,
//   a radix-8 pass over m2, whose output k3 of (k1, k2) is point k1 + 8 k2 + C k3: the thread's column again.
// So there is one block barrier a transform; the other exchanges stay inside a group, which a warp holds, and
// every value moves three times through shared memory (the general passes: five, with a barrier each).
#pragma once
#include "march_kernel.cuh"

namespace sssp {

template <int LOG2M>
struct DCfg {
  static constexpr int M = 1 << LOG2M;
  static constexpr int C = M / 8, Q = M / 64, H = Q / 8, NT = M / 8;
  static_assert(H == 1 || H == 2 || H == 4, "512, 1024 or 2048 points");
  // strides of the block exchange (row (k1, m2)), of a group's sub-rows (s, m2) and of its rows m2: the 64-bit
  // accesses of a half-warp fall on different banks (sub-rows: but for one pair)
  static constexpr int QP = Q + 2, SP = 9, ZP = Q + 2;
  static constexpr int X = 64 * QP, XA = H > 1 ? 8 * H * SP : 0, XZ = 8 * ZP;
  // two block exchanges (a warp may be a transform ahead of another's reads), then the groups' areas
  static constexpr int XN = 2 * X + 8 * (XA + XZ);
  static constexpr size_t SMEM = sizeof(float2) * (XN + M);  // and t_0
  static constexpr int MIN_BLOCKS = NT == 256 ? 1 : 65536 / (NT * 168);  // room for 168 registers a thread
};

template <int LOG2M>
struct DThread {
  int g, i, c;
  int m2, h;  // the row (g, m2) and sub-row h of the thread in the middle passes
  __device__ __forceinline__ DThread() {
    constexpr int Q = DCfg<LOG2M>::Q;
    g = int(threadIdx.x) / Q;
    i = int(threadIdx.x) % Q;
    c = g + 8 * i;
    m2 = i & 7;
    h = i >> 3;
  }
};

// twiddles kept in registers: w_M^{c k1}; w_Q^{v s} of the H-point sub-rows (v = h + H vv), hi + lo; w_{8Q}^{m2 k2},
// k2 = h + H w.  wM: the M FP32 roots, then the lo parts of w_Q^j, j < Q.
// The sub-rows' lo parts: a twiddle's FP32 representation error is the same in every transform and adds up over
// the steps, and the extra pass over H points gave these transforms more of it than the general passes have.
// Field error against complex128, 40 steps, [6/6], mean of 128 solves, general passes / all FP32 / sub-rows hi +
// lo: 1024 points 6.35e-7 / 6.60e-7 / 6.11e-7, 2048 7.85e-7 / 8.95e-7 / 6.70e-7.  March of 30 steps: 1024 points 1.73 ->
// 1.78 ms, 2048 points 2.98 -> 2.86 ms (the general passes: 2.25 and 4.48).  hi + lo in the third pass too gives 6.0e-7
// and 6.5e-7, but 2.11 ms at 1024 points (registers spill).
template <int LOG2M>
struct DTw {
  static constexpr int Q = DCfg<LOG2M>::Q, H = DCfg<LOG2M>::H;
  float2 a[7], m[8];
  float4 b[H > 1 ? 8 : 1];
  __device__ __forceinline__ void load(const float2* wM, const DThread<LOG2M>& th) {
#pragma unroll
    for (int k = 1; k < 8; ++k) a[k - 1] = __ldg(wM + th.c * k);
#pragma unroll
    for (int w = 0; w < 8; ++w) m[w] = __ldg(wM + 8 * th.m2 * (th.h + H * w));
    if constexpr (H > 1) {
#pragma unroll
      for (int vv = 0; vv < 8 / H; ++vv)
#pragma unroll
        for (int s = 0; s < H; ++s) {
          const int j = (th.h + H * vv) * s;  // below 8 H = Q
          const float2 hi = __ldg(wM + 64 * j), lo = __ldg(wM + DCfg<LOG2M>::M + j);
          b[vv * H + s] = make_float4(hi.x, hi.y, lo.x, lo.y);
        }
    }
  }
};

// Forward DFT of M points: a[r] = point c + C r on input and output.
template <int LOG2M>
__device__ __forceinline__ void dft_regs(float2 (&a)[8], const DTw<LOG2M>& tw, const DThread<LOG2M>& th, float2* x, int& ph) {
  using K = DCfg<LOG2M>;
  constexpr int H = K::H;
  float2* X = x + (ph & 1) * K::X;
  float2* A = x + 2 * K::X + th.g * (K::XA + K::XZ);
  float2* Z = A + K::XA;
  ++ph;
  dft8(a);
#pragma unroll
  for (int k = 0; k < 8; ++k) X[(k * 8 + th.g) * K::QP + th.i] = k ? cmul(a[k], tw.a[k ? k - 1 : 0]) : a[0];
  __syncthreads();
  const float2* s = X + (th.g * 8 + th.m2) * K::QP;
  if constexpr (H == 1) {
#pragma unroll
    for (int j = 0; j < 8; ++j) a[j] = s[j];
  } else {
    // points m1 = 8 u + v, u < H, of v = h + H vv
#pragma unroll
    for (int vv = 0; vv < 8 / H; ++vv) {
      const int v = th.h + H * vv;
      float2 b[H];
#pragma unroll
      for (int u = 0; u < H; ++u) b[u] = s[8 * u + v];
      if constexpr (H == 2) dft2(b[0], b[1]);
      else dft4(b[0], b[1], b[2], b[3]);
#pragma unroll
      for (int q = 0; q < H; ++q) A[(q * 8 + th.m2) * K::SP + v] = q ? ffmul(tw.b[vv * H + q], b[q]) : b[0];
    }
    __syncwarp();
#pragma unroll
    for (int j = 0; j < 8; ++j) a[j] = A[(th.h * 8 + th.m2) * K::SP + j];
  }
  dft8(a);
#pragma unroll
  for (int w = 0; w < 8; ++w) Z[th.m2 * K::ZP + th.h + H * w] = (H == 1 && w == 0) ? a[0] : cmul(a[w], tw.m[w]);
  __syncwarp();
#pragma unroll
  for (int j = 0; j < 8; ++j) a[j] = Z[j * K::ZP + th.i];
  dft8(a);
}

// A stage's tables, read once a stage from the L2: volatile keeps the loads together, in program order
__device__ __forceinline__ float4 ldv4(const float4* p) {
  float4 v;
  asm volatile("ld.global.nc.v4.f32 {%0, %1, %2, %3}, [%4];" : "=f"(v.x), "=f"(v.y), "=f"(v.z), "=f"(v.w) : "l"(p));
  return v;
}
__device__ __forceinline__ float2 ldv2(const float2* p) {
  float2 v;
  asm volatile("ld.global.nc.v2.f32 {%0, %1}, [%2];" : "=f"(v.x), "=f"(v.y) : "l"(p));
  return v;
}

// The march: blockIdx.x selects the solve.  (2048 points, one solve, 30 steps, the general kernel
// against this one: 4.48 -> 2.86 ms; 152 solves 5.46 -> 3.33, 304 9.29 -> 6.46.)
template <int LOG2M, bool CPLX>
__global__ void __launch_bounds__(DCfg<LOG2M>::NT, DCfg<LOG2M>::MIN_BLOCKS)
    sssp_march_dft_kernel(const SolveDesc* __restrict__ descs, const float2* __restrict__ wM) {
  using K = DCfg<LOG2M>;
  constexpr int M = K::M, C = K::C, NT = K::NT, NWARP = NT / 32;
  extern __shared__ __align__(16) unsigned char smem_raw[];
  __shared__ SolveDesc d;
  __shared__ float2 red[NWARP];
  const int t = threadIdx.x, lane = t & 31, warp = t >> 5;
  const DThread<LOG2M> th;
  float2* x = reinterpret_cast<float2*>(smem_raw);
  float2* t0s = x + K::XN + t;  // t_0, value i at i NT
  int ph = 0;
  {
    const int* src = reinterpret_cast<const int*>(descs + blockIdx.x);
    int* dst = reinterpret_cast<int*>(&d);
    for (int i = t; i < int(sizeof(SolveDesc) / sizeof(int)); i += NT) dst[i] = src[i];
  }
  DTw<LOG2M> tw;
  tw.load(wM, th);
  __syncthreads();
  if (d.terms > 1 && blockIdx.y > 0) return;  // only TL rows without Neumann terms are split (march_kernel.cuh)

  const float out_scale = 1.0f / float(M);
  const bool iso = d.terms <= 1;
  const float tol2f = float(d.tol2);
  int status = kStatusOk;
  unsigned int ndst = 0;
  int nrec = 0;
  int node = d.node0;
  double next_r = (node + 1 < d.nodes) ? d.node_r[node + 1] : 1e300;
  float vr[8], vi[8];
  auto load_v = [&](int nd) {
#pragma unroll
    for (int i = 0; i < 8; ++i) {
      vr[i] = __ldg(d.V + (size_t)nd * M + th.c + C * i);
      if constexpr (CPLX) vi[i] = __ldg(d.Vi + (size_t)nd * M + th.c + C * i);
    }
  };
  if (!iso) load_v(node);
  // x_n = sum_k X_k e^{+2 pi i n k/M} = conj(DFT(conj X)); a holds the conjugates, in and out
  auto inverse = [&](float2 (&a)[8]) { dft_regs<LOG2M>(a, tw, th, x, ph); };

  float2 y[8];
#pragma unroll
  for (int i = 0; i < 8; ++i) y[i] = d.yhat[th.c + C * i];
  auto depth = [&](float2 (&a)[8]) {  // the envelope, conjugated
#pragma unroll
    for (int i = 0; i < 8; ++i) a[i] = make_float2(out_scale * y[i].x, -out_scale * y[i].y);
    inverse(a);
    ++ndst;
  };
  auto record = [&](int s) {
    float2 a[8];
    depth(a);
    const float lr = float(10.0 * log10(d.r0 + double(s + 1) * d.dr));
    float* row = d.tl + (size_t)(d.rec0 + nrec) * d.N + th.c;
#pragma unroll
    for (int i = 0; i < 8; ++i) row[C * i] = fmaf(-10.f, log10f(cabs2(a[i])), lr);
  };

  for (int s = 0; s < d.steps && status == kStatusOk; ++s) {
    bool mine = true;
    if (iso) {
#pragma unroll
      for (int i = 0; i < 8; ++i) y[i] = ffmul(__ldg(d.G + th.c + C * i), y[i]);
      mine = nrec % int(gridDim.y) == int(blockIdx.y);
    } else {
      const double rmid = d.r0 + (double(s) + 0.5) * d.dr;
      if (rmid >= next_r) {  // advance to the node in force at this step's midpoint
        while (node + 1 < d.nodes && d.node_r[node + 1] <= rmid) ++node;
        next_r = (node + 1 < d.nodes) ? d.node_r[node + 1] : 1e300;
        load_v(node);
      }
      for (int j = 0; j < d.p && status == kStatusOk; ++j) {
        float2 acc[8], a[8], Bj[8];
        {
          const float2 *A = d.A + (size_t)j * M + th.c, *B = d.B + (size_t)j * M + th.c;
#pragma unroll
          for (int i = 0; i < 8; ++i) a[i] = ldv2(A + C * i);
#pragma unroll
          for (int i = 0; i < 8; ++i) Bj[i] = ldv2(B + C * i);
        }
#pragma unroll
        for (int i = 0; i < 8; ++i) {
          a[i] = cmul(a[i], y[i]);
          t0s[i * NT] = a[i];
          a[i].y = -a[i].y;
          acc[i] = make_float2(0.f, 0.f);
        }
        float first = 0.f;
        for (int m = 1; m < d.terms; ++m) {
          inverse(a);  // t_{m-1} in depth space
          if (m > 1) {  // the stop test of t_{m-1}, whose partials the transform's barriers published
            float snt = 0.f, snw = 0.f;
#pragma unroll
            for (int w = 0; w < NWARP; ++w) {  // the same order in every thread: a uniform decision
              snt += red[w].x;
              snw += red[w].y;
            }
            if (!isfinite(snt) || !isfinite(snw)) {
              status = kStatusNumeric;
              break;
            }
            if (m == 2) first = snt;
            else if (first > 0.f && snt > 1e8f * first) {
              status = kStatusDiverged;
              break;
            }
            if (neumann_stop_fast(snt, snw, d.tol2, tol2f)) break;
          }
          ++ndst;
#pragma unroll
          for (int i = 0; i < 8; ++i) {
            const float2 v = make_float2(a[i].x, -a[i].y);
            if constexpr (CPLX) a[i] = cmul(make_float2(vr[i], vi[i]), v);
            else a[i] = vr[i] * v;
          }
          dft_regs<LOG2M>(a, tw, th, x, ph);  // T(V t_{m-1})
          ++ndst;
          float nt = 0.f, nw = 0.f;
#pragma unroll
          for (int i = 0; i < 8; ++i) {
            a[i] = cmul(Bj[i], a[i]);
            acc[i] = acc[i] + a[i];
            nt += cabs2(a[i]);
            nw += cabs2(t0s[i * NT] + acc[i]);
            a[i].y = -a[i].y;
          }
          if (m == d.terms - 1) break;
#pragma unroll
          for (int o = 16; o > 0; o >>= 1) {
            nt += __shfl_xor_sync(0xffffffffu, nt, o);
            nw += __shfl_xor_sync(0xffffffffu, nw, o);
          }
          if (lane == 0) red[warp] = make_float2(nt, nw);
        }
        {
          const float4* R = d.R + (size_t)j * M + th.c;
          const float2 bj = d.beta[j];
          float4 r[8];
#pragma unroll
          for (int i = 0; i < 8; ++i) r[i] = ldv4(R + C * i);
#pragma unroll
          for (int i = 0; i < 8; ++i) y[i] = ffmul(r[i], y[i]) + cmul(bj, acc[i]);
        }
      }
      if (status != kStatusOk) break;
    }
    const long long gs = d.step0 + s + 1;
    if (d.tl_every > 0 && gs % d.tl_every == 0) {
      if (mine) record(s);
      ++nrec;
    }
  }
  if (iso && gridDim.y > 1) {  // the last CTA to finish writes the state (see sssp_march_kernel)
    __shared__ bool last;
    __syncthreads();
    if (t == 0) {
      __threadfence();
      last = atomicInc(reinterpret_cast<unsigned*>(d.ndst + 1), gridDim.y - 1) == gridDim.y - 1;
      if (!last) atomicAdd(d.ndst, (unsigned long long)ndst);
    }
    __syncthreads();
    if (!last) return;
  }
  float2 a[8];
  depth(a);  // physical envelope for pe_read_field
#pragma unroll
  for (int i = 0; i < 8; ++i) {
    d.yhat[th.c + C * i] = y[i];
    d.field[th.c + C * i] = make_float2(a[i].x, -a[i].y);
  }
  if (t == 0) {
    if (status != kStatusOk) atomicMax(d.status, status);
    atomicAdd(d.ndst, (unsigned long long)ndst);
  }
}

}  // namespace sssp
