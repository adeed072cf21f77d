// The DST-I with the modes split by parity over two halves of a CTA's warps (Dirichlet grids, L = N + 1 in
// [512, 4096]), and the range march of one solve per CTA built on it (L = 2048 and 4096).
//
// With M = L/2 the DST-I of x splits into two transforms of M points that never mix modes:
//   O_n = sum_k S_{2k+1} sin(pi (2k+1) n/L),  E_n = sum_k S_{2k} sin(pi k n/M),   n in [0, M]
//   x_n = O_n + E_n,  x_{L-n} = O_n - E_n,
// and its transpose (the DST-I matrix is symmetric).  So a Neumann term -- to depth, times V, back
// to the modes -- is, per half, one M-point complex FFT each way, and the halves meet once, at
// the depth points:
//   v_n = P_n O_n + D_n E_n  (odd half),  u_n = D_n O_n + P_n E_n  (even half),
//   P_n = V_n + V_{L-n},  D_n = V_n - V_{L-n}.
// The odd half (a type-II/III sine transform) takes r_j = S_{4j+1} (j < M/2), r_{M-1-j} = -S_{4j+3}:
//   g = FFT_M(r),  with c_n = e^{-i pi n/L}, p = c_n g_n, q = conj(c_n) g_{M-n}:
//   2 O_n = i (p - q),  2 O_{M-n} = p + q;
//   back: G_n = c_n (v_{M-n} + i v_n)/2, G_{M-n} = conj(c_n) (v_{M-n} - i v_n)/2, r = FFT_M(G).
// The even half (a DST-I of M - 1 points z_k = S_{2k}, odd about 0 and M) takes
//   y_m = z_{2m} + (z_{2m+1} - z_{2m-1}), y_{M-m} = -z_{2m} + (z_{2m+1} - z_{2m-1}):
//   f = FFT_M(y),  with b_n = 1/(2 sin(pi n/M)):
//   4 E_n = b_n (f_n + f_{M-n}) + i (f_n - f_{M-n}),  4 E_{M-n} = b_n (f_n + f_{M-n}) - i (f_n - f_{M-n});
//   back: Y_n = (b_n (u_n + u_{M-n}) + i (u_n - u_{M-n}))/4 (Y_{M-n} with -i), y = FFT_M(Y),
//   S_{4m} = y_m - y_{M-m},  S_{4m+2} = (y_m + y_{M-m}) - (y_{m+1} + y_{M-m-1}).
// No prefix scan over the modes is left, and neither half waits for the other but at the depth points.
//
// What bounds it: the chain of dependent passes (3 radix passes and 2 exchanges a transform, one block
// barrier a Neumann term) at a few warps a scheduler; then the shared-memory pipe.  8 points a thread: with 16, one solve of L = 2048 took 4200 cycles a transform
// (2.07 GHz), with 8 3040; the scan form it replaced 4600 (37 solves of N = 2047, complex n^2, [6/6],
// 40 steps: 9.1 -> 5.8 ms).  Complex n^2 leaves room for one solve of L = 2048 an SM (117 KB; the scan form
// held two): 304 solves, 20 steps, the scan form against this one 8.4 -> 6.3 ms, real n^2 7.9 -> 4.9.
// Its FP32 error is smaller too (no sums over L/2 modes): 3.1e-6 -> 1.2e-6
// against complex128 there.
#pragma once
#include "march_dft.cuh"  // ldv2, ldv4
#include "march_kernel.cuh"

namespace sssp {

// Tables of one size (device, FP64 rounded once to FP32)
struct EoTabs {
  const float2* wM;  // e^{-2 pi i e/M}, e in [0, M)
  const float2* cL;  // e^{-i pi n/L}, n in [0, M]
  const float* beta; // 1/(2 sin(pi n/M)), n in [1, M); 0 at n = 0
};

// M = 8 Q 8: two radix-8 passes around a pass of radix Q.  A thread holds one column of the first and
// last pass (points c + C r, C = M/8); the threads of the columns c and C - c are 16 lanes apart in one
// warp, so the point M - n of every point n is a shuffle away (columns 0 and C/2 mirror themselves).
template <int LOG2L>
struct ECfg {
  static constexpr int L = 1 << LOG2L;
  static constexpr int M = L / 2;
  static constexpr int C = M / 8;
  static constexpr int Q = M / 64;
  static constexpr int HL = C;       // threads per half, 8 points each
  static constexpr int NT = 2 * HL;
  static constexpr int W = HL / 32;  // warps per half
  // exchange 1: point n2 of the radix-8 column pass's row k1 at k1 S1 + n2; exchange 2: output c' of
  // the row (k1, m2) at m2 S2 + c'.  The strides keep every half-warp's 64-bit accesses conflict-free.
  static constexpr int S1 = C + 8, S2 = C + 2;
  static constexpr int X1 = 8 * S1, X2 = 8 * S2;
  // per half X1 and X2; the depth exchange (4 slots of two values a thread, both halves, double
  // buffered); t_0; the V coefficients
  static constexpr size_t SMEM = sizeof(float2) * (2 * (X1 + X2) + 2 * 2 * M + 8 * NT) + sizeof(float4) * 4 * NT;
  static constexpr size_t SMEM_CPLX = SMEM + sizeof(float4) * 4 * NT;
  static constexpr int MIN_BLOCKS = 65536 / (NT * 128);
};

template <int LOG2L>
struct EoThread {
  static constexpr int C = ECfg<LOG2L>::C, M = ECfg<LOG2L>::M;
  int e;    // 0: even modes, 1: odd modes
  int t;    // thread within the half
  int c;    // its column
  int src;  // lane of the column C - c
  bool z;   // column 0
  __device__ __forceinline__ EoThread() {
    e = int(threadIdx.x) / ECfg<LOG2L>::HL;
    t = int(threadIdx.x) % ECfg<LOG2L>::HL;
    const int lane = t & 31, i = 16 * (t >> 5) + (lane & 15);
    c = lane < 16 ? i : (i ? C - i : C / 2);
    src = i ? lane ^ 16 : lane;
    z = c == 0;
  }
  __device__ __forceinline__ int slot(int i) const { return c + C * i; }  // first index m of slot i < 4
  // mode of spectral value i, and its sign in the saved state.  Even half: i < 4 the mode 4 m of slot
  // i, else 4 m + 2 of slot i - 4.  Odd half: r_j of column entry i.
  __device__ __forceinline__ int mode(int i) const {
    const int m = c + C * (i & 3), j = c + C * i;
    return e == 0 ? 4 * m + (i < 4 ? 0 : 2) : (i < 4 ? 4 * j + 1 : 4 * (M - 1 - j) + 3);
  }
  __device__ __forceinline__ float sign(int i) const { return (e && i >= 4) ? -1.f : 1.f; }
};

template <int LOG2L>
__device__ __forceinline__ void half_sync(int e) {
  if constexpr (ECfg<LOG2L>::W == 1) __syncwarp();
  else if (e) asm volatile("bar.sync 2, %0;" ::"n"(ECfg<LOG2L>::HL) : "memory");
  else asm volatile("bar.sync 1, %0;" ::"n"(ECfg<LOG2L>::HL) : "memory");
}

// twiddles of the FFT a thread keeps in registers: after the first pass w_M^{c k1}, after the middle
// pass w_{8Q}^{m2 k2} (its outputs k2 = H q + h, H = Q/8 threads a row, for Q >= 8)
template <int LOG2L>
struct EoTw {
  static constexpr int Q = ECfg<LOG2L>::Q, H = Q >= 8 ? Q / 8 : 1, NM = Q >= 8 ? 8 : 4;
  float2 a[7], m[NM];
  __device__ __forceinline__ void load(const EoTabs& tb, const EoThread<LOG2L>& th) {
#pragma unroll
    for (int k = 1; k < 8; ++k) a[k - 1] = __ldg(tb.wM + th.c * k);
    const int m2 = th.t & 7, h = th.t >> 6;
#pragma unroll
    for (int q = 0; q < NM; ++q) m[q] = __ldg(tb.wM + 8 * m2 * (Q >= 8 ? H * q + h : q));
  }
};

// w_{8H}^{h j} (hi + lo), the rotation of a row's thread h > 0 before its 8-point transform
template <int H>
__device__ __forceinline__ float2 eo_rot(int h, int j, float2 v) {
  static_assert(H == 2 || H == 4, "threads per row");
  // cos(pi i/16), i = 0..8
  constexpr double W[9] = {1.0, 0.98078528040323044913, 0.92387953251128675613, 0.83146961230254523708,
                           0.70710678118654752440, 0.55557023301960222474, 0.38268343236508977173,
                           0.19509032201612826785, 0.0};
  // e^{-i pi g/16}
  auto rot = [&](int g) {
    const int o = g & 7, quad = (g >> 3) & 3;  // e^{-i pi g/16} = (-i)^quad (cos - i sin)(pi o/16)
    const double c = W[o], sn = W[8 - o];
    const double re = quad == 0 ? c : (quad == 1 ? -sn : (quad == 2 ? -c : sn));
    const double im = quad == 0 ? -sn : (quad == 1 ? -c : (quad == 2 ? sn : c));
    const float rh = float(re), ih = float(im);
    return ffmul(make_float4(rh, ih, float(re - double(rh)), float(im - double(ih))), v);
  };
  if constexpr (H == 2) return rot(2 * j);
  else return h == 1 ? rot(j) : (h == 2 ? rot(2 * j) : rot(3 * j));
}

// Forward FFT of M points over the threads of a half: entry r of column c is point c + C r, on input
// and output.
template <int LOG2L>
__device__ __forceinline__ void eo_fft(float2 (&a)[8], const EoTw<LOG2L>& tw, const EoThread<LOG2L>& th, float2* x1, float2* x2) {
  using K = ECfg<LOG2L>;
  constexpr int H = EoTw<LOG2L>::H;
  dft8(a);
  x1[th.c] = a[0];
#pragma unroll
  for (int k = 1; k < 8; ++k) x1[k * K::S1 + th.c] = cmul(a[k], tw.a[k - 1]);
  half_sync<LOG2L>(th.e);
  const int k1 = (th.t & 63) >> 3, m2 = th.t & 7;
  const float2* s = x1 + k1 * K::S1 + m2;
  float2* d = x2 + m2 * K::S2 + k1;
  if constexpr (K::Q == 4) {  // 32 threads, two rows each (k1 and k1 + 4)
    float2 b0[4], b1[4];
#pragma unroll
    for (int j = 0; j < 4; ++j) {
      b0[j] = s[8 * j];
      b1[j] = s[4 * K::S1 + 8 * j];
    }
    dft4(b0[0], b0[1], b0[2], b0[3]);
    dft4(b1[0], b1[1], b1[2], b1[3]);
#pragma unroll
    for (int k = 0; k < 4; ++k) {
      d[8 * k] = k ? cmul(b0[k], tw.m[k]) : b0[0];
      d[8 * k + 4] = k ? cmul(b1[k], tw.m[k]) : b1[0];
    }
  } else {
    const int h = th.t >> 6;  // uniform over a warp
    if constexpr (H == 1) {
#pragma unroll
      for (int j = 0; j < 8; ++j) a[j] = s[8 * j];
    } else if constexpr (H == 2) {
#pragma unroll
      for (int j = 0; j < 8; ++j) {
        const float2 p = s[8 * j], q = s[8 * (j + 8)];
        a[j] = h ? p - q : p + q;
      }
    } else {
#pragma unroll
      for (int j = 0; j < 8; ++j) {
        const float2 p0 = s[8 * j], p1 = s[8 * (j + 8)], p2 = s[8 * (j + 16)], p3 = s[8 * (j + 24)];
        if (h == 0) a[j] = (p0 + p2) + (p1 + p3);
        else if (h == 2) a[j] = (p0 + p2) - (p1 + p3);
        else {
          const float2 u = p0 - p2, v = p1 - p3;
          a[j] = h == 1 ? make_float2(u.x + v.y, u.y - v.x) : make_float2(u.x - v.y, u.y + v.x);
        }
      }
    }
    if constexpr (H > 1) {
      if (h) {
#pragma unroll
        for (int j = 1; j < 8; ++j) a[j] = eo_rot<H>(h, j, a[j]);
      }
    }
    dft8(a);
#pragma unroll
    for (int q = 0; q < 8; ++q) d[8 * (H * q + h)] = (H == 1 && q == 0) ? a[0] : cmul(a[q], tw.m[q]);
  }
  half_sync<LOG2L>(th.e);
#pragma unroll
  for (int r = 0; r < 8; ++r) a[r] = x2[r * K::S2 + th.c];
  dft8(a);
}

__device__ __forceinline__ float2 sel2(bool c, float2 x, float2 y) { return make_float2(c ? x.x : y.x, c ? x.y : y.y); }
__device__ __forceinline__ float2 shfl2(float2 v, int src) {
  return make_float2(__shfl_sync(0xffffffffu, v.x, src), __shfl_sync(0xffffffffu, v.y, src));
}

// column -> slots: p[i] = point m of slot i, q[i] = point M - m (slot 0 of column 0: q = point 0); the
// point M/2 (column 0's a[4]) has no slot.
template <int LOG2L>
__device__ __forceinline__ void to_slots(const EoThread<LOG2L>& th, const float2 (&a)[8], float2 (&p)[4], float2 (&q)[4]) {
#pragma unroll
  for (int i = 0; i < 4; ++i) {
    p[i] = a[i];
    q[i] = sel2(th.z, a[(8 - i) & 7], shfl2(a[7 - i], th.src));
  }
}
// slots -> column; x is the point M/2 (used by column 0)
template <int LOG2L>
__device__ __forceinline__ void to_cols(const EoThread<LOG2L>& th, const float2 (&p)[4], const float2 (&q)[4], float2 x, float2 (&a)[8]) {
#pragma unroll
  for (int i = 0; i < 4; ++i) {
    a[i] = p[i];
    a[7 - i] = sel2(th.z, i < 3 ? q[(i + 1) & 3] : x, shfl2(q[i], th.src));
  }
}

__device__ __forceinline__ float2 add_pi(float2 x, float2 y) { return make_float2(x.x - y.y, x.y + y.x); }  // x + i y
__device__ __forceinline__ float2 add_ni(float2 x, float2 y) { return make_float2(x.x + y.y, x.y - y.x); }  // x - i y
__device__ __forceinline__ float2 cmulc(float2 a, float2 b) {                                              // a conj(b)
  return make_float2(fmaf(a.x, b.x, a.y * b.y), fmaf(a.y, b.x, -a.x * b.y));
}
__device__ __forceinline__ float2 mul_sqrt2(float2 x) {  // hi + lo, like the butterflies' constants
  constexpr double R2 = 1.41421356237309504880;
  constexpr float h = float(R2), l = float(R2 - double(float(R2)));
  return make_float2(ff_mul(h, l, x.x), ff_mul(h, l, x.y));
}

// per-thread constants of the pair steps: c_n of the slots (odd half), b_n in x (even half)
struct EoPair {
  float2 c[4];
};

// Spectral values (mode(i) order) -> depth: 2 O (odd half) or 4 E (even half), p at m and q at M - m of
// every slot, x at M/2 (column 0).
template <int LOG2L>
__device__ __forceinline__ void eo_inverse(const float2 (&sp)[8], float2 (&p)[4], float2 (&q)[4], float2& x,
                                           const EoTw<LOG2L>& tw, const EoPair& pc, const EoThread<LOG2L>& th,
                                           float2* x1, float2* x2) {
  using K = ECfg<LOG2L>;
  float2 a[8];
  if (th.e) {
#pragma unroll
    for (int r = 0; r < 8; ++r) a[r] = sp[r];
  } else {
    // z_{2m+1} of every m at index m + 1; z_{-1} = -z_1
#pragma unroll
    for (int i = 0; i < 4; ++i) x2[th.slot(i) + 1] = sp[4 + i];
    if (th.z) x2[0] = make_float2(-sp[4].x, -sp[4].y);
    half_sync<LOG2L>(0);
#pragma unroll
    for (int i = 0; i < 4; ++i) {
      const float2 d = sp[4 + i] - x2[th.slot(i)];
      p[i] = d + sp[i];
      q[i] = d - sp[i];
    }
    x = make_float2(0.f, 0.f);
    if (th.z) x = -2.f * x2[K::M / 2];
    to_cols<LOG2L>(th, p, q, x, a);
  }
  eo_fft<LOG2L>(a, tw, th, x1, x2);
  float2 p0[4], q0[4];
  to_slots<LOG2L>(th, a, p0, q0);
  if (th.e) {
    x = mul_sqrt2(a[4]);
#pragma unroll
    for (int i = 0; i < 4; ++i) {
      const float2 u = cmul(pc.c[i], p0[i]), v = cmulc(q0[i], pc.c[i]);
      p[i] = make_float2(v.y - u.y, u.x - v.x);  // i (u - v)
      q[i] = u + v;
    }
  } else {
    x = a[4];
#pragma unroll
    for (int i = 0; i < 4; ++i) {
      const float bt = pc.c[i].x;
      const float2 u = p0[i] + q0[i], d = p0[i] - q0[i];
      p[i] = make_float2(fmaf(bt, u.x, -d.y), fmaf(bt, u.y, d.x));
      q[i] = make_float2(fmaf(bt, u.x, d.y), fmaf(bt, u.y, -d.x));
    }
  }
}

// Depth values of the half (slots: p at m, q at M - m; x at M/2), scaled by 1/2 (odd) or 1/4 (even),
// -> spectral values.
template <int LOG2L>
__device__ __forceinline__ void eo_forward(const float2 (&p)[4], const float2 (&q)[4], float2 x, float2 (&sp)[8],
                                           const EoTw<LOG2L>& tw, const EoPair& pc, const EoThread<LOG2L>& th,
                                           float2* x1, float2* x2) {
  using K = ECfg<LOG2L>;
  float2 a[8], p0[4], q0[4];
  if (th.e) {
    x = mul_sqrt2(x);
#pragma unroll
    for (int i = 0; i < 4; ++i) {
      p0[i] = cmul(pc.c[i], add_pi(q[i], p[i]));
      q0[i] = cmulc(add_ni(q[i], p[i]), pc.c[i]);
    }
  } else {
#pragma unroll
    for (int i = 0; i < 4; ++i) {
      const float bt = pc.c[i].x;
      const float2 u = p[i] + q[i], d = p[i] - q[i];
      p0[i] = make_float2(fmaf(bt, u.x, -d.y), fmaf(bt, u.y, d.x));
      q0[i] = make_float2(fmaf(bt, u.x, d.y), fmaf(bt, u.y, -d.x));
    }
  }
  to_cols<LOG2L>(th, p0, q0, x, a);
  eo_fft<LOG2L>(a, tw, th, x1, x2);
  if (th.e) {
#pragma unroll
    for (int r = 0; r < 8; ++r) sp[r] = a[r];
  } else {
    to_slots<LOG2L>(th, a, p0, q0);
    // y_m + y_{M-m} of every m in [0, M/2] at index m
#pragma unroll
    for (int i = 0; i < 4; ++i) {
      sp[i] = p0[i] - q0[i];
      sp[4 + i] = p0[i] + q0[i];
      x1[th.slot(i)] = sp[4 + i];
    }
    if (th.z) x1[K::M / 2] = 2.f * a[4];
    half_sync<LOG2L>(0);
#pragma unroll
    for (int i = 0; i < 4; ++i) sp[4 + i] = sp[4 + i] - x1[th.slot(i) + 1];
  }
}

// ---------------------------------------------------------------------------------------
// The march: blockIdx.x selects the solve.
// ---------------------------------------------------------------------------------------
template <int LOG2L, bool CPLX>
__global__ void __launch_bounds__(ECfg<LOG2L>::NT, ECfg<LOG2L>::MIN_BLOCKS)
    sssp_march_eo_kernel(const SolveDesc* __restrict__ descs, const EoTabs tb) {
  using K = ECfg<LOG2L>;
  constexpr int L = K::L, M = K::M, NT = K::NT, HL = K::HL, NWARP = NT / 32;
  extern __shared__ __align__(16) unsigned char smem_raw[];
  __shared__ SolveDesc d;
  __shared__ float2 red[2][NWARP];  // norm partials per warp, double buffered like the exchange
  __shared__ float2 mid[2][2];      // the point M/2 of both halves
  const int t = threadIdx.x, lane = t & 31, warp = t >> 5;
  const EoThread<LOG2L> th;
  const int e = th.e;
  float2* x1 = reinterpret_cast<float2*>(smem_raw) + e * (K::X1 + K::X2);
  float2* x2 = x1 + K::X1;
  float4* ex = reinterpret_cast<float4*>(reinterpret_cast<float2*>(smem_raw) + 2 * (K::X1 + K::X2));  // [buf][half][slot][thread]
  float4* cf = ex + 2 * 2 * 4 * HL + t;  // V coefficients, slot i at i NT
  float4* cfi = cf + 4 * NT;              // their imaginary parts (CPLX)
  float2* t0s = reinterpret_cast<float2*>(cf - t + (CPLX ? 8 : 4) * NT) + t;  // t_0, value i at i NT
  {
    const int* src = reinterpret_cast<const int*>(descs + blockIdx.x);
    int* dst = reinterpret_cast<int*>(&d);
    for (int i = t; i < int(sizeof(SolveDesc) / sizeof(int)); i += NT) dst[i] = src[i];
  }
  EoTw<LOG2L> tw;
  tw.load(tb, th);
  EoPair pc;
#pragma unroll
  for (int i = 0; i < 4; ++i) pc.c[i] = e ? __ldg(tb.cL + th.slot(i)) : make_float2(__ldg(tb.beta + th.slot(i)), 0.f);
  __syncthreads();

  const float out_scale = 2.0f / float(L);
  const bool iso = d.terms <= 1;
  const float tol2f = float(d.tol2);
  int status = kStatusOk;
  unsigned int ndst = 0;
  int nrec = 0, buf = 0;
  int node = d.node0;
  double next_r = (node + 1 < d.nodes) ? d.node_r[node + 1] : 1e300;

  // (own, other) coefficients of slot i at m (x, y) and M - m (z, w): the half's depth value is
  // own * mine + other * theirs, P/4 and D/8 (odd half), P/16 and D/8 (even half)
  float2 cmid = make_float2(0.f, 0.f), cmidi = cmid;  // the same at M/2
  auto coef = [&](const float* V, int n) {
    const float v = V[n], w = n ? V[L - n] : 0.f;
    return make_float2((e ? 0.25f : 0.0625f) * (v + w), 0.125f * (v - w));
  };
  auto load_v = [&](int nd) {
    const float* V = d.V + (size_t)nd * L;
#pragma unroll
    for (int i = 0; i < 4; ++i) {
      const float2 c0 = coef(V, th.slot(i)), c1 = coef(V, M - th.slot(i));
      cf[i * NT] = make_float4(c0.x, c0.y, c1.x, c1.y);
    }
    cmid = coef(V, M / 2);
    if constexpr (CPLX) {
      const float* Vi = d.Vi + (size_t)nd * L;
#pragma unroll
      for (int i = 0; i < 4; ++i) {
        const float2 c0 = coef(Vi, th.slot(i)), c1 = coef(Vi, M - th.slot(i));
        cfi[i * NT] = make_float4(c0.x, c0.y, c1.x, c1.y);
      }
      cmidi = coef(Vi, M / 2);
    }
  };
  if (!iso) load_v(node);

  // publish this half's depth values for the other half
  auto put = [&](const float2 (&p)[4], const float2 (&q)[4], float2 x) {
    float4* o = ex + ((buf * 2 + e) * 4) * HL + th.t;
#pragma unroll
    for (int i = 0; i < 4; ++i) o[i * HL] = make_float4(p[i].x, p[i].y, q[i].x, q[i].y);
    if (th.z) mid[buf][e] = x;
  };
  // a depth row: out(n, x_n) for the points of this thread (odd half n <= M, even half n > M)
  auto emit = [&](const float2 (&p)[4], const float2 (&q)[4], float2 x, auto&& out) {
    put(p, q, x);
    __syncthreads();
    const float4* o = ex + ((buf * 2 + 1 - e) * 4) * HL + th.t;
    const float ho = e ? 0.5f : -0.25f, he = e ? 0.25f : 0.5f;  // own, other weight
#pragma unroll
    for (int i = 0; i < 4; ++i) {
      const float4 w = o[i * HL];
      const int m = th.slot(i);
      const float2 u = make_float2(fmaf(ho, p[i].x, he * w.x), fmaf(ho, p[i].y, he * w.y));
      const float2 v = make_float2(fmaf(ho, q[i].x, he * w.z), fmaf(ho, q[i].y, he * w.w));
      if (e) {
        out(m, m ? u : make_float2(0.f, 0.f));
        out(M - m, v);
      } else if (m) {
        out(L - m, u);
        out(M + m, v);
      }
    }
    if (th.z) {
      const float2 w = mid[buf][1 - e];
      out(e ? M / 2 : L - M / 2, make_float2(fmaf(ho, x.x, he * w.x), fmaf(ho, x.y, he * w.y)));
    }
    buf ^= 1;
  };

  float2 y[8];  // the state of the thread's modes, kept in the plan's array inside a stage
#pragma unroll
  for (int i = 0; i < 8; ++i) y[i] = th.sign(i) * d.yhat[th.mode(i)];
  auto record = [&](int s) {
    float2 o[8], p[4], q[4], x;
#pragma unroll
    for (int i = 0; i < 8; ++i) o[i] = out_scale * y[i];
    eo_inverse<LOG2L>(o, p, q, x, tw, pc, th, x1, x2);
    const float lr = float(10.0 * log10(d.r0 + double(s + 1) * d.dr));
    float* row = d.tl + (size_t)(d.rec0 + nrec) * d.N;
    emit(p, q, x, [&](int n, float2 u) {
      if (n >= 1) row[n - 1] = fmaf(-10.f, log10f(cabs2(u)), lr);
    });
    ++ndst;
    ++nrec;
  };

  for (int s = 0; s < d.steps && status == kStatusOk; ++s) {
    if (iso) {  // V ignored: the step is the diagonal multiply by G = prod_j R_j
#pragma unroll
      for (int i = 0; i < 8; ++i) y[i] = ffmul(__ldg(d.G + th.mode(i)), y[i]);
    } else {
      const double rmid = d.r0 + (double(s) + 0.5) * d.dr;
      if (rmid >= next_r) {  // advance to the node in force at this step's midpoint
        while (node + 1 < d.nodes && d.node_r[node + 1] <= rmid) ++node;
        next_r = (node + 1 < d.nodes) ? d.node_r[node + 1] : 1e300;
        load_v(node);  // the coefficients are the thread's own
      }
      for (int j = 0; j < d.p && status == kStatusOk; ++j) {
        float2 acc[8], tp[8], Bj[8], p[4], q[4], x;
        {
          const float2 *A = d.A + (size_t)j * L, *B = d.B + (size_t)j * L;
#pragma unroll
          for (int i = 0; i < 8; ++i) tp[i] = ldv2(A + th.mode(i));
#pragma unroll
          for (int i = 0; i < 8; ++i) Bj[i] = ldv2(B + th.mode(i));
        }
#pragma unroll
        for (int i = 0; i < 8; ++i) {
          tp[i] = cmul(tp[i], y[i]);
          t0s[i * NT] = tp[i];
          d.yhat[th.mode(i)] = y[i];
          acc[i] = make_float2(0.f, 0.f);
        }
        float first = 0.f;
        for (int m = 1; m < d.terms; ++m) {
          eo_inverse<LOG2L>(tp, p, q, x, tw, pc, th, x1, x2);  // t_{m-1} in depth space
          put(p, q, x);
          __syncthreads();
          if (m > 1) {  // the stop test of t_{m-1}, whose norm partials the barrier published
            float snt = 0.f, snw = 0.f;
#pragma unroll
            for (int w = 0; w < NWARP; ++w) {  // the same order in every thread: a uniform decision
              snt += red[buf][w].x;
              snw += red[buf][w].y;
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
          {  // times V: own and other half's values
            const float4* o = ex + ((buf * 2 + 1 - e) * 4) * HL + th.t;
            auto mix = [&](float cr, float ci, float dr_, float di, float2 mine, float2 theirs) {
              if constexpr (CPLX) return cmul(make_float2(cr, ci), mine) + cmul(make_float2(dr_, di), theirs);
              else return make_float2(fmaf(cr, mine.x, dr_ * theirs.x), fmaf(cr, mine.y, dr_ * theirs.y));
            };
#pragma unroll
            for (int i = 0; i < 4; ++i) {
              const float4 w = o[i * HL], c = cf[i * NT];
              float4 ci = make_float4(0.f, 0.f, 0.f, 0.f);
              if constexpr (CPLX) ci = cfi[i * NT];
              p[i] = mix(c.x, ci.x, c.y, ci.y, p[i], make_float2(w.x, w.y));
              q[i] = mix(c.z, ci.z, c.w, ci.w, q[i], make_float2(w.z, w.w));
            }
            if (th.z) x = mix(cmid.x, cmidi.x, cmid.y, cmidi.y, x, mid[buf][1 - e]);
          }
          buf ^= 1;
          eo_forward<LOG2L>(p, q, x, tp, tw, pc, th, x1, x2);  // T(V t_{m-1})
          ++ndst;
          float nt = 0.f, nw = 0.f;
#pragma unroll
          for (int i = 0; i < 8; ++i) {
            tp[i] = cmul(Bj[i], tp[i]);
            acc[i] = acc[i] + tp[i];
            nt += cabs2(tp[i]);
            nw += cabs2(t0s[i * NT] + acc[i]);
          }
          if (m == d.terms - 1) break;
#pragma unroll
          for (int o = 16; o > 0; o >>= 1) {
            nt += __shfl_xor_sync(0xffffffffu, nt, o);
            nw += __shfl_xor_sync(0xffffffffu, nw, o);
          }
          if (lane == 0) red[buf][warp] = make_float2(nt, nw);
        }
        {
          const float4* R = d.R + (size_t)j * L;
          const float2 bj = d.beta[j];
          float4 r[8];
#pragma unroll
          for (int i = 0; i < 8; ++i) r[i] = ldv4(R + th.mode(i));
#pragma unroll
          for (int i = 0; i < 8; ++i) y[i] = d.yhat[th.mode(i)];
#pragma unroll
          for (int i = 0; i < 8; ++i) y[i] = ffmul(r[i], y[i]) + cmul(bj, acc[i]);
        }
      }
      if (status != kStatusOk) break;
    }
    const long long gs = d.step0 + s + 1;
    if (d.tl_every > 0 && gs % d.tl_every == 0) record(s);
  }
  float2 o[8], p[4], q[4], x;
#pragma unroll
  for (int i = 0; i < 8; ++i) {
    d.yhat[th.mode(i)] = th.sign(i) * y[i];
    o[i] = out_scale * y[i];
  }
  eo_inverse<LOG2L>(o, p, q, x, tw, pc, th, x1, x2);  // physical envelope for pe_read_field
  float2* field = d.field;
  emit(p, q, x, [&](int n, float2 u) { field[n] = u; });
  ++ndst;
  if (t == 0) {
    if (status != kStatusOk) atomicMax(d.status, status);
    atomicAdd(d.ndst, (unsigned long long)ndst);
  }
}

// DST-I of `count` fields: out = scale * DST(in), field b reads N values at in + b in_stride and writes its
// modes k >= 1 - off at out + b out_stride (off = 1: mode 0 first, L values; off = 0: N values).  A CTA
// takes fields b = blockIdx.x, blockIdx.x + gridDim.x, ..., so the twiddles are loaded once, and a
// field's modes leave through shared memory, in order.
//
// Against one CTA per field with its tables in shared memory (51 KB, 12 KB of tables loaded per
// field): more fields an SM, no table traffic, the march's shorter pass chain, and the packed result
// rows are written here.  On the device, 4096 fields of N = 1023: 98 -> 18.7 us (690 -> 3580 GB/s of input and
// output, 53 % of the copy bandwidth; the call takes 24.7 us, 2.7 TB/s), of N = 4095: 418 -> 129 us; one field:
// 16.6 -> 5.1 us.  It is bound by
// the same chain at 6 fields an SM, with the shared-memory pipe as the next limit.
template <int LOG2L>
struct EDst {
  using K = ECfg<LOG2L>;
  static constexpr int MIN_BLOCKS = 65536 / (K::NT * 80);
  static constexpr size_t SMEM = sizeof(float2) * 2 * (K::X1 + K::X2);
  static_assert(K::L + K::L / 16 <= 2 * (K::X1 + K::X2), "the ordered modes reuse the exchange buffers");
};

template <int LOG2L>
__global__ void __launch_bounds__(ECfg<LOG2L>::NT, EDst<LOG2L>::MIN_BLOCKS)
    sssp_dst_eo_kernel(const float2* in, float2* out, float scale, const EoTabs tb, int count, long long in_stride,
                       long long out_stride, int off, const StartArgs sa) {
  using K = ECfg<LOG2L>;
  constexpr int L = K::L, M = K::M, NT = K::NT;
  extern __shared__ __align__(16) unsigned char smem_raw[];
  float2* st = reinterpret_cast<float2*>(smem_raw);  // the modes in order (padded)
  const EoThread<LOG2L> th;
  const int t = threadIdx.x, e = th.e;
  float2* x1 = st + e * (K::X1 + K::X2);
  float2* x2 = x1 + K::X1;
  EoTw<LOG2L> tw;
  tw.load(tb, th);
  EoPair pc;
#pragma unroll
  for (int i = 0; i < 4; ++i) pc.c[i] = e ? __ldg(tb.cL + th.slot(i)) : make_float2(__ldg(tb.beta + th.slot(i)), 0.f);
  const float h = e ? 0.5f : 0.25f, g = e ? 0.5f : -0.25f;  // odd half (x_n + x_{L-n})/2, even half (x_n - x_{L-n})/4
  for (int b = blockIdx.x; b < count; b += gridDim.x) {
    const float2* x = in + b * in_stride - 1;  // x[n], n in [1, N]
    float2 p[4], q[4], xm = make_float2(0.f, 0.f), sp[8];
#pragma unroll
    for (int i = 0; i < 4; ++i) {
      const int m = th.slot(i);
      const float2 zero = make_float2(0.f, 0.f);
      const float2 a0 = m ? x[m] : zero, a1 = m ? x[L - m] : zero, b0 = x[M - m], b1 = x[M + m];
      p[i] = make_float2(fmaf(h, a0.x, g * a1.x), fmaf(h, a0.y, g * a1.y));
      q[i] = make_float2(fmaf(h, b0.x, g * b1.x), fmaf(h, b0.y, g * b1.y));
      if (sa.field) {  // the odd half writes n < M, the even half the rest
        if (e) {
          sa.field[m] = a0;
          if (m) sa.field[M - m] = b0;
        } else {
          if (m) sa.field[L - m] = a1;
          sa.field[M + m] = b1;
        }
      }
    }
    if (th.z) {
      const float2 a0 = x[M / 2], a1 = x[L - M / 2];
      xm = make_float2(fmaf(h, a0.x, g * a1.x), fmaf(h, a0.y, g * a1.y));
      if (sa.field) sa.field[e ? M / 2 : L - M / 2] = e ? a0 : a1;
    }
    if (sa.status && t == 0) *sa.status = kStatusOk;
    eo_forward<LOG2L>(p, q, xm, sp, tw, pc, th, x1, x2);
    __syncthreads();  // both halves are past the exchange buffers
#pragma unroll
    for (int i = 0; i < 8; ++i) st[pidx(th.mode(i))] = th.sign(i) * scale * sp[i];
    __syncthreads();
    float2* o = out + b * out_stride + off - 1;
    for (int k = t + 1 - off; k < L; k += NT) o[k] = st[pidx(k)];
    __syncthreads();
  }
}

}  // namespace sssp
