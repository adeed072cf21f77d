// SSSP range-march kernels for sm_103a.
//
// One CTA marches one solve for all of its range steps (a persistent, fused kernel): the
// field lives in registers in spectral (DST-I) space between stages and steps, every
// transform runs in shared memory, and only the profile rows, the Pade tables and the TL
// output touch global memory.
//
// Per range step (Algorithm 1, product form of the Section 2 Pade propagator):
//   for every Pade stage j:   y <- R_j(lambda) y + beta_j sum_{m>=1} t_m        (spectral)
//     t_0 = L_j^{-1} y,  t_m = -b_j L_j^{-1} (V t_{m-1})                    (Eq. Neumann)
//     L_j^{-1} = IDST diag(1/(1 + b_j lambda_m)) DST                         (Eq. inverse_isovel)
//   R_j = (1 + a_j lambda)/(1 + b_j lambda) is applied with a hi+lo (float-float) table so
//   that its rounding does not accumulate over thousands of steps; the Neumann terms are
//   plain FP32.  Without a profile (neumann_terms <= 1) the whole step is one diagonal
//   multiply by G = prod_j R_j.
//
// DST-I of length N = L - 1 (L a power of two) is one complex FFT of length L:
//   y_n = sin(pi n/L)(x_n + x_{L-n}) + (x_n - x_{L-n})/2,  Y = FFT_L(y),
//   S_{2k} = (i/2)(Y_k - Y_{L-k}),  S_{2k+1} = S_{2k-1} + (Y_k + Y_{L-k})/2,  S_{-1} = -S_1,
// with a block-wide prefix scan for the odd outputs.  The FFT is a Stockham autosort FFT
// with radix-P passes (P = 4, 8 or 16 points per thread: one radix-P butterfly per thread per
// pass) and a final smaller-radix pass, ping-ponging between two padded shared buffers (index i
// stored at i + i/16 to spread the strided accesses over the banks).  P trades threads for
// passes: P = 4 gives twice the warps of P = 8 (latency hiding) at more passes and barriers,
// P = 16 half the warps at fewer passes; the library times them per plan (pe_plan_autotune).
#pragma once
#include <cuda_runtime.h>
#include <stdint.h>

namespace sssp {

constexpr int kMaxStages = 8;
constexpr int kStatusOk = 0;
constexpr int kStatusDiverged = 4;
constexpr int kStatusNumeric = 7;

// Everything one CTA needs to march one solve.  Tables are indexed by mode m in [0, L)
// (m = 0 is a zero pad), profile rows and fields by depth index n in [0, L) (n = 0 is the
// zero boundary value).
struct SolveDesc {
  const float4* R;       // p x L  hi/lo of (1 + a_j lam_m)/(1 + b_j lam_m)
  const float2* A;       // p x L  (2/L) / (1 + b_j lam_m)
  const float2* B;       // p x L  (2/L) (-b_j) / (1 + b_j lam_m)
  const float4* G;       // L      hi/lo of prod_j R_j (isovelocity step)
  const float* V;        // nodes x L, V = n^2 - 1 (real part)
  const float* Vi;       // nodes x L imaginary part of n^2 (absorbing layers), or null
  const double* node_r;  // node ranges, non-decreasing
  float2* yhat;          // L  spectral state (DST-I coefficients, unnormalised)
  float2* work;          // 4 L workspace (grids beyond one CTA's shared memory only)
  float2* field;         // L  physical envelope written at the end of the march
  float* tl;             // TL rows, N floats each
  int* status;           // device status word
  unsigned long long* ndst;  // number of DST-I transforms executed (accumulated); the next word counts the
                             // finished CTAs of a march whose TL rows are split over CTAs (0 between marches)
  float2 beta[kMaxStages];   // (L/2)(1 - a_j/b_j)
  double r0;             // range at the start of this march
  double dr;
  double tol2;           // squared Neumann tolerance
  long long step0;       // steps marched since the field was set
  long long rec0;        // TL rows already recorded
  int node0;             // node in force at the first step's midpoint
  int nodes;
  int steps;
  int p;
  int terms;             // max Neumann terms incl. m = 0 (<= 1: V ignored)
  int tl_every;          // 0: no TL rows
  int N;
  const float4* fd;      // FD-SSP plans: nodes x p x L table entries (march_fd.cuh), else null
  const float4* fdc;     // FD-SSP plans: per stage hi/lo of a_j/b_j and 1 - a_j/b_j
};

// Whether the passes from span NS end with a radix-2 pass (span L/2)
template <int LOG2L, int NS, int PPT>
__host__ __device__ constexpr bool ends_radix2() {
  constexpr int L = 1 << LOG2L;
  if constexpr (NS >= L) {
    return false;
  } else if constexpr (L / NS == 2) {
    return true;
  } else {
    return ends_radix2<LOG2L, NS * ((L / NS) >= PPT ? PPT : (L / NS)), PPT>();
  }
}

constexpr bool kTwiddleRegisters = true;
constexpr bool kOperandRegisters = true;

template <int LOG2L, int PPT = 8>
struct Cfg {
  static constexpr int L = 1 << LOG2L;
  static constexpr int P = PPT;               // points per thread (radix of the passes)
  static constexpr int HALF = PPT / 2;        // DST-I output pairs per thread
  static constexpr int NT = L / PPT;          // threads per CTA
  // padded buffer length (64 more at L = 1024, P = 8 for the span-8 pass's layout, BufMap)
  static constexpr int PADL = L + L / 16 + 64 * (LOG2L == 10 && PPT == 8);
  static constexpr int WS = NT >= 32 ? 32 : NT;
  static constexpr int NW = (NT + 31) / 32;
  static constexpr unsigned MASK = NT >= 32 ? 0xffffffffu : ((1u << NT) - 1u);
  // per-thread twiddles of the one-butterfly-per-thread passes kept in registers (P = 4 and 8,
  // L <= 1024)
  static constexpr bool TWREG = kTwiddleRegisters && (PPT == 8 || PPT == 4) && L <= 1024;
  // the Neumann terms' per-thread operands (V row, B_j, t_0) and the sine weights in registers
  // too (the register file still holds two CTAs of the largest such grid)
  static constexpr bool OPREG = kOperandRegisters && TWREG;
  // CTAs per SM the register budget is sized for: 128 registers per thread for P = 4 and for
  // P = 8 beyond L = 1024, 255 for P = 8 with the register-resident twiddles and operands (two
  // CTAs of the 128-thread L = 1024 grid per SM) and for P = 16 (its 16-point butterflies hold
  // 3 x 16 complex values), at most 16 CTAs
  static constexpr int REGS = PPT == 8 ? (OPREG ? 255 : (TWREG ? 168 : 128)) : (PPT == 4 ? 128 : 256);
  static constexpr int MB0 = 65536 / ((NT < 32 ? 32 : NT) * REGS);  // registers go by whole warps
  static constexpr int MIN_BLOCKS = MB0 >= 16 ? 16 : (MB0 < 1 ? 1 : MB0);
  // dynamic shared memory: 2 padded buffers, twiddles, t_0 and B_j areas, sin weights, V row,
  // scan + reduce
  static constexpr size_t SMEM0 = sizeof(float2) * (2 * PADL + 3 * L) + sizeof(float) * (2 * L) +
                                  sizeof(float2) * NW + sizeof(float) * 2 * NW;
  // Up to L = 512 a stage's tables are staged in shared memory ahead of their use (R where t_0 and B_j are
  // otherwise, A and B in an area of their own) and the stop test rides on the next transform (StopHook):
  // N = 255 1400 -> 1300 cycles a transform.  At L = 1024 one solve gained 1 %, 256 solves lost 1 %.
  static constexpr bool AHEAD = OPREG && L <= 512;
  static constexpr size_t SMEM = SMEM0 + (AHEAD ? sizeof(float4) * L : 0);
  static constexpr size_t SMEM_CPLX = AHEAD ? SMEM : SMEM0 + sizeof(float) * L;  // + imaginary V row
};

// padded shared-memory index: one pad element per 16 (128 B), so contiguous half-warp
// accesses stay conflict-free and the stride-4 / stride-8 patterns spread over the banks
__device__ __forceinline__ int pidx(int i) { return i + (i >> 4); }

// Complex additions, subtractions and real scalings as packed two-lane FP32 instructions
// (add/sub/mul .f32x2 of sm_100-family GPUs): one instruction for both components, each lane
// rounded exactly as the scalar instruction would round it.
constexpr bool kPackedF32 = true;

__device__ __forceinline__ float2 operator+(float2 a, float2 b) {
  if constexpr (kPackedF32) {
    float2 r;
    asm("{\n\t.reg .b64 ra, rb, rd;\n\tmov.b64 ra, {%2, %3};\n\tmov.b64 rb, {%4, %5};\n\t"
        "add.rn.f32x2 rd, ra, rb;\n\tmov.b64 {%0, %1}, rd;\n\t}"
        : "=f"(r.x), "=f"(r.y)
        : "f"(a.x), "f"(a.y), "f"(b.x), "f"(b.y));
    return r;
  } else {
    return make_float2(a.x + b.x, a.y + b.y);
  }
}
__device__ __forceinline__ float2 operator-(float2 a, float2 b) {
  if constexpr (kPackedF32) {
    float2 r;
    asm("{\n\t.reg .b64 ra, rb, rd;\n\tmov.b64 ra, {%2, %3};\n\tmov.b64 rb, {%4, %5};\n\t"
        "sub.rn.f32x2 rd, ra, rb;\n\tmov.b64 {%0, %1}, rd;\n\t}"
        : "=f"(r.x), "=f"(r.y)
        : "f"(a.x), "f"(a.y), "f"(b.x), "f"(b.y));
    return r;
  } else {
    return make_float2(a.x - b.x, a.y - b.y);
  }
}
__device__ __forceinline__ float2 operator*(float s, float2 a) {
  if constexpr (kPackedF32) {
    float2 r;
    asm("{\n\t.reg .b64 ra, rs, rd;\n\tmov.b64 ra, {%2, %3};\n\tmov.b64 rs, {%4, %4};\n\t"
        "mul.rn.f32x2 rd, rs, ra;\n\tmov.b64 {%0, %1}, rd;\n\t}"
        : "=f"(r.x), "=f"(r.y)
        : "f"(a.x), "f"(a.y), "f"(s));
    return r;
  } else {
    return make_float2(s * a.x, s * a.y);
  }
}
__device__ __forceinline__ float2 cmul(float2 a, float2 b) {
  return make_float2(fmaf(a.x, b.x, -a.y * b.y), fmaf(a.x, b.y, a.y * b.x));
}
__device__ __forceinline__ float2 mul_negi(float2 x) { return make_float2(x.y, -x.x); }
__device__ __forceinline__ float2 conjf2(float2 a) { return make_float2(a.x, -a.y); }
__device__ __forceinline__ float cabs2(float2 a) { return fmaf(a.x, a.x, a.y * a.y); }

// Stop test of the Neumann series (Eq. Neumann; stop after term m once ||t_m|| <= tol ||w_j||),
// compared in FP64: the sums of squares nt2 = ||t_m||^2 and nw2 = ||w_j||^2 are widened to
// double and tested against tol^2 held in double.  (They are accumulated in FP32: a sum of
// positive terms carries a relative rounding error below 1e-6, which moves the threshold on the
// norm by less than a millionth of itself.)
__device__ __forceinline__ bool neumann_stop(float nt2, float nw2, double tol2) {
  return double(nt2) <= tol2 * double(nw2);
}

// The same decision with the FP64 comparison taken only near the threshold (FP64 instructions
// have a latency of ~64 cycles here): the FP32 product tol2f nw2 is within a few ulps of
// tol^2 nw2, so where nt2 lies outside [tol2f nw2 / 2, 2 tol2f nw2] the FP32 comparison already
// gives the FP64 comparison's answer.  Tiny or non-finite thresholds go to FP64 directly.
__device__ __forceinline__ bool neumann_stop_fast(float nt2, float nw2, double tol2, float tol2f) {
  const float th = tol2f * nw2;
  if (th > 1e-30f && th < 1e30f) {
    if (nt2 < 0.5f * th) return true;
    if (nt2 > 2.0f * th) return false;
  }
  return neumann_stop(nt2, nw2, tol2);
}

// y * (hi + lo) with the hi/lo split of a multiplier: the product is rounded, the
// multiplier is not, so no fixed per-mode error builds up over the steps.
__device__ __forceinline__ float2 ffmul(float4 g, float2 y) {
  const float re_lo = fmaf(g.z, y.x, -g.w * y.y);
  const float im_lo = fmaf(g.z, y.y, g.w * y.x);
  return make_float2(fmaf(g.x, y.x, fmaf(-g.y, y.y, re_lo)), fmaf(g.x, y.y, fmaf(g.y, y.x, im_lo)));
}

__device__ __forceinline__ void dft2(float2& a, float2& b) {
  const float2 t = a;
  a = t + b;
  b = t - b;
}
// forward DFT of length 4 in place, natural output order
__device__ __forceinline__ void dft4(float2& x0, float2& x1, float2& x2, float2& x3) {
  const float2 c0 = x0 + x2, d0 = x0 - x2, c1 = x1 + x3, d1 = mul_negi(x1 - x3);
  x0 = c0 + c1;
  x2 = c0 - c1;
  x1 = d0 + d1;
  x3 = d0 - d1;
}
// Irrational butterfly constants (cos and sin of pi/4, pi/8) are applied as hi + lo float
// pairs: a constant's FP32 representation error (up to 3e-8 relative) would be the same in
// every transform and add up coherently over thousands of range steps.
__device__ __forceinline__ float ff_mul(float hi, float lo, float s) { return fmaf(hi, s, lo * s); }

// forward DFT of length 8 (one radix-2 frequency split, then two length-4 DFTs)
__device__ __forceinline__ void dft8(float2 (&v)[8]) {
  constexpr double H = 0.70710678118654752440;
  constexpr float hh = float(H), hl = float(H - double(float(H)));
  float2 a0 = v[0] + v[4], a1 = v[1] + v[5], a2 = v[2] + v[6], a3 = v[3] + v[7];
  float2 b0 = v[0] - v[4], b1 = v[1] - v[5], b2 = v[2] - v[6], b3 = v[3] - v[7];
  b1 = make_float2(ff_mul(hh, hl, b1.x + b1.y), ff_mul(hh, hl, b1.y - b1.x));    // * e^{-i pi/4}
  b2 = mul_negi(b2);                                                              // * e^{-i pi/2}
  b3 = make_float2(ff_mul(hh, hl, b3.y - b3.x), -ff_mul(hh, hl, b3.x + b3.y));   // * e^{-3i pi/4}
  dft4(a0, a1, a2, a3);
  dft4(b0, b1, b2, b3);
  v[0] = a0; v[2] = a1; v[4] = a2; v[6] = a3;
  v[1] = b0; v[3] = b1; v[5] = b2; v[7] = b3;
}

// forward DFT of length 16 in natural order (one radix-2 frequency split, two length-8 DFTs)
__device__ __forceinline__ void dft16(float2 (&v)[16]) {
  constexpr double C1 = 0.92387953251128675613, S1 = 0.38268343236508977173, H = 0.70710678118654752440;
  constexpr float c1h = float(C1), c1l = float(C1 - double(float(C1)));
  constexpr float s1h = float(S1), s1l = float(S1 - double(float(S1)));
  constexpr float hh = float(H), hl = float(H - double(float(H)));
  // w16^r = e^{-2 pi i r/16}, r = 0..7, as hi + lo
  const float4 w[8] = {make_float4(1.f, 0.f, 0.f, 0.f),     make_float4(c1h, -s1h, c1l, -s1l),
                       make_float4(hh, -hh, hl, -hl),        make_float4(s1h, -c1h, s1l, -c1l),
                       make_float4(0.f, -1.f, 0.f, 0.f),     make_float4(-s1h, -c1h, -s1l, -c1l),
                       make_float4(-hh, -hh, -hl, -hl),      make_float4(-c1h, -s1h, -c1l, -s1l)};
  float2 a[8], b[8];
#pragma unroll
  for (int r = 0; r < 8; ++r) {
    a[r] = v[r] + v[r + 8];
    b[r] = (r == 0) ? v[r] - v[r + 8] : ffmul(w[r], v[r] - v[r + 8]);
  }
  dft8(a);
  dft8(b);
#pragma unroll
  for (int r = 0; r < 8; ++r) {
    v[2 * r] = a[r];
    v[2 * r + 1] = b[r];
  }
}

template <int N>
__device__ __forceinline__ void dftN(float2 (&v)[N]) {
  if constexpr (N == 16) dft16(v);
  else dft8(v);
}

template <int R>
__device__ __forceinline__ void dftR(float2 (&v)[R]) {
  if constexpr (R == 16) dft16(v);
  else if constexpr (R == 8) dft8(v);
  else if constexpr (R == 4) dft4(v[0], v[1], v[2], v[3]);
  else dft2(v[0], v[1]);
}

// One Stockham pass of radix R over span NS: butterfly j reads src[j + r L/R], applies the
// twiddles exp(-2 pi i r k/(NS R)), k = j mod NS, and writes dst[(j - k) R + k + r NS].
// Twiddles come from a per-pass table tw[(NS - P) + (r - 1) NS + k] (k contiguous, so a
// half-warp reads 16 consecutive entries or broadcasts), P the first pass's radix.
template <int LOG2L, int R, int NS, int PPT = 8>
__device__ __forceinline__ void fft_pass(const float2* __restrict__ src, float2* __restrict__ dst,
                                         const float2* __restrict__ tw) {
  constexpr int L = 1 << LOG2L, NT = L / PPT, NB = L / R, PER = NB / NT;
  constexpr int OFF = NS - PPT;  // the passes before span NS took (NS - PPT) entries
#pragma unroll
  for (int q = 0; q < PER; ++q) {
    const int j = threadIdx.x + q * NT;
    float2 v[R];
#pragma unroll
    for (int r = 0; r < R; ++r) v[r] = src[pidx(j + r * NB)];
    const int k = j & (NS - 1);
    if constexpr (NS > 1) {
#pragma unroll
      for (int r = 1; r < R; ++r) v[r] = cmul(v[r], tw[OFF + (r - 1) * NS + k]);
    }
    dftR<R>(v);
    const int base = (j - k) * R + k;
#pragma unroll
    for (int r = 0; r < R; ++r) dst[pidx(base + r * NS)] = v[r];
  }
}

// The passes from span NS on, leaving out a final radix-2 pass (the DST-I post-processing does
// it, see dst_block); returns the buffer holding the result
template <int LOG2L, int NS, int PPT>
__device__ __forceinline__ float2* fft_rest_x2(float2* src, float2* dst, const float2* tw) {
  constexpr int L = 1 << LOG2L;
  if constexpr (NS >= L || L / NS == 2) {
    return src;
  } else {
    constexpr int R = (L / NS) >= PPT ? PPT : (L / NS);
    fft_pass<LOG2L, R, NS, PPT>(src, dst, tw);
    __syncthreads();
    return fft_rest_x2<LOG2L, NS * R, PPT>(dst, src, tw);
  }
}

// Per-thread twiddles of the passes after the first, held in registers for a whole march: a pass
// with one butterfly per thread (L/R = L/P butterflies) applies the same twiddles in every
// transform, so they are loaded from the shared table once.  TwChain<LOG2L, NS, P> holds those of
// the passes from span NS on (nothing for passes with more butterflies per thread, and nothing
// for a final radix-2 pass, which the DST-I post-processing does with its own twiddles `post`).
template <int LOG2L, int NS, int PPT>
struct TwChain {
  static constexpr int L = 1 << LOG2L;
  static constexpr bool END = (NS >= L) || (L / NS == 2);
  static constexpr int R = END ? 1 : ((L / NS) >= PPT ? PPT : (L / NS));
  static constexpr bool REG = !END && (L / R) == (L / PPT);  // one butterfly per thread
  float2 w[REG ? R - 1 : 1];
  TwChain<LOG2L, (END ? L : NS * R), PPT> next;
  __device__ __forceinline__ void load(const float2* tw) {
    if constexpr (REG && NS > 1) {
      const int k = threadIdx.x & (NS - 1);
#pragma unroll
      for (int r = 1; r < R; ++r) w[r - 1] = tw[(NS - PPT) + (r - 1) * NS + k];
    }
    if constexpr (!END) next.load(tw);
  }
};
template <int LOG2L, int PPT>
struct TwChain<LOG2L, (1 << LOG2L), PPT> {  // past the last pass
  static constexpr bool END = true, REG = false;
  static constexpr int R = 1;
  __device__ __forceinline__ void load(const float2*) {}
};

// the whole chain of a transform plus the fused radix-2 pass's twiddles e^{-2 pi i k/L},
// k = (P/2) t + s
template <int LOG2L, int PPT>
struct TwRegs {
  TwChain<LOG2L, PPT, PPT> chain;
  float2 post[PPT / 2];
  float sw[PPT];  // sine weights of the first pass, n = t + r L/P (filled only with `sinw`)
  bool has_sw = false;
  __device__ __forceinline__ void load(const float2* tw, const float* sinw = nullptr) {
    constexpr int L = 1 << LOG2L;
    chain.load(tw);
    if constexpr (ends_radix2<LOG2L, PPT, PPT>()) {
#pragma unroll
      for (int s = 0; s < PPT / 2; ++s) post[s] = tw[(L / 2 - PPT) + (PPT / 2) * int(threadIdx.x) + s];
    }
    if (sinw) {
#pragma unroll
      for (int r = 0; r < PPT; ++r) sw[r] = sinw[int(threadIdx.x) + r * (L / PPT)];
      has_sw = true;
    }
  }
};

// Shared-memory layout of the buffer written by the pass of span NS (NS = 1: the first pass) on
// the register-twiddle path: pidx unless specialised.  At L = 1024, 8 points per thread, two
// buffers get layouts of their own (found by counting the bank wavefronts of every warp access
// of the transform), which make their accesses conflict-free where pidx gives 2-way conflicts:
// the span-8 pass writes butterfly outputs (j - k) 8 + k + 8 r, so one half-warp stores rows 0
// and 64 apart -- an extra 2 words per 32 elements moves them to different banks; the span-64
// pass's output is read by the DST-I post-processing forwards and backwards with stride 4 -- an
// XOR of the low index bits with (3 b) & 12 within each 16-element block b spreads both.
template <int LOG2L, int PPT, int NS>
struct BufMap {
  static constexpr bool DEFAULT = true;
  __device__ static __forceinline__ int at(int i) { return pidx(i); }
};
template <>
struct BufMap<10, 8, 8> {
  static constexpr bool DEFAULT = false;  // indices up to 1023 + 63 + 62 (Cfg::PADL has room)
  __device__ static __forceinline__ int at(int i) { return i + (i >> 4) + 2 * (i >> 5); }
};
template <>
struct BufMap<10, 8, 64> {
  static constexpr bool DEFAULT = false;
  __device__ static __forceinline__ int at(int i) {
    const int j = i ^ ((3 * (i >> 4)) & 12);
    return j + (j >> 4);
  }
};

// fft_pass with the twiddles of a register chain link, reading the layout SM and writing DM
template <int LOG2L, int R, int NS, int PPT, class SM, class DM>
__device__ __forceinline__ void fft_pass_reg(const float2* __restrict__ src, float2* __restrict__ dst,
                                             const float2 (&w)[R - 1]) {
  constexpr int L = 1 << LOG2L, NB = L / R;
  const int j = threadIdx.x;
  float2 v[R];
#pragma unroll
  for (int r = 0; r < R; ++r) v[r] = src[SM::at(j + r * NB)];
  const int k = j & (NS - 1);
#pragma unroll
  for (int r = 1; r < R; ++r) v[r] = cmul(v[r], w[r - 1]);
  dftR<R>(v);
  const int base = (j - k) * R + k;
#pragma unroll
  for (int r = 0; r < R; ++r) dst[DM::at(base + r * NS)] = v[r];
}

// span of the last pass fft_rest_x2r runs from span NS on (PREV: the span of the pass before)
template <int LOG2L, int NS, int PPT, int PREV>
__host__ __device__ constexpr int chain_last_span() {
  using Ch = TwChain<LOG2L, NS, PPT>;
  if constexpr (Ch::END) return PREV;
  else return chain_last_span<LOG2L, NS * Ch::R, PPT, NS>();
}

// fft_rest_x2 taking register twiddles where the chain holds them (for passes that do not end
// with radix 2 it runs them all, like fft_rest); src holds the output of the pass of span PREV,
// and the returned buffer is in the layout BufMap of the last pass's span
template <int LOG2L, int NS, int PPT, int PREV = 1>
__device__ __forceinline__ float2* fft_rest_x2r(float2* src, float2* dst, const float2* tw,
                                                const TwChain<LOG2L, NS, PPT>& c) {
  using Ch = TwChain<LOG2L, NS, PPT>;
  if constexpr (Ch::END) {
    return src;
  } else {
    using SM = BufMap<LOG2L, PPT, PREV>;
    using DM = BufMap<LOG2L, PPT, NS>;
    if constexpr (Ch::REG && NS > 1) {
      fft_pass_reg<LOG2L, Ch::R, NS, PPT, SM, DM>(src, dst, c.w);
    } else {
      static_assert(SM::DEFAULT && DM::DEFAULT, "shared-table passes use the pidx layout");
      fft_pass<LOG2L, Ch::R, NS, PPT>(src, dst, tw);
    }
    __syncthreads();
    return fft_rest_x2r<LOG2L, NS * Ch::R, PPT, NS>(dst, src, tw, c.next);
  }
}

template <int LOG2L, int NS, int PPT = 8>
__device__ __forceinline__ float2* fft_rest(float2* src, float2* dst, const float2* tw) {
  constexpr int L = 1 << LOG2L;
  if constexpr (NS >= L) {
    return src;
  } else {
    constexpr int R = (L / NS) >= PPT ? PPT : (L / NS);
    fft_pass<LOG2L, R, NS, PPT>(src, dst, tw);
    __syncthreads();
    return fft_rest<LOG2L, NS * R, PPT>(dst, src, tw);
  }
}

// Work a transform takes along on its first barrier: publish() before it, and stop() after it, which may
// end the transform there (every thread the same way).
struct NoHook {
  __device__ __forceinline__ void publish() {}
  __device__ __forceinline__ bool stop() { return false; }
};

// Unnormalised DST-I of the L values in `a` (natural order, padded; a[0] is ignored) into
// out[0..P) = S_{P t..P t+P) of thread t (S_0 = 0).  Uses `b` as the ping-pong buffer.
// On return every thread has finished reading both buffers.  False: the hook ended it.
template <int LOG2L, int PPT = 8, class HOOK = NoHook>
__device__ __forceinline__ bool dst_block(float2* a, float2* b, const float2* __restrict__ tw,
                                          const float* __restrict__ sinw, float2* scan_s, float2 (&out)[PPT],
                                          const TwRegs<LOG2L, PPT>* twr = nullptr, HOOK hook = {}) {
  using C = Cfg<LOG2L, PPT>;
  constexpr int L = C::L, H = C::HALF;
  const int t = threadIdx.x;
  {  // first radix-P pass (span 1, no twiddles), fused with the sine pre-weighting
    float2 v[PPT];
#pragma unroll
    for (int r = 0; r < PPT; ++r) {
      const int n = t + r * (L / PPT);
      const float2 xn = a[pidx(n)];
      const float2 xm = a[pidx((L - n) & (L - 1))];
      const float s = (twr && twr->has_sw) ? twr->sw[r] : sinw[n];
      v[r] = make_float2(fmaf(s, xn.x + xm.x, 0.5f * (xn.x - xm.x)), fmaf(s, xn.y + xm.y, 0.5f * (xn.y - xm.y)));
    }
    dftR<PPT>(v);
#pragma unroll
    for (int r = 0; r < PPT; ++r) b[pidx(PPT * t + r)] = v[r];
  }
  hook.publish();
  __syncthreads();
  if (hook.stop()) return false;
  // When the passes end with radix 2 (span L/2), that pass is fused into the post-processing:
  // with the earlier passes' result F and w = e^{-2 pi i/L}, Y_k = F_k + w^k F_{k+L/2} and
  // Y_{L-k} = F_{L/2-k} + conj(w^k) F_{L-k} (the butterfly of L/2 - k, whose twiddle is
  // -conj(w^k)) -- the same arithmetic, one barrier and one pass through shared memory fewer.
  constexpr bool X2 = ends_radix2<LOG2L, PPT, PPT>();
  const float2* F = twr ? fft_rest_x2r<LOG2L, PPT, PPT>(b, a, tw, twr->chain)
                        : (X2 ? fft_rest_x2<LOG2L, PPT, PPT>(b, a, tw) : fft_rest<LOG2L, PPT, PPT>(b, a, tw));
  using FM = BufMap<LOG2L, PPT, chain_last_span<LOG2L, PPT, PPT, 1>()>;  // F's layout (register path)
  auto fat = [&](int i) { return twr ? FM::at(i) : pidx(i); };
  // post-processing: even outputs from pairs (k, L-k), odd outputs by a prefix scan
  float2 se[H], dd[H];
#pragma unroll
  for (int s = 0; s < H; ++s) {
    const int k = H * t + s;
    float2 yk, ym;
    if constexpr (X2) {
      const float2 w = twr ? twr->post[s] : tw[(L / 2 - PPT) + k];  // the radix-2 pass's e^{-2 pi i k/L}
      yk = F[fat(k)] + cmul(F[fat(k + L / 2)], w);
      ym = (k == 0) ? yk : F[fat(L / 2 - k)] + cmul(F[fat(L - k)], conjf2(w));
    } else {
      yk = F[fat(k)];
      ym = F[fat((L - k) & (L - 1))];
    }
    se[s] = make_float2(-0.5f * (yk.y - ym.y), 0.5f * (yk.x - ym.x));
    dd[s] = (k == 0) ? 0.5f * yk : 0.5f * (yk + ym);
  }
#pragma unroll
  for (int s = 1; s < H; ++s) dd[s] = dd[s] + dd[s - 1];
  const int lane = t & 31, warp = t >> 5;
  float2 inc = dd[H - 1];
#pragma unroll
  for (int o = 1; o < C::WS; o <<= 1) {
    const float nx = __shfl_up_sync(C::MASK, inc.x, o, C::WS);
    const float ny = __shfl_up_sync(C::MASK, inc.y, o, C::WS);
    if (lane >= o) inc = inc + make_float2(nx, ny);
  }
  float2 excl = make_float2(__shfl_up_sync(C::MASK, inc.x, 1, C::WS), __shfl_up_sync(C::MASK, inc.y, 1, C::WS));
  if (lane == 0) excl = make_float2(0.f, 0.f);
  if constexpr (C::NW > 1) {
    if (lane == C::WS - 1) scan_s[warp] = inc;
    __syncthreads();
    float2 off = make_float2(0.f, 0.f);
    for (int w = 0; w < warp; ++w) off = off + scan_s[w];
    excl = excl + off;
  } else {
    __syncthreads();
  }
#pragma unroll
  for (int s = 0; s < H; ++s) {
    out[2 * s] = se[s];
    out[2 * s + 1] = dd[s] + excl;
  }
  return true;
}

// Boundary conditions of Section 3.1: homogeneous Dirichlet (DST-I, the workloads) and
// periodic (DFT).
constexpr int kBcDirichlet = 0;
constexpr int kBcPeriodic = 1;

// Unnormalised DFT of the L values in `a` (natural order, padded) into out[0..P) = X_{Pt..Pt+P)
// of thread t; INV uses e^{+2 pi i n m/L} (by conjugating input and output).  On return every
// thread has finished reading both buffers.
template <int LOG2L, bool INV, int PPT = 8, class HOOK = NoHook>
__device__ __forceinline__ bool dft_block(float2* a, float2* b, const float2* __restrict__ tw, float2 (&out)[PPT],
                                          HOOK hook = {}) {
  constexpr int L = 1 << LOG2L;
  const int t = threadIdx.x;
  {
    float2 v[PPT];
#pragma unroll
    for (int r = 0; r < PPT; ++r) {
      const float2 x = a[pidx(t + r * (L / PPT))];
      v[r] = INV ? conjf2(x) : x;
    }
    dftR<PPT>(v);
#pragma unroll
    for (int r = 0; r < PPT; ++r) b[pidx(PPT * t + r)] = v[r];
  }
  hook.publish();
  __syncthreads();
  if (hook.stop()) return false;
  const float2* F = fft_rest<LOG2L, PPT, PPT>(b, a, tw);
#pragma unroll
  for (int i = 0; i < PPT; ++i) {
    const float2 x = F[pidx(PPT * t + i)];
    out[i] = INV ? conjf2(x) : x;
  }
  __syncthreads();
  return true;
}

// The transform of the boundary condition: TO_DEPTH maps spectral coefficients to depth values
// (the inverse transform up to the scale folded into the tables), otherwise depth -> spectral.
template <int LOG2L, int BC, bool TO_DEPTH, int PPT = 8, class HOOK = NoHook>
__device__ __forceinline__ bool xform(float2* a, float2* b, const float2* __restrict__ tw,
                                      const float* __restrict__ sinw, float2* scan_s, float2 (&out)[PPT],
                                      const TwRegs<LOG2L, PPT>* twr = nullptr, HOOK hook = {}) {
  if constexpr (BC == kBcPeriodic) {
    return dft_block<LOG2L, TO_DEPTH, PPT>(a, b, tw, out, hook);
  } else {
    return dst_block<LOG2L, PPT>(a, b, tw, sinw, scan_s, out, twr, hook);  // DST-I is its own inverse
  }
}

// The stop test of the Neumann series.  As a hook it rides on the next (inverse) transform's first barrier:
// the warps reduce their norm partials while the transform's first pass runs, and the decision is taken one
// pass into it -- a pass wasted once a stage, against the reduction's chain of shuffles every term.
template <int WS, int NW, unsigned MASK>
struct StopHook {
  float nt, nw;  // this thread's partials
  float* red;
  int m;         // the term tested
  float* first;
  int* status;
  double tol2;
  float tol2f;
  __device__ __forceinline__ void publish() {
#pragma unroll
    for (int o = WS / 2; o > 0; o >>= 1) {
      nt += __shfl_xor_sync(MASK, nt, o, WS);
      nw += __shfl_xor_sync(MASK, nw, o, WS);
    }
    if ((threadIdx.x & 31) == 0) {
      red[2 * (threadIdx.x >> 5)] = nt;
      red[2 * (threadIdx.x >> 5) + 1] = nw;
    }
  }
  __device__ __forceinline__ bool stop() {
    // block totals: every thread adds the warps' partials in the same order (broadcast
    // reads, no dependent shuffles), so EVERY thread holds the same total — the stop
    // decision below must be uniform across the block (it guards __syncthreads).
    float snt = 0.f, snw = 0.f;
#pragma unroll
    for (int w = 0; w < NW; ++w) {
      const float2 pr = reinterpret_cast<const float2*>(red)[w];
      snt += pr.x;
      snw += pr.y;
    }
    if (!isfinite(snt) || !isfinite(snw)) {
      *status = kStatusNumeric;
      return true;
    }
    // blow-up: a term 1e4 times the first correction term.  (Growth over a few terms
    // alone is no evidence: the operator b_j L_j^{-1} V is not normal, so convergent
    // series can grow transiently.)
    if (m == 1) *first = snt;
    else if (*first > 0.f && snt > 1e8f * *first) {
      *status = kStatusDiverged;
      return true;
    }
    return neumann_stop_fast(snt, snw, tol2, tol2f);
  }
};

// 16 bytes global -> shared, asynchronously; the thread's own copies only, waited for by group
__device__ __forceinline__ void cp_async16(float4* dst, const float4* src) {
  asm volatile("cp.async.cg.shared.global [%0], [%1], 16;" ::"r"(unsigned(__cvta_generic_to_shared(dst))), "l"(src) : "memory");
}
__device__ __forceinline__ void cp_async_commit() { asm volatile("cp.async.commit_group;" ::: "memory"); }
template <int N>
__device__ __forceinline__ void cp_async_wait() { asm volatile("cp.async.wait_group %0;" ::"n"(N) : "memory"); }

template <int LOG2L, int PPT = 8>
__device__ __forceinline__ void load_tables(float2* tw, float* sinw, const float2* __restrict__ tw_g,
                                            const float* __restrict__ sin_g) {
  using C = Cfg<LOG2L, PPT>;
  for (int i = threadIdx.x; i < C::L; i += C::NT) {
    tw[i] = tw_g[i];
    sinw[i] = sin_g[i];
  }
}

template <int LOG2L, int PPT = 8>
struct Smem {
  float2* bufA;
  float2* bufB;
  float2* tw;
  float2* t0s;   // per-thread t_0 values, element i of thread t at i * NT + t
  float2* Bs;    // per-thread B_j multipliers, same layout
  float* sinw;
  float* Vs;
  float* Vis;
  float2* scan_s;
  float* red;
  __device__ __forceinline__ explicit Smem(unsigned char* base) {
    using C = Cfg<LOG2L, PPT>;
    bufA = reinterpret_cast<float2*>(base);
    bufB = bufA + C::PADL;
    tw = bufB + C::PADL;
    t0s = tw + C::L;
    Bs = t0s + C::L;
    sinw = reinterpret_cast<float*>(Bs + C::L);
    Vs = sinw + C::L;
    scan_s = reinterpret_cast<float2*>(Vs + C::L);
    red = reinterpret_cast<float*>(scan_s + C::NW);
    Vis = red + 2 * C::NW;  // only present in the complex-profile kernel (SMEM_CPLX)
  }
  // the tables staged ahead (Cfg::AHEAD)
  __device__ __forceinline__ float4* stage_r() const { return reinterpret_cast<float4*>(t0s); }
  __device__ __forceinline__ float4* stage_ab() const { return reinterpret_cast<float4*>(Vis); }
};

// P consecutive complex values of one thread, 16-byte vector accesses (P even, p 16-byte aligned)
template <int LOG2L, int PPT = 8>
__device__ __forceinline__ void load8(const float2* __restrict__ p, float2 (&v)[PPT]) {
  const float4* q = reinterpret_cast<const float4*>(p);
#pragma unroll
  for (int i = 0; i < PPT / 2; ++i) {
    const float4 x = __ldg(q + i);
    v[2 * i] = make_float2(x.x, x.y);
    v[2 * i + 1] = make_float2(x.z, x.w);
  }
}

template <int LOG2L, int PPT = 8>
__device__ __forceinline__ void store8(float2* p, const float2 (&v)[PPT]) {
  float4* q = reinterpret_cast<float4*>(p);
#pragma unroll
  for (int i = 0; i < PPT / 2; ++i) q[i] = make_float4(v[2 * i].x, v[2 * i].y, v[2 * i + 1].x, v[2 * i + 1].y);
}

// TL row after a step: physical envelope u = (2/L) DST(y), TL = -20 log10|u| + 10 log10 r.
template <int LOG2L, int BC, int PPT = 8>
__device__ __forceinline__ void record_tl(Smem<LOG2L, PPT>& sm, const SolveDesc& d, const float2 (&y)[PPT],
                                          float out_scale, int s, int nrec) {
  const int t = threadIdx.x;
#pragma unroll
  for (int i = 0; i < PPT; ++i) sm.bufA[pidx(PPT * t + i)] = out_scale * y[i];
  __syncthreads();
  float2 u[PPT];
  xform<LOG2L, BC, true, PPT>(sm.bufA, sm.bufB, sm.tw, sm.sinw, sm.scan_s, u);
  const float lr = float(10.0 * log10(d.r0 + double(s + 1) * d.dr));
  float* row = d.tl + (size_t)(d.rec0 + nrec) * d.N;
  constexpr int off = (BC == kBcPeriodic) ? 0 : 1;  // Dirichlet: depth index 0 is the boundary
#pragma unroll
  for (int i = 0; i < PPT; ++i) {
    const int n = PPT * t + i;
    if (n >= off) row[n - off] = fmaf(-10.f, log10f(cabs2(u[i])), lr);
  }
}

// ---------------------------------------------------------------------------------------
// The persistent march: blockIdx.x selects the solve; thread t owns the modes [P t, P t + P).
// A solve without V (terms <= 1) only transforms for its TL rows, and those do not depend on one another:
// gridDim.y CTAs all take the (cheap, diagonal) steps, each transforms every gridDim.y-th row, and the last
// to finish writes the state.  100 steps of N = 255 with a row each: 208 us on one CTA, see launch_march.
// ---------------------------------------------------------------------------------------
template <int LOG2L, bool CPLX, int BC, int PPT = 8>
__global__ void __launch_bounds__(Cfg<LOG2L, PPT>::NT, Cfg<LOG2L, PPT>::MIN_BLOCKS)
    sssp_march_kernel(const SolveDesc* __restrict__ descs, const float2* __restrict__ tw_g,
                      const float* __restrict__ sin_g) {
  using C = Cfg<LOG2L, PPT>;
  constexpr int L = C::L, P = PPT;
  extern __shared__ __align__(16) unsigned char smem_raw[];
  Smem<LOG2L, PPT> sm(smem_raw);
  __shared__ SolveDesc d;
  const int t = threadIdx.x;
  {  // the descriptor lives in shared memory so its fields need no registers
    const int* src = reinterpret_cast<const int*>(descs + blockIdx.x);
    int* dst = reinterpret_cast<int*>(&d);
    for (int i = t; i < int(sizeof(SolveDesc) / sizeof(int)); i += C::NT) dst[i] = src[i];
  }
  load_tables<LOG2L, PPT>(sm.tw, sm.sinw, tw_g, sin_g);
  __syncthreads();
  if (d.terms > 1 && blockIdx.y > 0) return;
  TwRegs<LOG2L, P> twr_v;
  const TwRegs<LOG2L, P>* twr = nullptr;
  if constexpr (C::TWREG) {
    twr_v.load(sm.tw, C::OPREG ? sm.sinw : nullptr);
    twr = &twr_v;
  }
  // register copies of the thread's V row entries (OPREG), else read from sm.Vs / sm.Vis
  float vr[P], vi[P];

  float2 y[P];
  load8<LOG2L, P>(d.yhat + P * t, y);
  const float out_scale = (BC == kBcPeriodic ? 1.0f : 2.0f) / float(L);
  const bool iso = d.terms <= 1;
  const float tol2f = float(d.tol2);
  int status = kStatusOk;
  unsigned int ndst = 0;
  int nrec = 0;
  int node = d.node0;
  double next_r = (node + 1 < d.nodes) ? d.node_r[node + 1] : 1e300;
  constexpr bool cplx = CPLX;  // complex n^2: launched only for solves with an imaginary profile
  auto load_v = [&](int nd) {
    const float* Vg = d.V + (size_t)nd * L;
    const float* Vig = cplx ? d.Vi + (size_t)nd * L : nullptr;
    if constexpr (C::OPREG) {
#pragma unroll
      for (int i = 0; i < P; i += 4) {
        const float4 q = *reinterpret_cast<const float4*>(Vg + P * t + i);
        vr[i] = q.x, vr[i + 1] = q.y, vr[i + 2] = q.z, vr[i + 3] = q.w;
        if constexpr (cplx) {
          const float4 qi = *reinterpret_cast<const float4*>(Vig + P * t + i);
          vi[i] = qi.x, vi[i + 1] = qi.y, vi[i + 2] = qi.z, vi[i + 3] = qi.w;
        }
      }
    } else {
      for (int i = t; i < L; i += C::NT) sm.Vs[i] = Vg[i];
      if constexpr (cplx) {
        for (int i = t; i < L; i += C::NT) sm.Vis[i] = Vig[i];
      }
    }
  };
  if (!iso) load_v(node);
  // Tables staged a stage ahead (A and B) or over the stage (R): each thread copies the entries of its own
  // modes, so no barrier is involved.
  auto stage_ab = [&](int j) {
    const float4* A = reinterpret_cast<const float4*>(d.A + (size_t)j * L + P * t);
    const float4* B = reinterpret_cast<const float4*>(d.B + (size_t)j * L + P * t);
#pragma unroll
    for (int i = 0; i < P / 2; ++i) {
      cp_async16(sm.stage_ab() + i * C::NT + t, A + i);
      cp_async16(sm.stage_ab() + (P / 2 + i) * C::NT + t, B + i);
    }
    cp_async_commit();
  };
  if constexpr (C::AHEAD) {
    if (!iso) stage_ab(0);
  }
  __syncthreads();

  if (iso) {
    // V ignored: every step is the diagonal multiply by G = prod_j R_j
    float4 G[P];
    {
      const float4* g = d.G + P * t;
#pragma unroll
      for (int i = 0; i < P; ++i) G[i] = __ldg(g + i);
    }
    for (int s = 0; s < d.steps; ++s) {
#pragma unroll
      for (int i = 0; i < P; ++i) y[i] = ffmul(G[i], y[i]);
      const long long gs = d.step0 + s + 1;
      if (d.tl_every > 0 && gs % d.tl_every == 0) {
        if (nrec % int(gridDim.y) == int(blockIdx.y)) {
          record_tl<LOG2L, BC, P>(sm, d, y, out_scale, s, nrec);
          ++ndst;
        }
        ++nrec;
      }
    }
    if (gridDim.y > 1) {  // every CTA has read the state it started from: the last one writes the new state
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
  } else {
    for (int s = 0; s < d.steps && status == kStatusOk; ++s) {
      const double rmid = d.r0 + (double(s) + 0.5) * d.dr;
      if (rmid >= next_r) {  // advance to the node in force at this step's midpoint
        while (node + 1 < d.nodes && d.node_r[node + 1] <= rmid) ++node;
        next_r = (node + 1 < d.nodes) ? d.node_r[node + 1] : 1e300;
        load_v(node);
        // first read of Vs is after the syncs of the stage's first transform
      }
      for (int j = 0; j < d.p && status == kStatusOk; ++j) {
        float2 acc[P], tp[P];
        float2 Bj[P], t0r[P];  // register copies of B_j and t_0 (OPREG), else in sm.Bs / sm.t0s
        {
          float2 Aj[P];
          if constexpr (C::AHEAD) {
            cp_async_wait<0>();
#pragma unroll
            for (int i = 0; i < P / 2; ++i) {
              const float4 a = sm.stage_ab()[i * C::NT + t], b = sm.stage_ab()[(P / 2 + i) * C::NT + t];
              Aj[2 * i] = make_float2(a.x, a.y), Aj[2 * i + 1] = make_float2(a.z, a.w);
              Bj[2 * i] = make_float2(b.x, b.y), Bj[2 * i + 1] = make_float2(b.z, b.w);
            }
          } else {
            load8<LOG2L, P>(d.B + (size_t)j * L + P * t, Bj);
            if constexpr (!C::OPREG) {
#pragma unroll
              for (int i = 0; i < P; ++i) sm.Bs[i * C::NT + t] = Bj[i];
            }
            load8<LOG2L, P>(d.A + (size_t)j * L + P * t, Aj);
          }
#pragma unroll
          for (int i = 0; i < P; ++i) {
            const float2 t0 = cmul(Aj[i], y[i]);
            if constexpr (C::OPREG) t0r[i] = t0;
            else sm.t0s[i * C::NT + t] = t0;
            sm.bufA[pidx(P * t + i)] = t0;
            acc[i] = make_float2(0.f, 0.f);
          }
        }
        __syncthreads();
        if constexpr (C::AHEAD) {  // R_j for this stage's end, then A and B of the next stage
#pragma unroll
          for (int i = 0; i < P; ++i) cp_async16(sm.stage_r() + i * C::NT + t, d.R + (size_t)j * L + P * t + i);
          cp_async_commit();
          stage_ab(j + 1 < d.p ? j + 1 : 0);
        }
        xform<LOG2L, BC, true, P>(sm.bufA, sm.bufB, sm.tw, sm.sinw, sm.scan_s, tp, twr);  // t_0 in depth space
        ++ndst;
        float first = 0.f;
        for (int m = 1; m < d.terms; ++m) {
#pragma unroll
          for (int i = 0; i < P; ++i) {
            if constexpr (C::OPREG) {
              if constexpr (cplx) sm.bufA[pidx(P * t + i)] = cmul(make_float2(vr[i], vi[i]), tp[i]);
              else sm.bufA[pidx(P * t + i)] = vr[i] * tp[i];
            } else if constexpr (cplx) {
              sm.bufA[pidx(P * t + i)] = cmul(make_float2(sm.Vs[P * t + i], sm.Vis[P * t + i]), tp[i]);
            } else {
              sm.bufA[pidx(P * t + i)] = sm.Vs[P * t + i] * tp[i];
            }
          }
          __syncthreads();
          xform<LOG2L, BC, false, P>(sm.bufA, sm.bufB, sm.tw, sm.sinw, sm.scan_s, tp, twr);  // T(V t_{m-1})
          ++ndst;
          float nt = 0.f, nw = 0.f;
#pragma unroll
          for (int i = 0; i < P; ++i) {
            tp[i] = cmul(C::OPREG ? Bj[i] : sm.Bs[i * C::NT + t], tp[i]);  // spectral t_m (scaled by 2/L)
            acc[i] = acc[i] + tp[i];
            nt += cabs2(tp[i]);
            nw += cabs2((C::OPREG ? t0r[i] : sm.t0s[i * C::NT + t]) + acc[i]);
          }
          if (m == d.terms - 1) break;
#pragma unroll
          for (int i = 0; i < P; ++i) sm.bufA[pidx(P * t + i)] = tp[i];
          // t_m in depth space, unless its stop test ends the series
          StopHook<C::WS, C::NW, C::MASK> hook{nt, nw, sm.red, m, &first, &status, d.tol2, tol2f};
          if constexpr (C::AHEAD) {
            __syncthreads();
            if (!xform<LOG2L, BC, true, P>(sm.bufA, sm.bufB, sm.tw, sm.sinw, sm.scan_s, tp, twr, hook)) break;
          } else {
            hook.publish();
            __syncthreads();
            if (hook.stop()) break;
            xform<LOG2L, BC, true, P>(sm.bufA, sm.bufB, sm.tw, sm.sinw, sm.scan_s, tp, twr);
          }
          ++ndst;
        }
        {
          const float4* rp = d.R + (size_t)j * L + P * t;
          const float2 bj = d.beta[j];
          if constexpr (C::AHEAD) cp_async_wait<1>();
#pragma unroll
          for (int i = 0; i < P; ++i)
            y[i] = ffmul(C::AHEAD ? sm.stage_r()[i * C::NT + t] : __ldg(rp + i), y[i]) + cmul(bj, acc[i]);
        }
      }
      if (status != kStatusOk) break;
      const long long gs = d.step0 + s + 1;
      if (d.tl_every > 0 && gs % d.tl_every == 0) {
        record_tl<LOG2L, BC, P>(sm, d, y, out_scale, s, nrec);
        ++ndst;
        ++nrec;
      }
    }
  }
  store8<LOG2L, P>(d.yhat + P * t, y);
  // physical envelope for pe_read_field
#pragma unroll
  for (int i = 0; i < P; ++i) sm.bufA[pidx(P * t + i)] = out_scale * y[i];
  __syncthreads();
  float2 u[P];
  xform<LOG2L, BC, true, P>(sm.bufA, sm.bufB, sm.tw, sm.sinw, sm.scan_s, u);
  ++ndst;
  store8<LOG2L, P>(d.field + P * t, u);
  if (t == 0) {
    if (status != kStatusOk) atomicMax(d.status, status);
    atomicAdd(d.ndst, (unsigned long long)ndst);
  }
}

// What setting a starter does beside its transform: the physical field as given (index 0 the zero
// boundary on Dirichlet grids) and a cleared status word.  Null in the transform entry points.
struct StartArgs {
  float2* field = nullptr;
  int* status = nullptr;
  int mirror = 0;  // K > 0: in holds K + 1 values and the grid is their even extension to 2 K points
};

// Point n of the grid, from the caller's values (Dirichlet: N interior points; periodic: all points)
template <int BC>
__device__ __forceinline__ float2 start_value(const float2* in, int n, int mirror) {
  if constexpr (BC == kBcPeriodic) return in[mirror > 0 && n > mirror ? 2 * mirror - n : n];
  else return n == 0 ? make_float2(0.f, 0.f) : in[n - 1];
}

// DST-I of one field per CTA: out = scale * DST(in); field b = blockIdx.x reads N values at
// in + b * in_stride (n = 1..N) and writes L values at out + b * out_stride.
template <int LOG2L, int BC = kBcDirichlet>
__global__ void __launch_bounds__(Cfg<LOG2L>::NT)
    sssp_dst_kernel(const float2* __restrict__ in, float2* __restrict__ out, float scale,
                    const float2* __restrict__ tw_g, const float* __restrict__ sin_g, long long in_stride,
                    long long out_stride, const StartArgs sa) {
  using C = Cfg<LOG2L>;
  extern __shared__ __align__(16) unsigned char smem_raw[];
  Smem<LOG2L> sm(smem_raw);
  const int t = threadIdx.x;
  in += blockIdx.x * in_stride;
  out += blockIdx.x * out_stride;
  load_tables<LOG2L>(sm.tw, sm.sinw, tw_g, sin_g);
  for (int n = t; n < C::L; n += C::NT) {
    const float2 v = start_value<BC>(in, n, sa.mirror);
    sm.bufA[pidx(n)] = v;
    if (sa.field) sa.field[n] = v;
  }
  if (sa.status && t == 0) *sa.status = kStatusOk;
  __syncthreads();
  float2 o[8];
  xform<LOG2L, BC, false>(sm.bufA, sm.bufB, sm.tw, sm.sinw, sm.scan_s, o);
#pragma unroll
  for (int i = 0; i < 8; ++i) o[i] = scale * o[i];
  store8<LOG2L>(out + 8 * t, o);
}

// The same without a transform (grids whose transform is another kernel; FD-SSP plans, which march
// depth values: state = field)
template <int BC>
__global__ void sssp_start_kernel(const float2* __restrict__ in, float2* __restrict__ state, int L, const StartArgs sa) {
  const int n = blockIdx.x * blockDim.x + threadIdx.x;
  if (n == 0) *sa.status = kStatusOk;
  if (n >= L) return;
  const float2 v = start_value<BC>(in, n, sa.mirror);
  sa.field[n] = v;
  if (state) state[n] = v;
}

}  // namespace sssp
