// Shared pieces of the fused pass over X: link modes, the pass's view of the
// solver state, 16-byte vector loads of every storage type of X, and the
// compensated FP32 pair arithmetic used for dot products and accumulations.
#pragma once
#include <cuda_bf16.h>
#include <cuda_fp8.h>

#include "common.cuh"

namespace relax {

enum Link : int {
  LINK_LS = 0,         // NF=1 NB=1: r = 2(z - y)
  LINK_LOGISTIC = 1,   // NF=1 NB=2: r = grad at z, r_y = grad at (1+mu) z - mu z_prev
  LINK_IDENT = 2,      // NF=1 NB=1: r = z             (power iteration on X'X)
  LINK_CERT_LS = 3,    // NF=2 NB=1: F at z0, r = 2(z1 - y)
  LINK_CERT_LOGI = 4,  // NF=2 NB=1: F at z0, r = grad at z1
  // both dual points of a certificate in one pass: NF=1 NB=2, F at z0,
  // r0 = the link at zd = ps.zprev (the loop's best dual point), r1 = the link
  // at z0 (zeta = -grad F(X beta)); the loss sums are F, the dual terms at zd
  // and those at z0
  LINK_CERT2_LS = 5,
  LINK_CERT2_LOGI = 6,
};

// Device-resident solver state that the pass reads (pointers rotate between
// iterations, so a captured graph can replay the same launches).
struct PassState {
  const void* beta;      // forward vector 0 (beta^t)
  const void* beta2;     // forward vector 1 (certification)
  void* zout;            // z^t output (logistic; NULL otherwise)
  const void* zprev;     // z^{t-1} (logistic)
  double mom;            // tentative momentum mu for z_y
  int done;              // solver finished: pass returns immediately
};

template <typename TX> struct XTraits;
// 16-byte vectors of X from shared memory
template <> struct XTraits<double> {
  static constexpr int VEC = 2;
  template <typename TA> __device__ static void cvt(const double2 v, TA* o) { o[0] = (TA)v.x; o[1] = (TA)v.y; }
  template <typename TA> __device__ static void load(const double* p, TA* o) { cvt(*reinterpret_cast<const double2*>(p), o); }
};
template <> struct XTraits<float> {
  static constexpr int VEC = 4;
  template <typename TA> __device__ static void cvt(const float4 v, TA* o) {
    o[0] = (TA)v.x; o[1] = (TA)v.y; o[2] = (TA)v.z; o[3] = (TA)v.w;
  }
  template <typename TA> __device__ static void load(const float* p, TA* o) { cvt(*reinterpret_cast<const float4*>(p), o); }
};
// Float-float sums (Knuth's TwoSum; about 48 significant bits from FP32
// instructions).  This GPU issues FP64 arithmetic, comparisons and
// conversions at about 1.6 lanes per clock per SM against about 112 for FP32
// (measured), so the loop's per-coordinate work on FP32 data (the FAST
// instantiation) is FP32 with float-float sums.
struct ffs {
  float hi, lo;
};
// s += x
__device__ __forceinline__ void ff_acc(ffs& s, float x) {
  const float t = s.hi + x;
  const float bp = t - s.hi;
  s.lo += (s.hi - (t - bp)) + (x - bp);
  s.hi = t;
}
// s += x for an FP64 x (split into two floats first)
__device__ __forceinline__ void ff_acc(ffs& s, double x) {
  const float h = (float)x;
  ff_acc(s, h);
  s.lo += (float)(x - (double)h);
}
// a + b, renormalised; symmetric in a and b (every lane of a butterfly gets
// the same bits)
__device__ __forceinline__ ffs ff_add(ffs a, ffs b) {
  const float t = a.hi + b.hi;
  const float bp = t - a.hi;
  const float e = (a.hi - (t - bp)) + (b.hi - bp);
  const float lo = e + (a.lo + b.lo);
  const float h = t + lo;
  return ffs{h, lo - (h - t)};
}
__device__ __forceinline__ ffs ff_of(double x) {
  const float h = (float)x;
  return ffs{h, (float)(x - (double)h)};
}
__device__ __forceinline__ bool is_zero_bits(double x) { return (__double_as_longlong(x) << 1) == 0; }

// The logistic loss terms of one row in FP32 (the FAST loop), t = y z:
// log(1 + exp(-t)), and the entropy -(u log u + v log v) of u = 1/(1 + e^t),
// v = 1 - u, written with e = exp(-|t|) <= 1 and L = log1p(e) so that
// neither term loses its small part when the sigmoid saturates.
__device__ __forceinline__ void logistic_terms_f(float t, float& f, float& h) {
  const float s = fabsf(t);
  const float e = expf(-s);
  const float L = log1pf(e);
  f = fmaxf(-t, 0.f) + L;
  const float big = 1.f / (1.f + e), small = e * big;   // the two probabilities
  // t >= 0: u = small (pays s + L), v = big (pays L); t < 0 the other way
  h = small * (s + L) + big * L;
}

// log(1 + exp(-t)) computed stably, in double
__device__ __forceinline__ double softplus_neg(double t) {
  return fmax(-t, 0.0) + log1p(exp(-fabs(t)));
}
// -(u log u + (1-u) log(1-u)) with u = 1/(1+exp(t)), in double
__device__ __forceinline__ double entropy_of(double t) {
  const double u = 1.0 / (1.0 + exp(t));
  const double v = 1.0 / (1.0 + exp(-t));
  double h = 0.0;
  if (u > 0.0) h -= u * log(u);
  if (v > 0.0) h -= v * log(v);
  return h;
}

// Compensated accumulation of FP32 partial sums into an (hi, lo) FP32 pair
// (Knuth's TwoSum): hi + lo carries the running sum to about twice the FP32
// precision without FP64 arithmetic.
// Packed FP32 pairs: Blackwell's f32x2 add / sub / fma issue one instruction
// for two independent FP32 operations, each rounded exactly as the scalar
// instruction rounds it (IEEE round to nearest even).
__device__ __forceinline__ unsigned long long f2_bits(float2 v) {
  return ((unsigned long long)__float_as_uint(v.y) << 32) | __float_as_uint(v.x);
}
__device__ __forceinline__ float2 f2_of(unsigned long long b) {
  return make_float2(__uint_as_float((unsigned)b), __uint_as_float((unsigned)(b >> 32)));
}
// a * b + c per half
__device__ __forceinline__ float2 fma2(float2 a, float2 b, float2 c) {
  unsigned long long r;
  asm("fma.rn.f32x2 %0, %1, %2, %3;" : "=l"(r) : "l"(f2_bits(a)), "l"(f2_bits(b)), "l"(f2_bits(c)));
  return f2_of(r);
}
__device__ __forceinline__ float2 add2(float2 a, float2 b) {
  unsigned long long r;
  asm("add.rn.f32x2 %0, %1, %2;" : "=l"(r) : "l"(f2_bits(a)), "l"(f2_bits(b)));
  return f2_of(r);
}
__device__ __forceinline__ float2 mul2(float2 a, float2 b) {
  unsigned long long r;
  asm("mul.rn.f32x2 %0, %1, %2;" : "=l"(r) : "l"(f2_bits(a)), "l"(f2_bits(b)));
  return f2_of(r);
}
__device__ __forceinline__ float2 sub2(float2 a, float2 b) {
  unsigned long long r;
  asm("sub.rn.f32x2 %0, %1, %2;" : "=l"(r) : "l"(f2_bits(a)), "l"(f2_bits(b)));
  return f2_of(r);
}
// two_sum_acc (below) on both halves of a pair
__device__ __forceinline__ void two_sum_acc2(float2& hi, float2& lo, float2 a) {
  const float2 s = add2(hi, a);
  const float2 bp = sub2(s, hi);
  const float2 err = add2(sub2(hi, sub2(s, bp)), sub2(a, bp));
  hi = s;
  lo = add2(lo, err);
}

// (hi, lo) += x (bh + bl) per half, bh and bl with nb = -bh: the product formed
// exactly as the pair (x bh, x bh - fl(x bh)) plus x bl, the sum by TwoSum;
// eleven packed instructions for two terms
__device__ __forceinline__ void dot_ff2(float2& hi, float2& lo, float2 x, float2 bh, float2 nb, float2 bl) {
  const float2 n = mul2(x, nb);                      // -fl(x bh)
  const float2 e = fma2(x, bl, fma2(x, bh, n));
  const float2 s = sub2(hi, n);
  const float2 bp = sub2(s, hi);
  const float2 err = sub2(sub2(hi, sub2(s, bp)), add2(n, bp));
  hi = s;
  lo = add2(lo, add2(err, e));
}

__device__ __forceinline__ void two_sum_acc(float& hi, float& lo, float a) {
  const float s = hi + a;
  const float bp = s - hi;
  const float err = (hi - (s - bp)) + (a - bp);
  hi = s;
  lo += err;
}

}  // namespace relax
