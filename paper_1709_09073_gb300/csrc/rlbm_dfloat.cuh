// Double-float arithmetic: a value is the unevaluated sum hi + lo of two FP32
// numbers (about 48 significant bits), built from the error-free
// transformations TwoSum (Knuth) and TwoProduct (via FMA). GB300 executes FP64
// at 1/64 of the FP32 rate, so the mixed-precision step keeps its few
// precision-critical quantities (moment totals, Landau residual, gamma, n, eps)
// in this form on the FP32 pipe. Every operation is written with the
// round-to-nearest intrinsics, which the compiler neither reassociates nor
// contracts into an FMA with a neighbouring product: the error-free
// transformations are exact only as written, and every kernel that inlines
// them gets the same roundings. Each is written once for scalars and for pairs (f2):
// df2 holds two double-floats, the x and y components of a vector, at the
// instruction count of one.
#pragma once
#include <cuda_runtime.h>

#include "rlbm_f32x2.cuh"

namespace rlbm {

template <class V>
struct dft {
  V hi, lo;
};
using df = dft<float>;
using df2 = dft<f2>;

template <class V>
__device__ __forceinline__ dft<V> df_make(V hi, V lo) {
  dft<V> r;
  r.hi = hi;
  r.lo = lo;
  return r;
}

// two double-floats as a pair, and the parts of a pair
__device__ __forceinline__ df2 df_join(df a, df b) { return df_make(f2_make(a.hi, b.hi), f2_make(a.lo, b.lo)); }
__device__ __forceinline__ df df_first(df2 a) { return df_make(f2_lo(a.hi), f2_lo(a.lo)); }
__device__ __forceinline__ df df_second(df2 a) { return df_make(f2_hi(a.hi), f2_hi(a.lo)); }
__device__ __forceinline__ df2 df_dup(df a) { return df_make(f2_dup(a.hi), f2_dup(a.lo)); }

// s + e = a + b exactly
template <class V>
__device__ __forceinline__ dft<V> two_sum(V a, V b) {
  const V s = vadd(a, b);
  const V v = vsub(s, a);
  const V e = vadd(vsub(a, vsub(s, v)), vsub(b, v));
  return df_make(s, e);
}

// s + e = a + b exactly, requires |a| >= |b|
template <class V>
__device__ __forceinline__ dft<V> quick_two_sum(V a, V b) {
  const V s = vadd(a, b);
  return df_make(s, vsub(b, vsub(s, a)));
}

// p + e = a * b exactly
template <class V>
__device__ __forceinline__ dft<V> two_prod(V a, V b) {
  const V p = vmul(a, b);
  return df_make(p, vfma(a, b, vneg(p)));
}

template <class V>
__device__ __forceinline__ dft<V> df_add(dft<V> a, dft<V> b) {
  dft<V> s = two_sum(a.hi, b.hi);
  s.lo = vadd(s.lo, vadd(a.lo, b.lo));
  return quick_two_sum(s.hi, s.lo);
}

template <class V>
__device__ __forceinline__ dft<V> df_add(dft<V> a, V b) {
  dft<V> s = two_sum(a.hi, b);
  s.lo = vadd(s.lo, a.lo);
  return quick_two_sum(s.hi, s.lo);
}

template <class V>
__device__ __forceinline__ dft<V> df_neg(dft<V> a) { return df_make(vneg(a.hi), vneg(a.lo)); }
template <class V>
__device__ __forceinline__ dft<V> df_sub(dft<V> a, dft<V> b) { return df_add(a, df_neg(b)); }

template <class V>
__device__ __forceinline__ dft<V> df_mul(dft<V> a, dft<V> b) {
  dft<V> p = two_prod(a.hi, b.hi);
  p.lo = vfma(a.hi, b.lo, vfma(a.lo, b.hi, p.lo));
  return quick_two_sum(p.hi, p.lo);
}

template <class V>
__device__ __forceinline__ dft<V> df_mul(dft<V> a, V b) {
  dft<V> p = two_prod(a.hi, b);
  p.lo = vfma(a.lo, b, p.lo);
  return quick_two_sum(p.hi, p.lo);
}

// exact scaling by a power of two
__device__ __forceinline__ df df_scale(df a, float pow2) { return df_make(__fmul_rn(a.hi, pow2), __fmul_rn(a.lo, pow2)); }

// 1 / sqrt(a): rsqrtf seed and one Newton step evaluated in double-float
__device__ __forceinline__ df df_rsqrt(df a) {
  const float g = rsqrtf(a.hi);
  // e = 1 - a g^2 (small), g1 = g + g e / 2
  const df ag2 = df_mul(df_mul(a, g), g);
  const float e = __fsub_rn(__fsub_rn(1.0f, ag2.hi), ag2.lo);
  return quick_two_sum(g, __fmul_rn(__fmul_rn(0.5f, g), e));
}

// FP32 to FP64 on the integer pipe, with the roundings of the FP64 instructions: those
// take the FP64 unit 64 clocks for a warp, these about 20 (read-out of a 4096^2 BE
// domain: 1,383 -> 1,130 us). Values outside the ranges stated take the instructions.
// float -> double (exact): zeros and normal values
__device__ __forceinline__ double f32_to_f64(float x) {
  const unsigned b = __float_as_uint(x), m = b & 0x7fffffffu;
  if (m - 0x00800000u >= 0x7f000000u && m) return (double)x;  // denormal, infinity, NaN
  const unsigned hi = (b & 0x80000000u) | (m ? (m >> 3) + 0x38000000u : 0u);
  return __hiloint2double((int)hi, (int)(b << 29));
}
// the double nearest to hi + lo, |lo| <= ulp(hi) / 2: lo, rounded to a whole number of
// ulps of the result, is added to hi's bit pattern. |hi| from 2^-70, and not a power of two
// that lo reduces (the ulp halves there)
__device__ __forceinline__ double df_to_f64(df a) {
  const unsigned b = __float_as_uint(a.hi), m = b & 0x7fffffffu, e = m >> 23;
  if (e < 57u || e == 255u || !(b & 0x7fffffu)) return f32_to_f64(a.hi) + f32_to_f64(a.lo);
  const int n = __float2int_rn(__fmul_rn(a.lo, __uint_as_float((306u - e) << 23)));
  const long long mag = ((long long)((m >> 3) + 0x38000000u) << 32) + (long long)(unsigned long long)(m << 29) +
                        (long long)((b >> 31) ? -n : n);
  return __hiloint2double((int)((unsigned)(mag >> 32) | (b & 0x80000000u)), (int)mag);
}

template <class V>
__device__ __forceinline__ V df_to_float(dft<V> a) { return vadd(a.hi, a.lo); }

}  // namespace rlbm
