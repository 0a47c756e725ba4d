// Double-float ("df64") arithmetic: a value is the unevaluated sum hi + lo of two FP32 numbers
// with |lo| <= ulp(hi) / 2, which carries a 48-bit significand.  GB300 runs FP32 at 64 times its
// FP64 rate, so an FFT written in df64 on the FP32 pipes delivers FP64-class accuracy
// (normwise relative error ~1e-14 per transform) several times faster than native FP64.
//
// The primitives are the classical error-free transformations (Knuth's TwoSum, Dekker's
// FastTwoSum, and the FMA form of TwoProduct).  Every FP32 operation that belongs to an
// error-free transformation uses an explicit round-to-nearest intrinsic: the compiler never
// fuses those into an FMA, which would break the exactness the transformations rely on.
//
// Additions are the "sloppy" variant: the error is bounded by a small multiple of
// 2^-48 (|a| + |b|), not of |a + b|.  That is the bound an FFT's normwise error analysis uses,
// and it is what FP64 itself guarantees for a sum up to the constant.
#pragma once

#include <cuda_runtime.h>
#include <stdint.h>

#include "fft_smem.cuh"

namespace mm {

struct df {
  float hi, lo;
  df() = default;
  __host__ __device__ constexpr df(float h, float l, int) : hi(h), lo(l) {}
  // rounding split of a double: hi = fl32(d), lo = fl32(d - hi)
  __host__ __device__ constexpr explicit df(double d)
      : hi((float)d), lo((float)(d - (double)(float)d)) {}
};

__device__ __forceinline__ df df_make(float h, float l) { return df(h, l, 0); }

// s + e = a + b exactly (no ordering assumption)
__device__ __forceinline__ void two_sum(float a, float b, float& s, float& e) {
  s = __fadd_rn(a, b);
  const float bb = __fsub_rn(s, a);
  e = __fadd_rn(__fsub_rn(a, __fsub_rn(s, bb)), __fsub_rn(b, bb));
}
// s + e = a + b exactly, given |a| >= |b| (or a == 0)
__device__ __forceinline__ df fast_two_sum(float a, float b) {
  const float s = __fadd_rn(a, b);
  return df_make(s, __fsub_rn(b, __fsub_rn(s, a)));
}

__device__ __forceinline__ df operator+(df a, df b) {
  float s, e;
  two_sum(a.hi, b.hi, s, e);
  e = __fadd_rn(e, __fadd_rn(a.lo, b.lo));
  return fast_two_sum(s, e);
}
__device__ __forceinline__ df operator-(df a) { return df_make(-a.hi, -a.lo); }
__device__ __forceinline__ df operator-(df a, df b) { return a + (-b); }
__device__ __forceinline__ df operator*(df a, df b) {
  const float p = __fmul_rn(a.hi, b.hi);
  float e = __fmaf_rn(a.hi, b.hi, -p);            // exact error of the leading product
  e = __fmaf_rn(a.hi, b.lo, e);
  e = __fmaf_rn(a.lo, b.hi, e);
  return fast_two_sum(p, e);
}
__device__ __forceinline__ df& operator+=(df& a, df b) { return a = a + b; }

// Exact FP32 -> FP64 widening by moving the fields of the IEEE-754 encodings (sign, exponent
// re-biased by 1023 - 127, significand shifted by 52 - 23) with integer instructions: on GB300 the
// conversion instruction runs on the FP64 pipe, 1/64 of the FP32 rate.  Zeros and subnormals map
// to a signed zero (a df64 low part is subnormal only when |hi| < 2^-102); infinities and NaNs
// keep their class.
__device__ __forceinline__ double f32_to_f64_bits(float f) {
  const uint32_t u = __float_as_uint(f);
  const uint32_t e = (u >> 23) & 0xffu;
  const uint64_t sign = (uint64_t)(u >> 31) << 63;
  if (e == 0) return __longlong_as_double((long long)sign);
  const uint64_t ed = (e == 0xffu) ? 0x7ffull : (uint64_t)(e + 896u);
  const uint64_t man = (uint64_t)(u & 0x7fffffu) << 29;
  return __longlong_as_double((long long)(sign | (ed << 52) | man));
}

// FP64 -> FP32, rounded to nearest even, by moving and rounding the encoding with integer instructions (the
// conversion instruction runs on the FP64 pipe, 1/64 of the FP32 rate).  |d| below 2^-126 gives a signed zero,
// magnitudes of 2^127 and more and NaN are not for it.
__device__ __forceinline__ float f64_to_f32_bits(double d) {
  const uint64_t u = (uint64_t)__double_as_longlong(d);
  const uint32_t sign = (uint32_t)(u >> 32) & 0x80000000u;
  const uint64_t mag = u & 0x7fffffffffffffffull;
  if (mag < ((uint64_t)(1023 - 126) << 52)) return __uint_as_float(sign);
  const uint64_t r = mag + 0x0fffffffull + ((mag >> 29) & 1);   // round the 29 dropped bits, ties to even
  return __uint_as_float(sign | ((uint32_t)(r >> 29) - (896u << 23)));
}

// exact widening of each part, then one FP64 rounding of their sum
__device__ __forceinline__ double df_to_double(df a) { return f32_to_f64_bits(a.hi) + f32_to_f64_bits(a.lo); }

// a b + c d with one renormalisation: both leading products and their exact errors, one TwoSum,
// and the low-order cross terms folded into the error word (19 FP32 operations instead of 25
// for two products and a sum)
__device__ __forceinline__ df df_prod_sum(df a, df b, df c, df d) {
  const float p1 = __fmul_rn(a.hi, b.hi);
  const float p2 = __fmul_rn(c.hi, d.hi);
  const float e1 = __fmaf_rn(a.hi, b.hi, -p1);
  const float e2 = __fmaf_rn(c.hi, d.hi, -p2);
  float s, e;
  two_sum(p1, p2, s, e);
  float t = __fadd_rn(e1, e2);
  t = __fmaf_rn(a.hi, b.lo, t);
  t = __fmaf_rn(a.lo, b.hi, t);
  t = __fmaf_rn(c.hi, d.lo, t);
  t = __fmaf_rn(c.lo, d.hi, t);
  return fast_two_sum(s, __fadd_rn(e, t));
}

// ---- complex double-float values ---------------------------------------------------------------
// (x, y) = (hi.x + lo.x, hi.y + lo.y): both high words in one register pair, both low words in another, so
// that the error-free transformations of the two components run as packed FP32 instructions (half the
// instructions of two scalar ones; the same lane operations per clock).  This is also their layout in
// memory (tables, shared memory).
struct __align__(16) dfc {
  float2 hi, lo;
};
template <> struct V2<df> { using t = dfc; };
template <> struct GenericProduct<dfc> { static constexpr bool value = false; };

__device__ __forceinline__ dfc dfc_make(df x, df y) { return dfc{make_float2(x.hi, y.hi), make_float2(x.lo, y.lo)}; }
__device__ __forceinline__ df dfc_x(dfc a) { return df_make(a.hi.x, a.lo.x); }
__device__ __forceinline__ df dfc_y(dfc a) { return df_make(a.hi.y, a.lo.y); }
__device__ __forceinline__ float2 neg2(float2 a) { return make_float2(-a.x, -a.y); }
__device__ __forceinline__ float2 sub2_rn(float2 a, float2 b) { return __ffma2_rn(b, make_float2(-1.f, -1.f), a); }
__device__ __forceinline__ float2 swap2(float2 a) { return make_float2(a.y, a.x); }
__device__ __forceinline__ void two_sum2(float2 a, float2 b, float2& s, float2& e) {
  s = __fadd2_rn(a, b);
  const float2 bb = sub2_rn(s, a);
  e = __fadd2_rn(sub2_rn(a, sub2_rn(s, bb)), sub2_rn(b, bb));
}
__device__ __forceinline__ dfc fast_two_sum2(float2 a, float2 b) {
  const float2 s = __fadd2_rn(a, b);
  return dfc{s, sub2_rn(b, sub2_rn(s, a))};
}
__device__ __forceinline__ dfc c_add(dfc a, dfc b) {
  float2 s, e;
  two_sum2(a.hi, b.hi, s, e);
  return fast_two_sum2(s, __fadd2_rn(e, __fadd2_rn(a.lo, b.lo)));
}
__device__ __forceinline__ dfc c_neg(dfc a) { return dfc{neg2(a.hi), neg2(a.lo)}; }
__device__ __forceinline__ dfc c_sub(dfc a, dfc b) { return c_add(a, c_neg(b)); }
// a b + c d per component, as df_prod_sum
__device__ __forceinline__ dfc dfc_prod_sum(dfc a, dfc b, dfc c, dfc d) {
  const float2 p1 = __fmul2_rn(a.hi, b.hi), p2 = __fmul2_rn(c.hi, d.hi);
  const float2 e1 = __ffma2_rn(a.hi, b.hi, neg2(p1)), e2 = __ffma2_rn(c.hi, d.hi, neg2(p2));
  float2 s, e;
  two_sum2(p1, p2, s, e);
  float2 t = __fadd2_rn(e1, e2);
  t = __ffma2_rn(a.hi, b.lo, t);
  t = __ffma2_rn(a.lo, b.hi, t);
  t = __ffma2_rn(c.hi, d.lo, t);
  t = __ffma2_rn(c.lo, d.hi, t);
  return fast_two_sum2(s, __fadd2_rn(e, t));
}
// a b + c per component
__device__ __forceinline__ dfc dfc_fma(dfc a, dfc b, dfc c) {
  const float2 p = __fmul2_rn(a.hi, b.hi);
  const float2 e = __ffma2_rn(a.hi, b.hi, neg2(p));
  float2 s, e2;
  two_sum2(p, c.hi, s, e2);
  float2 t = __fadd2_rn(__fadd2_rn(e, e2), c.lo);
  t = __ffma2_rn(a.hi, b.lo, t);
  t = __ffma2_rn(a.lo, b.hi, t);
  return fast_two_sum2(s, t);
}
__device__ __forceinline__ dfc dfc_xx(dfc a) { return dfc{make_float2(a.hi.x, a.hi.x), make_float2(a.lo.x, a.lo.x)}; }
__device__ __forceinline__ dfc dfc_yy(dfc a) { return dfc{make_float2(a.hi.y, a.hi.y), make_float2(a.lo.y, a.lo.y)}; }
// (-y, x): i a
__device__ __forceinline__ dfc dfc_i(dfc a) {
  return dfc{make_float2(-a.hi.y, a.hi.x), make_float2(-a.lo.y, a.lo.x)};
}
__device__ __forceinline__ dfc dfc_conj(dfc a) {
  return dfc{make_float2(a.hi.x, -a.hi.y), make_float2(a.lo.x, -a.lo.y)};
}
__device__ __forceinline__ dfc c_mul(dfc a, dfc b) { return dfc_prod_sum(dfc_xx(a), b, dfc_yy(a), dfc_i(b)); }
// a * conj(b)
__device__ __forceinline__ dfc c_mulc(dfc a, dfc b) { return c_mul(a, dfc_conj(b)); }

template <bool FWD>
__device__ __forceinline__ dfc rot16(dfc a, int e) {
  e &= 15;
  if (e == 0) return a;
  if (e == 8) return c_neg(a);
  if (e == 4) return FWD ? c_neg(dfc_i(a)) : dfc_i(a);
  if (e == 12) return FWD ? dfc_i(a) : c_neg(dfc_i(a));
  return c_mul(a, dfc_make(df(cos16(e)), df(FWD ? -sin16(e) : sin16(e))));
}
template <bool FWD>
__device__ __forceinline__ void dft4(dfc& a0, dfc& a1, dfc& a2, dfc& a3) {
  const dfc s02 = c_add(a0, a2), d02 = c_sub(a0, a2), s13 = c_add(a1, a3), jd = dfc_i(c_sub(a1, a3));
  a0 = c_add(s02, s13);
  a2 = c_sub(s02, s13);
  a1 = FWD ? c_sub(d02, jd) : c_add(d02, jd);
  a3 = FWD ? c_add(d02, jd) : c_sub(d02, jd);
}

// 16-byte read-only load of a df64 complex value
template <>
__device__ __forceinline__ dfc ldg_c<dfc>(const dfc* p) {
  const float4 v = __ldg(reinterpret_cast<const float4*>(p));
  return dfc{make_float2(v.x, v.y), make_float2(v.z, v.w)};
}

}  // namespace mm
