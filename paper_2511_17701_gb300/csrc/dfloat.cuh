// dfloat.cuh -- unevaluated sums of two floats ("double-float", about 48 significant bits).
// GB300's FP64 pipe bounds the FP64 pusher while its FP32 pipe and instruction issue are mostly
// idle, so work carried in pairs of FP32 numbers (Dekker's and Knuth's error-free
// transformations: the rounding error of an FP32 sum is recovered with two-sum, that of a product
// with one fused multiply-add) costs it little. Two kinds of use: a predictor that lands within
// about 1e-14 of an FP64 fixed point, whose result is an FP64 evaluation checked in FP64; and
// quantities whose 2^-48 is enough because they are a small part of what they are added to in
// FP64 (inc.cuh) or are rounded to FP32 (the mixed path's guard zones). A pair has FP32's range of
// exponents: what is outside about 2^-74 to 2^128 has to be kept from it (df_of).
#pragma once
#include <cuda_runtime.h>
#include <stdint.h>

namespace {

struct DF {
  float hi, lo;  // value hi + lo, |lo| <= ulp(hi) / 2
  DF() = default;
  __host__ __device__ constexpr DF(float h, float l) : hi(h), lo(l) {}
  // from a float or an integer constant (exact for |i| < 2^24)
  __host__ __device__ constexpr DF(float f) : hi(f), lo(0.0f) {}
  __host__ __device__ constexpr DF(int i) : hi((float)i), lo(0.0f) {}
  // from a double: meant for literal constants, which the compiler folds (a runtime double
  // would cost FP64 conversions: df_of splits those on the integer pipe)
  __host__ __device__ constexpr DF(double d) : hi((float)d), lo((float)(d - (double)(float)d)) {}
};

// a double constant as a pair, at compile time (literals only: used for the series
// coefficients)
__host__ __device__ constexpr DF dfc(double x) {
  return DF((float)x, (float)(x - (double)(float)x));
}

// The roundings below are explicit (__fadd_rn, __fmul_rn): a compiler that contracted a
// product into a following sum would break the error terms.
// s + e = a + b exactly (Knuth's two-sum)
__device__ __forceinline__ DF two_sum(float a, float b) {
  const float s = __fadd_rn(a, b), bb = __fsub_rn(s, a);
  return DF(s, __fadd_rn(__fsub_rn(a, __fsub_rn(s, bb)), __fsub_rn(b, bb)));
}
// s + e = a + b exactly when |a| >= |b| (or a = 0)
__device__ __forceinline__ DF fast_two_sum(float a, float b) {
  const float s = __fadd_rn(a, b);
  return DF(s, __fsub_rn(b, __fsub_rn(s, a)));
}

// The sum's high parts are added exactly, the low parts rounded: the error is within about
// 2^-47 (|a| + |b|), 11 instructions (20 for a bound relative to |a + b|, which no use needs:
// the terms that cancel here do so mildly).
__device__ __forceinline__ DF operator+(DF a, DF b) {
  const DF s = two_sum(a.hi, b.hi);
  return fast_two_sum(s.hi, __fadd_rn(s.lo, __fadd_rn(a.lo, b.lo)));
}
__device__ __forceinline__ DF operator-(DF a) { return DF(-a.hi, -a.lo); }
__device__ __forceinline__ DF operator-(DF a, DF b) { return a + (-b); }
__device__ __forceinline__ DF operator*(DF a, DF b) {
  const float p = __fmul_rn(a.hi, b.hi);
  float e = fmaf(a.hi, b.hi, -p);  // the product's rounding error, exactly
  e = fmaf(a.hi, b.lo, fmaf(a.lo, b.hi, e));
  return fast_two_sum(p, e);
}
// a b + c without normalising the product first
__device__ __forceinline__ DF fma_(DF a, DF b, DF c) {
  const float p = __fmul_rn(a.hi, b.hi);
  float e = fmaf(a.hi, b.hi, -p);
  e = fmaf(a.hi, b.lo, fmaf(a.lo, b.hi, e));
  const DF s = two_sum(p, c.hi);
  return fast_two_sum(s.hi, __fadd_rn(s.lo, __fadd_rn(e, c.lo)));
}
// a times a power of two (exact)
__device__ __forceinline__ DF df_scale(DF a, float p2) { return DF(a.hi * p2, a.lo * p2); }

// 1/b: the FP32 reciprocal r (within 2 ulp) refined in pairs, r (1 + e + e^2) with
// e = 1 - b r (|e| < 2^-21, so the third order is below 2^-63)
__device__ __forceinline__ DF df_rcp(DF b) {
  const float r = __fdividef(1.0f, b.hi);
  const float p = __fmul_rn(b.hi, r);
  // 1 - b r: 1 - p is exact (p within 2^-21 of 1), the other terms are small
  const DF e = two_sum(__fsub_rn(1.0f, p), -fmaf(b.lo, r, fmaf(b.hi, r, -p)));
  const float q = __fmul_rn(r, e.hi);
  const float ql = fmaf(r, e.hi, -q) + r * fmaf(e.hi, e.hi, e.lo);
  const DF s = fast_two_sum(r, q);
  return fast_two_sum(s.hi, __fadd_rn(s.lo, ql));
}
__device__ __forceinline__ DF operator/(DF a, DF b) { return a * df_rcp(b); }
// 1/sqrt(x): the FP32 value r refined in pairs, r (1 + e/2 + 3 e^2 / 8) with e = 1 - x r^2
// (|e| < 2^-20, so the third order is below 2^-61)
__device__ __forceinline__ DF df_rsqrt(DF x) {
  const float r = rsqrtf(x.hi);
  const float y = __fmul_rn(r, r);
  const DF xr = x * DF(y, fmaf(r, r, -y));
  const DF e = two_sum(__fsub_rn(1.0f, xr.hi), -xr.lo);
  const float h = 0.5f * r;
  const float q = __fmul_rn(h, e.hi);
  const float ql = fmaf(h, e.hi, -q) + h * fmaf(0.75f * e.hi, e.hi, e.lo);
  const DF s = fast_two_sum(r, q);
  return fast_two_sum(s.hi, __fadd_rn(s.lo, ql));
}
__device__ __forceinline__ DF rsqrt_(DF x) { return df_rsqrt(x); }

// a double split into a pair on the integer pipe: hi its leading 24 bits (truncated), lo
// the next 24 of the remaining 29 (rounded by the integer-to-float conversion), so the pair
// holds the double to about 2^-48 of itself. Below 2^-74 the low part is left out (24 bits), below
// 2^-126 the result is zero, from 2^128 on infinite: callers for which that matters test or scale
// the double first (inc_charge, photon_unit).
__device__ __forceinline__ DF df_of(double x) {
  const unsigned hi32 = (unsigned)__double2hiint(x), lo32 = (unsigned)__double2loint(x);
  const unsigned sign = hi32 & 0x80000000u, ex = (hi32 >> 20) & 0x7ffu;
  const int e = (int)ex - 896;  // rebias 1023 -> 127
  float h;
  if (e <= 0) h = __uint_as_float(sign);
  else if (e >= 255) h = __uint_as_float(sign | 0x7f800000u);
  else h = __uint_as_float(sign | ((unsigned)e << 23) | ((hi32 & 0xfffffu) << 3) | (lo32 >> 29));
  float l = 0.0f;
  const int es = (int)ex - 1075 + 127;  // biased FP32 exponent of the low part's unit 2^(ex - 1075)
  if (e > 0 && e < 255 && es >= 1) {
    const unsigned m = lo32 & 0x1fffffffu;  // the 29 bits below hi
    l = (float)m * __uint_as_float((unsigned)es << 23);
    if (sign) l = -l;
  }
  return DF(h, l);
}

}  // namespace
