// Double-float arithmetic, and FP64 reciprocals and roots that spare the FP64
// units (device code).
#pragma once
#include "ctm_internal.h"

// ---------------------------------------------------------------------------
// Double-float arithmetic (a value is an unevaluated sum hi + lo of two FP32
// numbers, about 48 significand bits; Dekker 1971, Knuth's TwoSum): the
// precision form's Jacobi runs its dot products and row rotations on the
// FP32 pipe, which this part executes at 64 times its FP64 rate.  The
// intrinsics below are never contracted into fused multiply-adds, which the
// error-free transformations rely on.
// ---------------------------------------------------------------------------
struct df2 {
  float h, l;
};

__device__ __forceinline__ df2 df_of(double x) {
  const float h = __double2float_rn(x);
  return {h, __double2float_rn(x - (double)h)};
}

__device__ __forceinline__ double df_val(df2 a) { return (double)a.h + (double)a.l; }

// s + e = a + b exactly
__device__ __forceinline__ void two_sum(float a, float b, float& s, float& e) {
  s = __fadd_rn(a, b);
  const float bb = __fadd_rn(s, -a);
  e = __fadd_rn(__fadd_rn(a, -__fadd_rn(s, -bb)), __fadd_rn(b, -bb));
}

// acc += a b: the leading product exactly (its rounding error by an FMA), the
// cross terms and the tails in FP32, the leading sum's rounding error carried
// into acc.l
__device__ __forceinline__ void acc_mul(df2& acc, df2 a, df2 b) {
  const float p = __fmul_rn(a.h, b.h);
  float e = __fmaf_rn(a.h, b.h, -p);
  e = __fmaf_rn(a.h, b.l, e);
  e = __fmaf_rn(a.l, b.h, e);
  float s, t;
  two_sum(acc.h, p, s, t);
  acc.h = s;
  acc.l = __fadd_rn(acc.l, __fadd_rn(t, e));
}

__device__ __forceinline__ df2 df_norm(df2 a) {
  df2 r;
  two_sum(a.h, a.l, r.h, r.l);
  return r;
}

__device__ __forceinline__ df2 df_negate(df2 a) { return {-a.h, -a.l}; }

// a b, the leading product exactly, the cross terms in FP32
__device__ __forceinline__ df2 df_mul(df2 a, df2 b) {
  const float p = __fmul_rn(a.h, b.h);
  float e = __fmaf_rn(a.h, b.h, -p);
  e = __fmaf_rn(a.h, b.l, e);
  e = __fmaf_rn(a.l, b.h, e);
  return {p, e};
}

__device__ __forceinline__ df2 df_add(df2 a, df2 b) {
  df2 r;
  two_sum(a.h, b.h, r.h, r.l);
  r.l = __fadd_rn(r.l, __fadd_rn(a.l, b.l));
  return df_norm(r);
}

// 1/sqrt(a) of a normalised a > 0: an FP32 root refined by one Householder step
// of third order, x (1 + e/2 + 3 e^2/8) with e = 1 - a x^2 in double-float
__device__ __forceinline__ df2 df_rsqrt(df2 a) {
  const float x = rsqrtf(a.h);
  const df2 xx = {x, 0.f};
  const df2 ax2 = df_norm(df_mul(df_norm(df_mul(a, xx)), xx));
  const float e = __fadd_rn(__fadd_rn(1.0f, -ax2.h), -ax2.l);
  df2 r = {x, __fmul_rn(x, __fmul_rn(e, __fmaf_rn(0.375f, e, 0.5f)))};
  return df_norm(r);
}

// ---------------------------------------------------------------------------
// FP64 reciprocals and reciprocal roots from an FP32 seed and one step of third
// order (Householder, The Numerical Treatment of a Single Nonlinear Equation,
// 1970): three to five FP64 instructions in place of a divide's or a root's
// serial chain.  Scaling and conversion run on the integer pipe.
// ---------------------------------------------------------------------------
// 1/a to 2^-52 of itself, for 2^-1021 <= a < 2^1021 (a and 1/a normal):
// x (1 + e + e^2) with e = 1 - a x below 2^-21
__device__ __forceinline__ double rcp64_pos(double a) {
  const long long b = __double_as_longlong(a);
  const int ex = (int)(b >> 52) - 1023;
  const double m = __longlong_as_double(b - ((long long)ex << 52));  // [1, 2)
  const double x = f2d_bits(__frcp_rn(d2f_bits(m)));
  const double e = fma(-m, x, 1.0);
  const double r = fma(x, fma(e, e, e), x);
  return __longlong_as_double(__double_as_longlong(r) - ((long long)ex << 52));
}

// the same for either sign
__device__ __forceinline__ double rcp64_normal(double a) {
  const long long b = __double_as_longlong(a), sign = b & (long long)0x8000000000000000ull;
  return __longlong_as_double(__double_as_longlong(rcp64_pos(__longlong_as_double(b ^ sign))) | sign);
}

// 1/sqrt(a) of a normal a > 0 to 2^-52 of itself: the argument scaled into [1, 4),
// the step's error (5/16) e^3 with |e| below 2^-21
__device__ __forceinline__ double rsqrt64_normal(double a) {
  const long long b = __double_as_longlong(a);
  const int ex = (int)(b >> 52) - 1023, half = ex >> 1;                  // a = m 4^half, m in [1, 4)
  const double m = __longlong_as_double(b - ((long long)half << 53));
  const double x = f2d_bits(rsqrtf(d2f_bits(m)));
  const double e = fma(-(m * x), x, 1.0);
  const double r = fma(x * e, fma(0.375, e, 0.5), x);
  return __longlong_as_double(__double_as_longlong(r) - ((long long)half << 52));
}

// the same for every a: CUDA's function for zero, subnormals, infinity, NaN and a < 0
__device__ __forceinline__ double rsqrt64(double a) {
  const unsigned E = (unsigned)(__double_as_longlong(a) >> 52);  // with the sign bit on top
  return E - 1u < 2046u ? rsqrt64_normal(a) : rsqrt(a);
}
