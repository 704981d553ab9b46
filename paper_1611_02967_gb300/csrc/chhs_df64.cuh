// chhs_df64.cuh -- double-single ("df64") arithmetic: a value carried as an
// unevaluated sum hi + lo of two single-precision numbers, about 48
// significant bits, computed on the single-precision pipes.
//
// GB300 runs double precision at 1/64 of the single-precision rate, and the
// mixed-precision form's one double-precision kernel per iteration -- the
// defect-correction residual f - N(u) -- was bound by that pipe.  The
// residual only has to be accurate to far below the stopping tolerance
// (1e-10 against values of order one), which 48 bits give.  The operations
// are the error-free transformations of Knuth (two-sum) and of Dekker and
// Kahan (the exact product error through a fused multiply-add), combined as
// in the double-single libraries of the GPU literature (for instance
// Thall, "Extended-precision floating-point numbers for GPU computation",
// 2006): a sum or product is formed in single precision together with its
// rounding error, then renormalised.  Every step uses the round-to-nearest
// intrinsics so that the compiler never contracts a product into a
// following sum, which would break the error terms.
//
// Usable from host code too (plain single-precision operations with
// std::fmaf; build with -ffp-contract=off), so the host tests can check
// the arithmetic against long double references.
#pragma once
#include <stdint.h>
#include <string.h>

#if defined(__CUDACC__)
#define DF_HD __host__ __device__ __forceinline__
#else
#include <cmath>
#define DF_HD inline
#endif

namespace chhs_dev {

struct df64 {
  float hi, lo;
};

DF_HD float df_fadd(float a, float b) {
#if defined(__CUDA_ARCH__)
  return __fadd_rn(a, b);
#else
  return a + b;
#endif
}
DF_HD float df_fsub(float a, float b) {
#if defined(__CUDA_ARCH__)
  return __fsub_rn(a, b);
#else
  return a - b;
#endif
}
DF_HD float df_fmul(float a, float b) {
#if defined(__CUDA_ARCH__)
  return __fmul_rn(a, b);
#else
  return a * b;
#endif
}
DF_HD float df_ffma(float a, float b, float c) {
#if defined(__CUDA_ARCH__)
  return __fmaf_rn(a, b, c);
#else
  return std::fmaf(a, b, c);
#endif
}

DF_HD uint64_t df_bits(double x) {
#if defined(__CUDA_ARCH__)
  return (uint64_t)__double_as_longlong(x);
#else
  uint64_t b;
  memcpy(&b, &x, sizeof b);
  return b;
#endif
}
DF_HD float df_from_bits(uint32_t b) {
#if defined(__CUDA_ARCH__)
  return __uint_as_float(b);
#else
  float f;
  memcpy(&f, &b, sizeof f);
  return f;
#endif
}

DF_HD float df_from_uint(uint32_t m) {  // rounded to nearest
#if defined(__CUDA_ARCH__)
  return __uint2float_rn(m);
#else
  return (float)m;
#endif
}

// x split into hi + lo with integer and single-precision operations only (a
// conversion from double runs at the double-precision rate on this GPU): hi is
// x with its significand cut to 24 bits, lo the other 29 rounded to 24, so
// |x - (hi + lo)| <= 2^-48 |x|.  (The residual's error is mostly that of its
// inputs: with lo cut to 23 bits, 2^-46, it was twice as large.)  Magnitudes
// below 2^-126 give 0 (an absolute error far below anything the residual
// resolves), magnitudes beyond the float range and non-finite values give
// +-infinity in hi, so a non-finite state still yields a non-finite residual.
DF_HD df64 df_split(double x) {
  const uint64_t b = df_bits(x);
  const uint32_t hw = (uint32_t)(b >> 32), lw = (uint32_t)b;
  const uint32_t sign = hw & 0x80000000u;
  const int e = (int)((hw >> 20) & 0x7FFu);
  if (e < 897) return df64{df_from_bits(sign), 0.f};
  if (e > 1150) return df64{df_from_bits(sign | 0x7F800000u), 0.f};
  const float hi = df_from_bits(sign | ((uint32_t)(e - 896) << 23) | ((hw & 0xFFFFFu) << 3) | (lw >> 29));
  // the place value of the last bit is 2^(e - 1075), here as 2^-6 2^(e - 1069)
  const float mf = df_fmul(df_from_uint(lw & 0x1FFFFFFFu), 0.015625f);
  const int se = e - 942;
  const float scale = se > 0 ? df_from_bits((uint32_t)se << 23) : 0.f;
  const float lo_mag = df_fmul(mf, scale);
  const float lo = sign ? -lo_mag : lo_mag;
  return df64{hi, lo};
}

// The conversion (float)x with integer instructions wherever the result is a
// normal single: rounded to nearest, ties to even, a carry out of the
// significand raising the exponent (beyond the largest, to infinity).  Zeros,
// subnormal results, infinities and NaNs take the conversion itself.
DF_HD float f64_to_f32_rn(double x) {
  const uint64_t b = df_bits(x);
  const uint32_t hw = (uint32_t)(b >> 32), lw = (uint32_t)b;
  const int e = (int)((hw >> 20) & 0x7FFu) - 896;
  if ((unsigned)(e - 1) >= 254u) return (float)x;
  const uint32_t mag = (uint32_t)e << 23 | (hw & 0xFFFFFu) << 3 | lw >> 29;
  return df_from_bits((hw & 0x80000000u) | (mag + (((lw & 0x1FFFFFFFu) + 0x0FFFFFFFu + (mag & 1u)) >> 29)));
}

// Knuth's two-sum: s + err = a + b exactly.
DF_HD df64 df_two_sum(float a, float b) {
  const float s = df_fadd(a, b);
  const float bb = df_fsub(s, a);
  const float err = df_fadd(df_fsub(a, df_fsub(s, bb)), df_fsub(b, bb));
  return df64{s, err};
}

// Renormalisation for |a| >= |b| (or a = 0): s + err = a + b exactly.
DF_HD df64 df_quick_sum(float a, float b) {
  const float s = df_fadd(a, b);
  return df64{s, df_fsub(b, df_fsub(s, a))};
}

DF_HD df64 df_add(df64 x, df64 y) {
  const df64 s = df_two_sum(x.hi, y.hi);
  return df_quick_sum(s.hi, df_fadd(s.lo, df_fadd(x.lo, y.lo)));
}

DF_HD df64 df_neg(df64 x) { return df64{-x.hi, -x.lo}; }

DF_HD df64 df_sub(df64 x, df64 y) { return df_add(x, df_neg(y)); }

// Product: p + e = x.hi * y.hi exactly through the fused multiply-add; the
// cross terms are added to the error before the renormalisation.
DF_HD df64 df_mul(df64 x, df64 y) {
  const float p = df_fmul(x.hi, y.hi);
  float e = df_ffma(x.hi, y.hi, -p);
  e = df_ffma(x.hi, y.lo, e);
  e = df_ffma(x.lo, y.hi, e);
  return df_quick_sum(p, e);
}

// Sum and product without the renormalisation (8 and 4 instructions instead of
// 11 and 7): the high parts' sum with its error, the low parts added to it.
// The sum is exact to 2^-44 of the larger operand, the product of freshly split
// numbers to 2^-43 of itself.  After a cancellation the result's low part may
// be as large as its high part, and a product with it, which drops the low
// parts' product, is exact to 2^-44 of the product of the magnitudes before the
// cancellation; df_mul_wide keeps that product for such a factor.
DF_HD df64 df_add_raw(df64 x, df64 y) {
  const df64 s = df_two_sum(x.hi, y.hi);
  return df64{s.hi, df_fadd(s.lo, df_fadd(x.lo, y.lo))};
}

DF_HD df64 df_sub_raw(df64 x, df64 y) { return df_add_raw(x, df_neg(y)); }

DF_HD df64 df_mul_raw(df64 x, df64 y) {
  const float p = df_fmul(x.hi, y.hi);
  float e = df_ffma(x.hi, y.hi, -p);
  e = df_ffma(x.hi, y.lo, e);
  return df64{p, df_ffma(x.lo, y.hi, e)};
}

DF_HD df64 df_mul_wide(df64 x, df64 y) {
  const float p = df_fmul(x.hi, y.hi);
  float e = df_ffma(x.hi, y.hi, -p);
  e = df_ffma(x.lo, y.lo, e);
  e = df_ffma(x.hi, y.lo, e);
  return df64{p, df_ffma(x.lo, y.hi, e)};
}

DF_HD float df_to_float(df64 x) { return df_fadd(x.hi, x.lo); }

DF_HD double df_to_double(df64 x) { return (double)x.hi + (double)x.lo; }

// A host double as an exact-as-possible df64 (kernel arguments).
inline df64 df_from_double_host(double x) {
  const float hi = (float)x;
  return df64{hi, (float)(x - (double)hi)};
}

}  // namespace chhs_dev
