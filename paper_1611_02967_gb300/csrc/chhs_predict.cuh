// chhs_predict.cuh -- how many V-cycles the step's loop runs before the next
// stopping norm.  Usable from host code.
//
// The contraction per V-cycle measured over the last iteration,
// rho = (num/den)^(1/ran) within [0.001, 0.9], predicts how many V-cycles the
// norms (r against tol, the pointwise rmax against tol_max) still need, rounded
// to the nearest.
//
// One thread decides this at the end of every norm, on the critical path of
// every iteration: with log and pow in double precision (chains of FP64
// instructions of ~64 cycles each) it took ~8 us.  So it runs in single
// precision, with log2 of a double taken from its exponent and its leading
// significand bits, and a bound on its error; where a tie lies within the
// bound (about one decision in a thousand) the double-precision prediction
// decides.  The count is that one's always.
#pragma once
#include <math.h>

#include "chhs_df64.cuh"

namespace chhs_dev {

DF_HD float log2_f64(double x) {  // x > 0, normal
  const uint64_t b = df_bits(x);
  return (float)((int)(b >> 52) - 1023) + log2f(df_from_bits(0x3F800000u | ((uint32_t)(b >> 29) & 0x7FFFFFu)));
}

// The prediction in double precision.
#if defined(__CUDACC__)
static __host__ __device__ __noinline__
#else
inline
#endif
double predict_f64(double r, double rmax, double tol, double tol_max, double num, double den, int ran) {
  const double lr = log(fmin(fmax(pow(num / den, 1.0 / ran), 1e-3), 0.9));
  double need = r > tol ? log(tol / r) / lr : 0.0;
  if (rmax > tol_max) need = fmax(need, log(tol_max / rmax) / lr);
  return need;
}

// V-cycles of the next iteration, 1 .. cap (cap >= 1).
DF_HD int predict_inner(double r, double rmax, double tol, double tol_max, double num, double den, int ran, int cap) {
  if (cap <= 1) return 1;
  const float ln = log2_f64(num), ld = log2_f64(den);
  const float lr = fminf(fmaxf((ln - ld) / (float)ran, -9.9657843f), -0.15200309f);
  float need = 0.f, err = 0.f;
  auto row = [&](double bound, double value) {
    const float lb = log2_f64(bound), lv = log2_f64(value), n = (lb - lv) / lr;
    // each log2 is off by at most 2^-23 of its size and of its significand's; three times that
    const float e = -4e-7f * ((1.f + fabsf(lb) + fabsf(lv)) + n * (1.f + fabsf(ln) + fabsf(ld))) / lr;
    need = fmaxf(need, n);
    err = fmaxf(err, e);
  };
  if (r > tol) row(tol, r);
  if (rmax > tol_max) row(tol_max, rmax);
  const float x = need + 0.5f, tie = rintf(x);
  if (tie >= 2.f && tie <= (float)cap && fabsf(x - tie) <= err) {
    const int n = (int)floor(predict_f64(r, rmax, tol, tol_max, num, den, ran) + 0.5);
    return n < 1 ? 1 : n > cap ? cap : n;
  }
  return x < 2.f ? 1 : x >= (float)cap ? cap : (int)x;
}

}  // namespace chhs_dev
