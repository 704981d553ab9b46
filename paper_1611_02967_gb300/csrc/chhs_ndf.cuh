// chhs_ndf.cuh -- the mixed form's residual for one face and one cell, in
// double-single arithmetic (the marching kernel is chhs_norm_df.cuh).  Usable
// from host code, as chhs_df64.cuh.
//
// Sums and products skip the renormalisation; where a cancellation would leave
// a large low part for a product to drop, they do not: the differences of
// neighbour cells and the cubic's inner sum are renormalised, and the cubic's
// products keep the low parts' product.  Measured against 80-bit values on the
// measured workloads' fields (noise, domains and bubbles of 128^2, 192 x 128 and
// 32^3 ... 48^3, eps/h 0.8 ... 2.4, gamma 0 ... 4, at the solved state), as a
// fraction of the error with inputs cut to 2^-46 and every operation
// renormalised: root mean square 0.39 ... 0.44, largest 0.30 ... 0.80.  (With
// inputs cut to 2^-46 and nothing renormalised 1.05 ... 1.26 and up to 1.9.)
#pragma once
#include "chhs_df64.cuh"

namespace chhs_dev {

struct NdfSingle {
  using V = df64;
  static DF_HD V from(double x) { return df_split(x); }
  static DF_HD V add(V a, V b) { return df_add_raw(a, b); }
  static DF_HD V sub(V a, V b) { return df_sub_raw(a, b); }
  static DF_HD V diff(V a, V b) { return df_sub(a, b); }
  static DF_HD V mul(V a, V b) { return df_mul_raw(a, b); }
  static DF_HD V mul_wide(V a, V b) { return df_mul_wide(a, b); }
  static DF_HD V fma(V a, V b, V c) { return df_add_raw(df_mul_raw(a, b), c); }
  static DF_HD V fma_wide(V a, V b, V c) { return df_add(df_mul_wide(a, b), c); }
  static DF_HD V half(V a) { return df64{0.5f * a.hi, 0.5f * a.lo}; }
  static DF_HD V zero() { return df64{0.f, 0.f}; }
  static DF_HD float cut(V a) { return df_to_float(a); }
  static DF_HD float base(V a) { return a.hi; }
};

// A face's fluxes from the cell below it to the one above, and the four
// fields of a cell (phi, mu, p, phi*).  A: the arithmetic, NdfSingle or the
// kernel's double-precision one.
template <class A>
struct NdfFlux {
  typename A::V v, w, d;
};
template <class A>
struct NdfCell {
  typename A::V phi, mu, p, ps;
};

template <class A>
DF_HD NdfFlux<A> ndf_face(const NdfCell<A>& lo, const NdfCell<A>& hi, typename A::V gamma) {
  NdfFlux<A> F;
  const typename A::V a = A::half(A::add(lo.ps, hi.ps)), dmu = A::diff(hi.mu, lo.mu);
  F.d = A::diff(hi.phi, lo.phi);
  F.w = A::fma(gamma, A::mul(a, dmu), A::diff(hi.p, lo.p));
  F.v = A::fma(a, F.w, dmu);
  return F;
}

// The residual's rows at a cell u from its summed fluxes, phi^m and f_mu.
template <class A>
DF_HD void ndf_residual(const NdfCell<A>& u, typename A::V sv, typename A::V sw, typename A::V sd, typename A::V pm,
                        typename A::V fmu, typename A::V sih2, typename A::V ih2, typename A::V e34ih2,
                        typename A::V& r1, typename A::V& r2, typename A::V& r3) {
  using V = typename A::V;
  r1 = A::fma(sih2, sv, A::sub(pm, u.phi));
  const V quad = A::fma_wide(u.phi, A::add(u.phi, pm), A::mul(pm, pm));
  const V cub = A::half(A::half(A::mul_wide(u.phi, quad)));
  r2 = A::sub(A::add(A::sub(fmu, u.mu), cub), A::mul(e34ih2, sd));
  r3 = A::mul(ih2, sw);
}

}  // namespace chhs_dev
