// FP64 parts of Algorithm 1 that the K-averaged collision kernel and its
// pathwise adjoint share.
#pragma once

#include "pic_internal.cuh"

namespace pic {

// The accept decision of one candidate in FP64, as the paper writes it
// (U < sigma(g) g / (sigma g)_max), with the near-tie and g > g_max flags.
static __device__ __noinline__ int ntc_decide64(const Params& P, uint32_t w, double dx, double dy, double dz) {
  const double g2 = __dadd_rn(__dadd_rn(__dmul_rn(dx, dx), __dmul_rn(dy, dy)), __dmul_rn(dz, dz));
  const double g = __dsqrt_rn(g2);
  const double ratio = P.n_sigma == 0 ? __ddiv_rn(__dmul_rn(P.sigma0, g), P.sg_max)
                                      : __ddiv_rn(sigma_g(P, g2), P.sg_max);
  const double U = unif32(w);
  return (U < ratio ? 1 : 0) | (fabs(U - ratio) < 1e-12 ? 2 : 0) | (g > P.gmax ? 4 : 0);
}

// R(a) of hs_R at u = a^2: polynomials of degree 7 on intervals of 1/8 up to
// kR64Max (interpolation error below 1e-17), the closed form beyond.
__device__ __forceinline__ double hs_R64(const Params& P, double u) {
  if (!(u < (double)kR64Max)) return hs_R(P, sqrt(u));
  const double t = u * (double)kR64PerUnit;
  const double r = floor_small(t);
  const double2* q = reinterpret_cast<const double2*>(P.ginv + 2 * (P.ginv_M + 1) + kQuantileDoubles) + 4 * (int)r;
  const double x = t - r - 0.5;
  const double2 q0 = __ldg(q), q1 = __ldg(q + 1), q2 = __ldg(q + 2), q3 = __ldg(q + 3);
  return fma(fma(fma(fma(fma(fma(fma(q3.y, x, q3.x), x, q2.y), x, q2.x), x, q1.y), x, q1.x), x, q0.y), x, q0.x);
}

// The same with R'(a) / a = 2 dR/du (the polynomial's derivative: as exact as
// the closed form, whose terms cancel, is at its best).
__device__ __forceinline__ void hs_R64_both(const Params& P, double u, double* R, double* Rp_over_a) {
  if (!(u < (double)kR64Max)) {
    const double a = sqrt(u), ia = 1.0 / a, ia2 = ia * ia;
    const double sq2pi = 0.79788456080286535588;
    *R = hs_R(P, a);
    *Rp_over_a = ia * (sq2pi * exp(-0.5 * u) * (ia - 3.0 * ia2 * ia) +
                       (1.0 - 2.0 * ia2 + 3.0 * ia2 * ia2) * erf(a * 0.70710678118654752440));
    return;
  }
  const double t = u * (double)kR64PerUnit;
  const double r = floor_small(t);
  const double2* q = reinterpret_cast<const double2*>(P.ginv + 2 * (P.ginv_M + 1) + kQuantileDoubles) + 4 * (int)r;
  const double x = t - r - 0.5;
  const double2 q0 = __ldg(q), q1 = __ldg(q + 1), q2 = __ldg(q + 2), q3 = __ldg(q + 3);
  double d = q3.y, v = fma(q3.y, x, q3.x);
  const double c[6] = {q2.y, q2.x, q1.y, q1.x, q0.y, q0.x};
#pragma unroll
  for (int i = 0; i < 6; ++i) {
    d = fma(d, x, v);
    v = fma(v, x, c[i]);
  }
  *R = v;
  *Rp_over_a = (2.0 * kR64PerUnit) * d;
}

}  // namespace pic
