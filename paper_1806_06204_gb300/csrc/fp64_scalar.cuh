// Scalar FP64 roots and reciprocals for the latency-bound factorisation kernels: the
// library's sqrt and division are long dependent sequences on this part's FP64 units.
#pragma once

namespace zolo {

// 1 / sqrt(x) and sqrt(x) for a normal x away from the ends of the range: the
// hardware's approximation r (its error e = 1 - x r^2 is below 2^-18), the cubically
// convergent step r (1 + e / 2 + 3 e^2 / 8), and one Newton correction of the root.
__device__ __forceinline__ void root_pair(double x, double* root, double* inv) {
  double r;
  asm("rsqrt.approx.ftz.f64 %0, %1;" : "=d"(r) : "d"(x));
  const double e = fma(-x * r, r, 1.0);
  r = fma(r * e, fma(e, 0.375, 0.5), r);
  const double h = x * r;
  *root = fma(fma(-h, h, x), 0.5 * r, h);
  *inv = r;
}
// 1 / x, likewise: r (1 + e + e^2) with e = 1 - x r.
__device__ __forceinline__ double reciprocal(double x) {
  double r;
  asm("rcp.approx.ftz.f64 %0, %1;" : "=d"(r) : "d"(x));
  const double e = fma(-x, r, 1.0);
  return fma(r, fma(e, e, e), r);
}

}  // namespace zolo
