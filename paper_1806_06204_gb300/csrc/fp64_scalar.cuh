// Scalar FP64 roots and reciprocals for the latency-bound factorisation kernels: the
// library's sqrt and division are long dependent sequences on this part's FP64 units, where
// every instruction of a warp takes its unit 64 clocks.
//
// Newton-Raphson iterations in FMA arithmetic (Muller et al., Handbook of Floating-Point
// Arithmetic, the chapter on division and square root with an FMA; the last correction of
// the root is Markstein's, IBM J. Res. Dev. 34, 1990), from the PTX approximations with 20
// fraction bits.  A step takes a relative error d of 1/x to d^2 and of 1/sqrt(x) to 3/2
// d^2: two of them make 2^-18 into less than 2^-70, and even 2^-14 into 2^-54.
// tests/test_gpu_fp64_scalar.py holds the results to the bounds below.
#pragma once

namespace zolo {

// inv = 1 / sqrt(x) within 1.5 2^-53 of its value (x y is rounded once in the last step,
// which halves that, and the step itself: 1 / sqrt(x) formed by CUDA's two operations is
// within 2 2^-53), root = sqrt(x) within 0.501 ulp.  For x in [1e-280, 1e280].
__device__ __forceinline__ void root_pair(double x, double* root, double* inv) {
  double y;
  asm("rsqrt.approx.ftz.f64 %0, %1;" : "=d"(y) : "d"(x));
  auto half = [](double v) { return __hiloint2double(__double2hiint(v) - (1 << 20), __double2loint(v)); };
#pragma unroll
  for (int k = 0; k < 2; ++k) y = fma(half(y), fma(-(x * y), y, 1.0), y);
  const double g = x * y;
  *root = fma(fma(-g, g, x), half(y), g);
  *inv = y;
}
// 1 / x within 0.501 ulp, for |x| in [2^-1020, 2^1020].
__device__ __forceinline__ double reciprocal(double x) {
  double r;
  asm("rcp.approx.ftz.f64 %0, %1;" : "=d"(r) : "d"(x));
#pragma unroll
  for (int k = 0; k < 2; ++k) r = fma(r, fma(-x, r, 1.0), r);
  return r;
}

}  // namespace zolo
