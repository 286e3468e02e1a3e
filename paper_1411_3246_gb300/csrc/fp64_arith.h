// FP64 reciprocals, roots and quotients for GB300's narrow FP64 pipe, shared by the marches and the
// adjoint.  Device: the hardware's approximations, refined by Newton's iteration with exact residuals
// (fused multiply-add); host: the plain operations.  Held against the IEEE operations over their ranges
// by tests/test_gpu_arith.py.
#pragma once

#include <cmath>

#if defined(__CUDACC__)
#define WAKE_HD __host__ __device__
#else
#define WAKE_HD
#endif

namespace wake {

// 1/x for x and 1/x normal (0, subnormal and infinite x give NaN): the approximation r (about 20 bits)
// and one third-order Newton step r (1 + e + e^2), e = 1 - x r.  The series leaves e^3, below 2^-60, so
// the result is 1/x rounded, or its neighbour where 1/x lies beside a midpoint: three FP64 instructions
// after the seed, where an IEEE division costs three times as many.
WAKE_HD inline double rcp64(double x) {
#ifdef __CUDA_ARCH__
  double r;
  asm("rcp.approx.ftz.f64 %0, %1;" : "=d"(r) : "d"(x));
  const double e = fma(-x, r, 1.0);
  return fma(r, fma(e, e, e), r);
#else
  return 1.0 / x;
#endif
}

// sqrt(x) and its reciprocal, x > 0 normal: the approximation y and one third-order Newton step
// y (1 + e/2 + 3 e^2 / 8), e = 1 - x y^2, which leaves the rounding of x y in it (two ulp at most); the
// root x y is corrected once, to the root rounded or its neighbour.
WAKE_HD inline void root64(double x, double &r, double &ir) {
#ifdef __CUDA_ARCH__
  double y;
  asm("rsqrt.approx.ftz.f64 %0, %1;" : "=d"(y) : "d"(x));
  const double e = fma(-(x * y), y, 1.0);
  y = fma(fma(0.375, e, 0.5), e * y, y);
  const double g = x * y;
  r = fma(fma(-g, g, x), 0.5 * y, g);
  ir = y;
#else
  r = std::sqrt(x);
  ir = 1.0 / r;
#endif
}

// a / b from b and rb = 1/b rounded: the product and one correction by its exact residual (Markstein
// 1990), three FP64 instructions where a division costs three times as many.  Rounded as the division
// rounds it, but for about one pair in 10^6, where it is the neighbour.
WAKE_HD inline double quot64(double a, double b, double rb) {
#ifdef __CUDA_ARCH__
  const double q = a * rb;
  return fma(fma(-q, b, a), rb, q);
#else
  (void)rb;
  return a / b;
#endif
}

}  // namespace wake
