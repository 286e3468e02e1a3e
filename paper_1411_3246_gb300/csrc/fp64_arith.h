// FP64 arithmetic for GB300's narrow FP64 pipe, shared by host and device code.
#pragma once

#include <cmath>

#if defined(__CUDACC__)
#define WAKE_HD __host__ __device__
#else
#define WAKE_HD
#endif

namespace wake {

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
