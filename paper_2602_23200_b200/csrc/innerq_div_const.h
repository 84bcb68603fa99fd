// Division by the quantisers' level counts without a division.  Plain C++ on the host, where a test goes through it
// (tests/div_const_check.cpp), single correctly rounded intrinsics on the device.
#pragma once
#include <cmath>

#include "innerq_layout.h"

namespace iq {

// x / DEN for DEN = 1, 3, 7, 15, correctly rounded: the product with the rounded reciprocal, corrected by its
// FMA-computed (hence exact) remainder, which is exact for divisors known in advance (Brisebarre, Muller and Raina,
// "Accelerating correctly rounded floating-point division when the divisor is known in advance", 2004).  Results below
// the normal range may be one unit off: the callers round to fp16, where they are zero.
template <int DEN> IQ_HD float div_const(float x) {
  if constexpr (DEN == 1) return x;
  constexpr float r = 1.0f / (float)DEN;
#ifdef __CUDA_ARCH__
  const float q = __fmul_rn(x, r);
  const float q1 = __fmaf_rn(__fmaf_rn(-(float)DEN, q, x), r, q);
  return fabsf(q) < INFINITY ? q1 : q;      // an infinite (or NaN) quotient has no remainder
#else
  const float q = x * r;
  const float q1 = std::fmaf(std::fmaf(-(float)DEN, q, x), r, q);
  return std::fabs(q) < INFINITY ? q1 : q;
#endif
}

}  // namespace iq
