// fl32((a r) c) for a float a and doubles r, c from float pairs, bit for bit what the FP64
// products give, and without their pipe.  Also plain C++, to be checked on any machine.
#pragma once

#include <cmath>

#include "rules.h"

namespace mpax {

// (A product that must not be contracted into a fused multiply-add with the sums below.)
MPAX_RULE float mul_rn(float a, float b) {
#ifdef __CUDA_ARCH__
  return __fmul_rn(a, b);
#else
  return a * b;
#endif
}

// d = hi + lo to 48 bits.  Below 2^-100 lo would lose bits to the end of the float range: such
// a factor has hi = lo = 0, which sends its products to FP64.
template <class Pair>
MPAX_RULE Pair float_pair(double d) {
  Pair p;
  p.x = (float)d;
  p.y = 0.0f;
  if (fabsf(p.x) < 7.8886091e-31f) p.x = 0.0f;  // 2^-100
  else if (fabsf(p.x) <= 3.4028235e38f) p.y = (float)(d - (double)p.x);
  return p;
}

// r and c as pairs and, for the cases that they leave open, at dr and dc: error-free FP32
// products give a r c to within 2^-44.  Where that margin leaves the rounding to a float open
// (about one value in 10^6), or a product leaves the range in which the pairs are exact, the
// value is formed in FP64.
template <class Pair>
MPAX_RULE float scale_pair(float a, Pair r, Pair c, const double* dr, const double* dc) {
  const float p = mul_rn(a, r.x);
  const float pl = fmaf(a, r.y, fmaf(a, r.x, -p));
  const float q = mul_rn(p, c.x);
  const float ql = fmaf(p, c.y, fmaf(pl, c.x, fmaf(p, c.x, -q)));
  const float ap = fabsf(p), aq = fabsf(q);
  const float d = mul_rn(aq, 1.1368684e-13f);  // 2^-43
  const float up = q + (ql + d), dn = q + (ql - d);
  // (false for NaN, infinities, zeros and values near the ends of the range)
  if (up == dn && ap > 1e-22f && ap < 1e30f && aq > 1e-22f && aq < 1e30f) return up;
  if (a == 0.0f) return a;
  return (float)(((double)a * *dr) * *dc);
}

}  // namespace mpax
