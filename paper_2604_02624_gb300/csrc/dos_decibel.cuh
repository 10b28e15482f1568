// dos_decibel.cuh - ten times the decimal logarithm, to FP32, in FP32 arithmetic.
#pragma once

#include "dos_fft.cuh"

namespace dos {

// 10 log10(x) rounded to FP32, within 0.03 of a unit in its last place before
// that rounding.  An FP64 logarithm is a few hundred dependent FP64
// instructions, the longest chain of a small objective launch (96 channels of
// 41 x 41: step 200.7 us with it).  Here x = (m + l) 2^e with m an FP32 number
// in [2/3, 4/3) and l what its rounding left, and
//   ln(m + l) = 2 artanh(S) = 2 (S + S^3 / 3 + S^5 / 5 + ...),
//   S = (m + l - 1) / (m + l + 1), |S| <= 1/5,
// with S as an FP32 pair s + r (r from the exact remainder of the quotient) and
// the terms from S^3 on, at most 0.0027, in FP32 up to S^11 (what follows is
// below 1e-10); the sum with e log10 2 is FP64.  (With FP32's own logarithm of m
// the result was off by up to 2.8 units, just below one.)
DOS_HD float ten_log10(double x) {
  const float f = (float)x;
  if (!(f > 1e-30f && f < 1e30f)) return (float)(10.0 * log10(x));  // also 0, infinities, NaN
  if (fabsf(f - 1.f) < 1e-3f) {  // l is not small beside m - 1: ln(1 + d), four terms
    const double d = x - 1.0;
    return (float)(4.3429448190325183 * (d * (1.0 - d * (0.5 - d * (1.0 / 3.0 - d * 0.25)))));
  }
  int e;
  float m = frexpf(f, &e);  // [0.5, 1)
  if (m < 0.66666667f) m *= 2.f, --e;
  const float l = scalbnf((float)(x - (double)f), -e);
  const float a = m - 1.f, b = m + 1.f;  // a is exact, m + 1 = b + be
  const float be = m - (b - 1.f);
  const float inv = 1.f / b;
  const float s = a * inv;
  const float r = (fmaf(-s, b, a) + fmaf(-s, be + l, l)) * inv;
  const float u = s * s;
  float q = fmaf(u, 0.090909091f, 0.11111111f);
  q = fmaf(u, q, 0.14285714f);
  q = fmaf(u, q, 0.2f);
  q = fmaf(u, q, 0.33333333f);
  const float t = fmaf(s * u, q, fmaf(r, u, r));  // artanh(s + r): its slope there is 1 + u + ...
  // 10 log10 2 and 20 / ln 10
  return (float)fma((double)e, 3.0102999566398120, 8.6858896380650366 * ((double)s + (double)t));
}

}  // namespace dos
