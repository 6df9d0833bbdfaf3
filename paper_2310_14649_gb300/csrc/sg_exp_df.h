// exp of a double-FP32 argument in FP32 arithmetic, the same on host and
// device (no contraction changes its result beyond the stated bound).
#pragma once

#include <cmath>

#ifdef __CUDACC__
#define SG_HD __host__ __device__
#else
#define SG_HD
#endif

namespace sg {

// float(exp(a)) for a double-FP32 argument: a = n ln 2 + r with |r| <= 0.35,
// the Taylor series of exp(r) with its terms up to r^2 / 2 summed exactly
// enough that only the last addition rounds: at most 0.556 ulp for normal
// results (the last rounding, 0.032 from the terms from r^3 on, 0.023 from
// adding them).
SG_HD inline float exp_df(float ah, float al) {
  if (!(ah < 100.f)) return ah != ah ? ah : INFINITY;
  if (ah < -110.f) return 0.f;
  const float n = rintf(ah * 1.44269504088896341f);
  // ln 2 in two parts (Cody and Waite); n has at most 8 bits, so n * c1 is exact
  const float c1 = 0.693145751953125f;             // 16 significant bits
  const float c2 = 1.4286068e-06f;                 // ln 2 - c1
  const float rh = fmaf(-n, c1, ah);               // exact (Sterbenz range)
  const float rm = fmaf(-n, c2, al);
  // r = rh + rm as a normalised pair
  const float r = rh + rm;
  const float rl = rm - (r - rh);
  const float r2 = r * r;
  float t = 2.7557319e-06f;                        // 1/9!
  t = fmaf(t, r, 2.4801587e-05f);
  t = fmaf(t, r, 1.9841270e-04f);
  t = fmaf(t, r, 1.3888889e-03f);
  t = fmaf(t, r, 8.3333333e-03f);
  t = fmaf(t, r, 4.1666667e-02f);
  t = fmaf(t, r, 1.6666667e-01f);
  t = t * r * r2;                                  // r^3 (1/6 + ...)
  const float q = 0.5f * r2;                       // r^2 / 2 and its rounding error
  const float qe = 0.5f * fmaf(r, r, -r2);
  // s = r + q + t with the errors kept
  const float s1 = r + q;
  const float e1 = fabsf(r) >= q ? q - (s1 - r) : r - (s1 - q);
  const float low = e1 + (qe + (t + fmaf(rl, r, rl)));
  const float s = s1 + low;
  const float se = low - (s - s1);
  const float h = 1.0f + s;
  const float he = s - (h - 1.0f);
  return ldexpf(h + (he + se), int(n));
}

}  // namespace sg
