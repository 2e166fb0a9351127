// exp(i pi t) for the pupil table, on host and device.
#pragma once

#include "float_sums.cuh"

namespace ssoct {

// exp(i pi t) (-1)^odd from t = m / 128 + d / pi: the tabulated exponential at m mod
// 256 (cis, pairs of floats) turned by d, |d| <= pi / 256, by the series of sine and
// cosine.  The remainder is reduced in float64 and held as a pair of floats, and
// every product and sum that the last bit of the result depends on is kept with its
// rounding error: one rounding to float32 at the end, plus 2^-35 (from the terms of
// cos d - 1), where single precision throughout left 2^-30.
__host__ __device__ __forceinline__ float2 cis_turn(double t, int odd, const float4* cis) {
  const double m = rint(t * 128.0);
  const double d = (t - m * (1.0 / 128.0)) * 3.14159265358979323846;  // the difference is exact
  // m mod 256 selects the table entry (period 2); the half turn is 128 entries
  const float4 w = cis[((int)(long long)m + 128 * odd) & 255];
  const float dh = (float)d, dl = (float)(d - (double)dh);
  const float d2 = mul_rn(dh, dh);
  const float sl = fmaf(mul_rn(d2, dh), -1.f / 6.f, dl);         // sin d = dh + sl
  const float c1 = mul_rn(d2, fmaf(d2, 1.f / 24.f, -0.5f));      // cos d = 1 + c1
  // re = w.x - w.z sin d + ..., im = w.z + w.x sin d + ...
  const float p = mul_rn(w.z, dh), q = mul_rn(w.x, dh);
  float ep, eq;
  const float re = two_sum(w.x, -p, ep), im = two_sum(w.z, q, eq);
  const float lp = fmaf(w.z, sl, fmaf(w.w, dh, fmaf(w.z, dh, -p)));  // the rest of w.z sin d
  const float lq = fmaf(w.x, sl, fmaf(w.y, dh, fmaf(w.x, dh, -q)));
  return make_float2(add_rn(re, add_rn(fmaf(w.x, c1, -lp), add_rn(ep, w.y))),
                     add_rn(im, add_rn(fmaf(w.z, c1, lq), add_rn(eq, w.w))));
}

}  // namespace ssoct
