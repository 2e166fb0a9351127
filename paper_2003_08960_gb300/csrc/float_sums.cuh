// Sums that FP64 would hold, in expansions of floats, on host and device: GB300
// does two FP64 operations per clock and SM, 128 FP32 ones.
#pragma once

#include <cuda_runtime.h>
#include <math.h>

namespace ssoct {

// FP32 operations rounded one by one (no contraction, no reordering).
__host__ __device__ __forceinline__ float add_rn(float a, float b) {
#ifdef __CUDA_ARCH__
  return __fadd_rn(a, b);
#else
  const volatile float s = a + b;
  return s;
#endif
}
__host__ __device__ __forceinline__ float mul_rn(float a, float b) {
#ifdef __CUDA_ARCH__
  return __fmul_rn(a, b);
#else
  const volatile float s = a * b;
  return s;
#endif
}

// s + err = a + b exactly (Knuth 1969).
__host__ __device__ __forceinline__ float two_sum(float a, float b, float& err) {
  const float s = add_rn(a, b);
  const float bb = add_rn(s, -a);
  err = add_rn(add_rn(a, -add_rn(s, -bb)), add_rn(b, -bb));
  return s;
}

// Running sum h + l + m of non-negative floats.  Four at a time: their own sum is
// s + e, whose error terms are rounded together (2^-49 of the four); every rounding
// error of h then goes to l and every rounding error of l to m, so that small terms
// after a large one lose nothing (a pair of floats keeps 2^-45 of the large one
// there).  The error terms kept apart as well would leave 2^-53 of the sum, as FP64
// does, for 57 us at 512 x 512 x 128 where this takes 42.
struct FloatSum {
  float h, l, m;
  __host__ __device__ __forceinline__ void add(float s, float e) {
    float a, b;
    h = two_sum(h, s, a);
    l = two_sum(l, e, b);
    m = add_rn(m, b);
    l = two_sum(l, a, b);
    m = add_rn(m, b);
  }
  __host__ __device__ __forceinline__ void add4(float v0, float v1, float v2, float v3, float rest) {
    float a, b, c;
    const float p = two_sum(v0, v1, a), q = two_sum(v2, v3, b);
    const float s = two_sum(p, q, c);
    add(s, add_rn(add_rn(add_rn(a, b), c), rest));
  }
  __host__ __device__ __forceinline__ void add(const FloatSum& o) {
    add(o.h, o.l);
    m = add_rn(m, o.m);
  }
  __host__ __device__ __forceinline__ double value() const { return (double)h + ((double)l + (double)m); }
};

// Sum of values and sum of their squares, a square as its rounded value and the
// exact remainder.
struct FloatSums {
  FloatSum p, q;
  __host__ __device__ __forceinline__ void add4(float v0, float v1, float v2, float v3) {
    p.add4(v0, v1, v2, v3, 0.f);
    const float q0 = mul_rn(v0, v0), q1 = mul_rn(v1, v1), q2 = mul_rn(v2, v2), q3 = mul_rn(v3, v3);
    const float r01 = add_rn(fmaf(v0, v0, -q0), fmaf(v1, v1, -q1)), r23 = add_rn(fmaf(v2, v2, -q2), fmaf(v3, v3, -q3));
    q.add4(q0, q1, q2, q3, add_rn(r01, r23));
  }
};

}  // namespace ssoct
