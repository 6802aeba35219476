// Double-float arithmetic of the FP32 inner solves.  Device code, and plain C++ so
// that its rounding can be tested on the host.
#pragma once

#ifdef __CUDACC__
#include <cuda_runtime.h>
#define FCT_DF __device__ __forceinline__
#else
#include <cmath>
#define FCT_DF inline
struct float2 {
  float x, y;
};
inline float2 make_float2(float x, float y) { return float2{x, y}; }
inline float fmaf(float a, float b, float c) { return std::fma(a, b, c); }
inline float __fmul_rn(float a, float b) { return a * b; }
inline float __fdividef(float a, float b) { return a / b; }
#endif

// ---------------------------------------------------------------------------
// Sums of squares of FP32 vectors at FP64 accuracy on the FP32 pipe
// (double-float arithmetic): the square of a float is exact as a pair
// hi + lo (hi = v v rounded, lo = fma(v, v, -hi)), and pairs are added with
// Knuth's two-sum, so a warp's sum carries about 48 significant bits.  GB300
// runs FP64 at a small fraction of its FP32 rate, so the FP32 inner solves
// form their inner products this way, sums across warps and units and the
// scalars alpha and beta included (an FP64 quotient by one thread between two
// team barriers took about 0.8 us: D = 6 degree 10 mixed 1.00 -> 0.89 ms with the
// plan's header in shared memory).  alpha and beta are rounded to FP32 as they
// were with FP64 scalars; measured, the coefficients of 49 plans of the two-matrix
// and W forms (three targets each) keep their bits.
// ---------------------------------------------------------------------------
FCT_DF float2 df_two_sum(float a, float b) {
  const float s = a + b;
  const float bb = s - a;
  return make_float2(s, (a - (s - bb)) + (b - bb));
}
FCT_DF float2 df_add(float2 x, float2 y) {
  const float2 s = df_two_sum(x.x, y.x);
  const float e = s.y + (x.y + y.y);
  const float hi = s.x + e;
  return make_float2(hi, e - (hi - s.x));
}
FCT_DF float2 df_square(float t) {
  const float hi = __fmul_rn(t, t);  // not contracted into the sum that follows
  return make_float2(hi, fmaf(t, t, -hi));
}
// Products and quotients of pairs (about 44 bits), for the scalars of the FP32
// inner solves.
FCT_DF float2 df_mul(float2 a, float2 b) {
  const float p = __fmul_rn(a.x, b.x);
  const float e = fmaf(a.x, b.x, -p) + fmaf(a.x, b.y, __fmul_rn(a.y, b.x));
  const float hi = p + e;
  return make_float2(hi, e - (hi - p));
}
FCT_DF float2 df_div(float2 a, float2 b) {
  const float q1 = __fdividef(a.x, b.x);
  const float2 qb = df_mul(make_float2(q1, 0.0f), b);
  const float2 r = df_add(a, make_float2(-qb.x, -qb.y));
  const float q2 = __fdividef(r.x, b.x);
  const float hi = q1 + q2;
  return make_float2(hi, q2 - (hi - q1));
}
FCT_DF float2 df_of(double v) {
  const float hi = static_cast<float>(v);
  return make_float2(hi, static_cast<float>(v - static_cast<double>(hi)));
}
// a < b of pairs in normal form (their high words first): the stopping tests of
// the inner solves, which a comparison of the high words alone would hold to 24 bits.
FCT_DF bool df_less(float2 a, float2 b) { return a.x < b.x || (a.x == b.x && a.y < b.y); }
