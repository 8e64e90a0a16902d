// Double-float arithmetic on the FP32 units, for the near terms of the double-layer sums.
// A value is the unevaluated sum hi + lo of two floats (about 48 significant bits), built
// from Knuth's TwoSum, the FMA form of Dekker's TwoProduct and the sums and products of
// Dekker (1971).  The narrow FP64 pipe would need ~12 operations per (point, node) term.
// Coordinates are in grid units: a grid point is an exact integer pair, a node or an
// off-grid point an integer cell index plus a double-float fraction, so every
// coordinate difference is an integer minus a fraction, accurate to ~2^-48 of a cell.
// With d' = d/h, r2' = r2/h^2 the term (a dx - b dy)/r2 = (a dx' - b dy')/(h r2').
#pragma once
#include <cuda_runtime.h>

namespace fc2d {

struct dfl {
  float hi, lo;
};
__device__ __forceinline__ dfl two_sum(float a, float b) {
  const float s = a + b, bb = s - a;
  return {s, (a - (s - bb)) + (b - bb)};
}
__device__ __forceinline__ dfl fast_two_sum(float a, float b) {  // |a| >= |b|
  const float s = a + b;
  return {s, b - (s - a)};
}
__device__ __forceinline__ dfl df_add(dfl x, dfl y) {
  dfl s = two_sum(x.hi, y.hi);
  const dfl t = two_sum(x.lo, y.lo);
  s = fast_two_sum(s.hi, s.lo + t.hi);
  return fast_two_sum(s.hi, s.lo + t.lo);
}
__device__ __forceinline__ dfl df_mul(dfl x, dfl y) {
  const float p = __fmul_rn(x.hi, y.hi);  // never fused into the sum below
  float e = fmaf(x.hi, y.hi, -p);
  e = fmaf(x.hi, y.lo, e);
  e = fmaf(x.lo, y.hi, e);
  return fast_two_sum(p, e);
}
// integer n minus the fraction (fh, fl)
__device__ __forceinline__ dfl int_minus(float n, float fh, float fl) {
  const dfl s = two_sum(n, -fh);
  return fast_two_sum(s.hi, s.lo - fl);
}
// (a dx - b dy) / (dx^2 + dy^2) with a = (ah, al), b = (bh, bl)
__device__ __forceinline__ dfl dl_term(dfl dx, dfl dy, float ah, float al, float bh, float bl) {
  const dfl xx = df_mul(dx, dx), yy = df_mul(dy, dy);
  const dfl r2 = df_add(xx, yy);
  const dfl num = df_add(df_mul({ah, al}, dx), df_mul({-bh, -bl}, dy));
  // 1/r2: the correctly rounded float reciprocal and one Newton step (relative error
  // about the square of the seed's, 2^-46)
  const float y0 = __frcp_rn(r2.hi);
  float t = fmaf(-r2.hi, y0, 1.0f);
  t = fmaf(-r2.lo, y0, t);
  return df_mul(num, fast_two_sum(y0, y0 * t));
}
__device__ __forceinline__ void split_df(double v, float& hi, float& lo) {
  hi = (float)v;
  lo = (float)(v - (double)hi);
}

}  // namespace fc2d
