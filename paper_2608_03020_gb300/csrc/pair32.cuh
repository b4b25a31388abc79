// Numbers as pairs of fp32: x the value, y the rest that x leaves (|y| <= 2^-24 |x| when normalised),
// together 2^-48.  For the few serial or fp64-bound steps of the solves: the fp64 pipe takes 2 operations per
// clock and SM, the fp32 pipe 128.  Sums by Knuth's two-sum, products by fma (two-product).
#pragma once

#include <cuda_runtime.h>

namespace loca {

__device__ __forceinline__ float2 pair_of(double v) {
  const float h = float(v);
  return make_float2(h, isfinite(h) ? float(v - double(h)) : 0.f);
}
// a + b for pairs (value, rest), renormalised.
__device__ __forceinline__ float2 pair_add(float2 a, float2 b) {
  const float t = a.x + b.x, bb = t - a.x;
  const float e = (a.x - (t - bb)) + (b.x - bb) + (a.y + b.y);
  const float h = t + e;
  return make_float2(h, e - (h - t));
}
__device__ __forceinline__ float2 pair_norm(float2 a) {
  const float h = a.x + a.y;
  return make_float2(h, a.y - (h - a.x));
}
__device__ __forceinline__ float2 pair_mul(float2 a, float2 b) {
  const float p = a.x * b.x;
  float e = fmaf(a.x, b.x, -p);
  e = fmaf(a.x, b.y, e);
  e = fmaf(a.y, b.x, e);
  return pair_norm(make_float2(p, e));
}
// m + a b for numbers a, b and for a pair a, not renormalised.
__device__ __forceinline__ float2 pair_mac(float2 m, float a, float b) {
  const float p = a * b, e = fmaf(a, b, -p), t = m.x + p, bb = t - m.x;
  return make_float2(t, m.y + ((m.x - (t - bb)) + (p - bb) + e));
}
__device__ __forceinline__ float2 pair_mac(float2 m, float2 a, float b) {
  const float2 s = pair_mac(m, a.x, b);
  return make_float2(s.x, fmaf(a.y, b, s.y));
}
// m - a b, not renormalised.
__device__ __forceinline__ float2 pair_nmac(float2 m, float2 a, float2 b) {
  const float p = a.x * b.x;
  float e = fmaf(a.x, b.x, -p);
  e = fmaf(a.x, b.y, e);
  e = fmaf(a.y, b.x, e);
  const float t = m.x - p, bb = t - m.x;
  return make_float2(t, m.y + ((m.x - (t - bb)) - (p + bb) - e));
}
// 1 / a and 1 / sqrt(a), a > 0: the fp32 value and one step of the binomial series in what it leaves.
__device__ __forceinline__ float2 pair_rcp(float2 a) {
  const float y = __frcp_rn(a.x);
  const float r = fmaf(-a.y, y, fmaf(-a.x, y, 1.f));
  return pair_norm(make_float2(y, y * fmaf(r, r, r)));
}
__device__ __forceinline__ float2 pair_rsqrt(float2 a) {
  const float y = rsqrtf(a.x), q = y * y, qe = fmaf(y, y, -q);
  float r = fmaf(-a.x, q, 1.f);
  r = fmaf(-a.x, qe, r);
  r = fmaf(-a.y, q, r);
  return pair_norm(make_float2(y, y * fmaf(0.375f * r, r, 0.5f * r)));
}

}  // namespace loca
