// Double-float arithmetic: a value is the pair h + l of two FP32 numbers,
// about 48 significant bits.  FP64 issues at 1/64 of the FP32 rate on this
// GPU, so a sum that needs more than FP32 but not all of FP64 is several
// times faster as pairs.  Products keep the rounding error of their leading
// part (FMA two-product) and the cross terms; sums keep it by two-sum (Knuth).
#pragma once
#include <cuda_runtime.h>

namespace fep3m {

struct df {
  float h, l;
};

// x as a pair: h = fl32(x), l = fl32(x - h)
__host__ __device__ __forceinline__ df df_split(double x) {
  const float h = (float)x;
  return {h, (float)(x - (double)h)};
}
__device__ __forceinline__ double df_value(df a) { return (double)a.h + (double)a.l; }
// a + b exactly, as a rounded sum and its error
__device__ __forceinline__ df df_two_sum(float a, float b) {
  const float s = a + b, v = s - a;
  return {s, (a - (s - v)) + (b - v)};
}
// a + b for pairs, renormalised (h the rounding of the whole)
__device__ __forceinline__ df df_add(df a, df b) {
  const df s = df_two_sum(a.h, b.h);
  const float e = s.l + (a.l + b.l), h = s.h + e;
  return {h, e - (h - s.h)};
}
__device__ __forceinline__ df df_sqr(df a) {
  const float p = a.h * a.h;
  return {p, fmaf(a.h + a.h, a.l, fmaf(a.h, a.h, -p))};
}
__device__ __forceinline__ df df_mul(df a, df b) {
  const float p = a.h * b.h;
  return {p, fmaf(a.l, b.h, fmaf(a.h, b.l, fmaf(a.h, b.h, -p)))};
}
// s += a b, s unnormalised (h + l the running value)
__device__ __forceinline__ void df_fma(df& s, df a, df b) {
  const float p = a.h * b.h;
  const float e = fmaf(a.l, b.h, fmaf(a.h, b.l, fmaf(a.h, b.h, -p)));
  const df t = df_two_sum(s.h, p);
  s.h = t.h;
  s.l += t.l + e;
}
// s += a, s unnormalised
__device__ __forceinline__ void df_acc(df& s, df a) {
  const df t = df_two_sum(s.h, a.h);
  s.h = t.h;
  s.l += t.l + a.l;
}
// the hardware estimate of 1 / sqrt(x) (PTX rsqrt.approx, relative error
// about 2^-23; subnormals flushed to zero)
__device__ __forceinline__ float rsqrt_est(float x) {
  float y;
  asm("rsqrt.approx.ftz.f32 %0, %1;" : "=f"(y) : "f"(x));
  return y;
}
// The range in which the two functions below keep their full accuracy (their
// intermediate values stay normal FP32 numbers): x in [2^-60, 2^60), that is
// distances between 1e-9 and 1e9 elements.  Outside it (also for zero, NaN
// and infinities) a caller takes FP64.
__device__ __forceinline__ bool df_in_range(df x) {
  return ((__float_as_uint(x.h) >> 23) - 67u) < 120u;   // sign and biased exponent
}
// 1 / sqrt(x) as a pair: the estimate y with one third-order (Householder)
// step, y (1 + e/2 + 3 e^2/8), e = 1 - x y^2 formed from the exact square of
// y.  |e| < 2^-21, so the dropped term is below 2^-64 and what is left is the
// rounding of e and of the correction, about 2^-46; FINE: y after one FP32
// Newton step, whose |e| and roundings are four times smaller (the FP64 paths)
template <bool FINE>
__device__ __forceinline__ df df_rsqrt(df x) {
  float y = rsqrt_est(x.h);
  if (FINE) y = fmaf(0.5f * y, fmaf(-x.h * y, y, 1.f), y);
  const float p = y * y, pe = fmaf(y, y, -p);
  const float e = fmaf(-x.l, p, fmaf(-x.h, pe, fmaf(-x.h, p, 1.f)));
  return {y, y * (e * fmaf(0.375f, e, 0.5f))};
}
// x^(-3/2) as a pair, from the same estimate: y^3 (1 + 3 e/2 + 15 e^2/8)
template <bool FINE>
__device__ __forceinline__ df df_rsqrt3(df x) {
  float y = rsqrt_est(x.h);
  if (FINE) y = fmaf(0.5f * y, fmaf(-x.h * y, y, 1.f), y);
  const float p = y * y, pe = fmaf(y, y, -p);
  const float e = fmaf(-x.l, p, fmaf(-x.h, pe, fmaf(-x.h, p, 1.f)));
  const float c = p * y, cl = fmaf(pe, y, fmaf(p, y, -c));
  return {c, fmaf(c, e * fmaf(1.875f, e, 1.5f), cl)};
}

// An FP64 value exactly as three floats (24 + 24 + 5 bits), and the difference
// of two as a pair: all rounding errors above 2^-48 of the difference are
// carried, so that it is as good for nearby as for distant values.
struct tf {
  float h, m, l;
};
__host__ __device__ __forceinline__ tf tf_split(double x) {
  const float h = (float)x;
  const double r = x - (double)h;
  const float m = (float)r;
  return {h, m, (float)(r - (double)m)};
}
__device__ __forceinline__ df tf_diff(tf a, tf b) {
  const df s = df_two_sum(a.h, -b.h), u = df_two_sum(a.m, -b.m), w = df_two_sum(s.l, u.h), v = df_two_sum(s.h, w.h);
  return {v.h, v.l + (w.l + (u.l + (a.l - b.l)))};
}

// s += a b with the running value as three floats: the roundings of the low
// word are carried too, so that a sum of many terms is as good as each term
// (a df sum's low word grows with the terms and loses about n 2^-50)
__device__ __forceinline__ void df_fma(tf& s, df a, df b) {
  const float p = a.h * b.h;
  const float e = fmaf(a.l, b.h, fmaf(a.h, b.l, fmaf(a.h, b.h, -p)));
  const df t = df_two_sum(s.h, p), u = df_two_sum(t.l, e), w = df_two_sum(s.m, u.h);
  s.h = t.h;
  s.m = w.h;
  s.l += w.l + u.l;
}
// s += a: a pair, or another running value
__device__ __forceinline__ void tf_add(tf& s, df a) {
  const df t = df_two_sum(s.h, a.h), u = df_two_sum(t.l, a.l), w = df_two_sum(s.m, u.h);
  s.h = t.h;
  s.m = w.h;
  s.l += w.l + u.l;
}
__device__ __forceinline__ void tf_add(tf& s, tf a) {
  const df t = df_two_sum(s.h, a.h), u = df_two_sum(s.m, a.m), w = df_two_sum(t.l, u.h);
  s.h = t.h;
  s.m = w.h;
  s.l += a.l + (w.l + u.l);
}
__device__ __forceinline__ double df_value(tf a) { return (double)a.h + ((double)a.m + (double)a.l); }

}  // namespace fep3m
