// Numbers kept as three floats, about 72 bits: sums and scalars for which double-float
// (48 bits) is too little and FP64, of which an SM retires two lanes a cycle, too slow.
// FP32 operations rounded one by one: host code is compiled without contraction.
#pragma once
#include <math.h>
#ifdef __CUDACC__
#define TF_HD __host__ __device__ __forceinline__
#else
#define TF_HD inline
#endif

struct tfl {
  float s, e, f;
};
struct tf_pair {
  float h, l;
};
TF_HD tf_pair tf_two_sum(float a, float b) {
  const float s = a + b, bb = s - a;
  return {s, (a - (s - bb)) + (b - bb)};
}
TF_HD tf_pair tf_fast_two_sum(float a, float b) {   // |a| >= |b|
  const float s = a + b;
  return {s, b - (s - a)};
}
TF_HD tf_pair tf_two_prod(float a, float b) {
  const float p = a * b;
  return {p, fmaf(a, b, -p)};
}
// a += h + l, to 2^-72 of the larger
TF_HD void tf_add(tfl& a, float h, float l) {
  const tf_pair t = tf_two_sum(a.s, h), u = tf_two_sum(a.e, l), w = tf_two_sum(u.h, t.l);
  a.s = t.h;
  a.e = w.h;
  a.f += u.l + w.l;
}
TF_HD tfl operator+(tfl a, tfl b) {   // as it comes: see tf_norm
  tf_add(a, b.s, b.e);
  a.f += b.f;
  return a;
}
// each word within half an ulp of the one before
TF_HD tfl tf_norm(tfl a) {
  const tf_pair t = tf_two_sum(a.s, a.e), u = tf_two_sum(t.l, a.f);
  return {t.h, u.h, u.l};
}
TF_HD tfl operator-(tfl a, tfl b) { return tf_norm(a + tfl{-b.s, -b.e, -b.f}); }
// the product of normalised numbers, to 2^-70 of it: the first product exactly, the two of
// the next order exactly, those of the third order in FP32
TF_HD tfl operator*(tfl a, tfl b) {
  const tf_pair p = tf_two_prod(a.s, b.s), q = tf_two_prod(a.s, b.e), r = tf_two_prod(a.e, b.s);
  const tf_pair u = tf_two_sum(q.h, r.h), v = tf_two_sum(p.l, u.h);
  const float t = fmaf(a.e, b.e, fmaf(a.s, b.f, a.f * b.s)) + ((q.l + r.l) + (u.l + v.l));
  return tf_norm({p.h, v.h, t});
}
// 1 / sqrt(a) of a normalised number, 0 for a <= 0, to 2^-67 of it: a double-float step with
// its second-order term from x0, FP32's value (2^-22 -> 2^-44), then a three-float step
TF_HD tfl tf_rsqrt_from(tfl a, float x0) {
  if (!(a.s > 0.f)) return {0.f, 0.f, 0.f};
  const tf_pair x2 = tf_two_prod(x0, x0), p = tf_two_prod(a.s, x2.h);
  const float d = (1.f - p.h) - fmaf(a.e, x2.h, fmaf(a.s, x2.l, p.l));   // 1 - p.h is exact
  const tf_pair x1 = tf_fast_two_sum(x0, x0 * fmaf(0.375f * d, d, 0.5f * d));
  const tfl x = {x1.h, x1.l, 0.f};
  const tfl y = a * (x * x);
  const float e = ((1.f - y.s) - y.e) - y.f;
  return tf_norm({x1.h, x1.l, x1.h * (0.5f * e)});
}
TF_HD double tf_to_double(tfl a) { return (double)a.s + ((double)a.e + (double)a.f); }
