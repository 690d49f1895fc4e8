// Sums of FP32 terms held as unevaluated sums of three floats, two sums at a time: additions that keep their
// rounding errors (Knuth's TwoSum).  FP64 additions would do, but an SM issues one warp of them in about 19
// cycles and four warps of FP32 in one.  The packed instructions take two sums with one issue slot.
#pragma once

#ifdef __CUDACC__
#define TBK_SUM __device__ __forceinline__
#else  // host tests
#define TBK_SUM inline
struct float2 {
  float x, y;
};
inline float2 make_float2(float x, float y) { return {x, y}; }
#endif

namespace tbk {

TBK_SUM float2 add2(float2 a, float2 b) {
#ifdef __CUDACC__
  return __fadd2_rn(a, b);
#else
  return {a.x + b.x, a.y + b.y};
#endif
}
// a - b, rounded once
TBK_SUM float2 sub2(float2 a, float2 b) {
#ifdef __CUDACC__
  return __ffma2_rn(b, make_float2(-1.f, -1.f), a);
#else
  return {a.x - b.x, a.y - b.y};
#endif
}
// s + e = s + a exactly.
TBK_SUM void two_sum(float2& s, float2& e, float2 a) {
  const float2 t = add2(s, a), z = sub2(t, s);
  e = add2(sub2(s, sub2(t, z)), sub2(a, z));
  s = t;
}

// Three floats, of which the second takes the rounding errors of the first and the third those of the second:
// the sum of n terms is off by about n 2^-72 of the terms' magnitudes, where an FP64 sum is off by n 2^-53 and
// one of two floats by n 2^-47.
struct Sum3 {
  float2 h, m, l;
};
TBK_SUM void sum3_add(Sum3& s, float2 a) {
  float2 e, f;
  two_sum(s.h, e, a);
  two_sum(s.m, f, e);
  s.l = add2(s.l, f);
}
TBK_SUM void sum3_add(Sum3& s, const Sum3& o) {
  float2 e, f, g;
  two_sum(s.h, e, o.h);
  two_sum(s.m, f, o.m);
  two_sum(s.m, g, e);
  s.l = add2(add2(s.l, o.l), add2(f, g));
}
TBK_SUM double sum3_value(float h, float m, float l) { return (double)h + ((double)m + (double)l); }

}  // namespace tbk
