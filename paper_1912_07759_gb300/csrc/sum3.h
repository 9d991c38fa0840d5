// sum3.h -- sums of FP32 terms to FP64 accuracy without FP64 additions: GB300 completes one of a
// warp's per 19 cycles of an SM, and a dependent one takes about 140.
#pragma once
#include <cfloat>
#include <cmath>

#ifdef __CUDACC__
#define TR_SUM_FN __device__ __forceinline__
#else
#define TR_SUM_FN inline
#endif

namespace tr {

// Two FP32 values that are added side by side (one instruction; the halves round as scalars do).
struct Two {
  float x, y;
};
#ifdef __CUDACC__
#define TR_TWO_OP(name, op)                                                                     \
  TR_SUM_FN Two name(Two a, Two b) {                                                            \
    Two r;                                                                                      \
    asm("{\n\t.reg .b64 a, b;\n\tmov.b64 a, {%2, %3};\n\tmov.b64 b, {%4, %5};\n\t" op          \
        " a, a, b;\n\tmov.b64 {%0, %1}, a;\n\t}"                                               \
        : "=f"(r.x), "=f"(r.y) : "f"(a.x), "f"(a.y), "f"(b.x), "f"(b.y));                       \
    return r;                                                                                   \
  }
TR_TWO_OP(add_two, "add.rn.f32x2")
TR_TWO_OP(sub_two, "sub.rn.f32x2")
#undef TR_TWO_OP
#else
inline Two add_two(Two a, Two b) { return {a.x + b.x, a.y + b.y}; }
inline Two sub_two(Two a, Two b) { return {a.x - b.x, a.y - b.y}; }
#endif

// The rounded sums a + b and, in e, what the rounding left out, exactly (Knuth's TwoSum).
TR_SUM_FN Two two_sum_rn(Two a, Two b, Two& e) {
  const Two s = add_two(a, b), bb = sub_two(s, a);
  e = add_two(sub_two(a, sub_two(s, bb)), sub_two(b, bb));
  return s;
}

// A sum as three FP32 parts (two of them side by side): the remainder of every addition to the
// first part goes to the second, that one's to the third exactly, and only the third is rounded.
struct Sum3 {
  Two hi = {0.f, 0.f}, mid = {0.f, 0.f}, lo = {0.f, 0.f};
  TR_SUM_FN void add(Two t) {
    Two e;
    hi = two_sum_rn(hi, t, e);
    mid = two_sum_rn(mid, e, e);
    lo = add_two(lo, e);
  }
};

// The sum of the FP32 terms that `terms` passes to its argument, two at a time; it may be called
// twice.  n terms are off by less than n^2 2^-72 of the largest partial sum, and the result by that
// and its rounding to FP64 (with FP64 additions: n 2^-53; with two parts: n 2^-48).  Terms or partial
// sums beyond FP32's range: added again in FP64.
template <class Terms>
TR_SUM_FN double sum_fp32_terms(const Terms& terms) {
  Sum3 s;
  terms([&](float t, float u) { s.add({t, u}); });
  s.add({s.hi.y, 0.f});                             // the second sum into the first
  s.add({s.mid.y, 0.f});
  s.add({s.lo.y, 0.f});
  if (fabsf(s.hi.x) <= FLT_MAX && fabsf(s.mid.x) <= FLT_MAX)
    return (double)s.hi.x + ((double)s.mid.x + (double)s.lo.x);
  double d = 0.0;
  terms([&](float t, float u) { d += (double)t; d += (double)u; });
  return d;
}

}  // namespace tr
