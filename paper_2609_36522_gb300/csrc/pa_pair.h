// Pairs: an unevaluated sum h + l of two fp32 values, |l| <= ulp(h) / 2, about 48
// bits. Error-free sums and products (Knuth, Dekker: TwoSum, FastTwoSum, and
// TwoProd by fused multiply-add); a product is within a few 2^-48 of the exact
// one. Where a value is not finite the error terms are not either, and the plain
// fp32 result stands alone.
// Compiles for the device and, in plain C++ without contraction, for the host.
#pragma once

#include <math.h>

#ifdef __CUDACC__
#define PA_HD __host__ __device__ __forceinline__
#else
#define PA_HD inline
#endif

namespace pa {

struct Pair {
  float h, l;
};

// one rounding each: nothing here may be contracted into a multiply-add
#ifdef __CUDA_ARCH__
PA_HD float rn_add(float a, float b) { return __fadd_rn(a, b); }
PA_HD float rn_sub(float a, float b) { return __fsub_rn(a, b); }
PA_HD float rn_mul(float a, float b) { return __fmul_rn(a, b); }
#else
PA_HD float rn_add(float a, float b) { return a + b; }
PA_HD float rn_sub(float a, float b) { return a - b; }
PA_HD float rn_mul(float a, float b) { return a * b; }
#endif

PA_HD Pair pair_quick(float a, float b) {  // |a| >= |b|
  const float s = rn_add(a, b);
  return {s, rn_sub(b, rn_sub(s, a))};
}
PA_HD Pair pair_sum(float a, float b) {
  const float s = rn_add(a, b), bb = rn_sub(s, a);
  return {s, rn_add(rn_sub(a, rn_sub(s, bb)), rn_sub(b, bb))};
}
// Within a few 2^-48 of |a| + |b|: for operands of one sign, and where the result
// is added to something of the operands' size.
PA_HD Pair pair_add(Pair a, Pair b) {
  const Pair s = pair_sum(a.h, b.h);
  return pair_quick(s.h, rn_add(s.l, rn_add(a.l, b.l)));
}
PA_HD Pair pair_sub(Pair a, Pair b) { return pair_add(a, Pair{-b.h, -b.l}); }
// Within a few 2^-48 of the result, also where the operands cancel.
PA_HD Pair pair_sub_full(Pair a, Pair b) {
  const Pair s = pair_sum(a.h, -b.h), t = pair_sum(a.l, -b.l);
  const Pair v = pair_quick(s.h, rn_add(s.l, t.h));
  return pair_quick(v.h, rn_add(t.l, v.l));
}
PA_HD Pair pair_mul(Pair a, float b) {
  const float p = rn_mul(a.h, b);
  return {p, fmaf(a.l, b, fmaf(a.h, b, -p))};
}
PA_HD Pair pair_mul(Pair a, Pair b) {
  const float p = rn_mul(a.h, b.h);
  return {p, fmaf(a.l, b.h, fmaf(a.h, b.l, fmaf(a.h, b.h, -p)))};
}
PA_HD bool finite(float v) { return fabsf(v) <= 3.402823466e38f; }
PA_HD Pair pair_or(Pair a, float plain) {  // the pair, or the fp32 value where it is not finite
  return finite(rn_add(a.h, a.l)) ? a : Pair{plain, 0.f};
}
PA_HD double pair_value(Pair a) { return (double)a.h + (double)a.l; }

}  // namespace pa
