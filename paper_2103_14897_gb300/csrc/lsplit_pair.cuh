// Pairs of floats (an unevaluated sum of a high and a low part, about 2^-46
// relative): the FP32 pipe of sm_103a runs at 64 times the FP64 rate, so a
// pair operation of ten to twenty FP32 operations is the cheaper way to that
// accuracy.  Knuth's two-sum, Dekker's quick-two-sum, and products split by a
// fused multiply-add.  Explicit round-to-nearest intrinsics: nothing may be
// contracted.
#pragma once
namespace lsk {
struct DF { float h, l; };
__device__ __forceinline__ void two_sum(float a, float b, float& s, float& e) {
  s = __fadd_rn(a, b);
  const float bb = __fsub_rn(s, a);
  e = __fadd_rn(__fsub_rn(a, __fsub_rn(s, bb)), __fsub_rn(b, bb));
}
__device__ __forceinline__ DF quick(float h, float l) {
  const float s = __fadd_rn(h, l);
  return DF{s, __fsub_rn(l, __fsub_rn(s, h))};
}
// acc += p + e, p exact up to the small e (the parts of acc unnormalised)
__device__ __forceinline__ void pair_acc(DF& acc, float p, float e) {
  float r;
  two_sum(acc.h, p, acc.h, r);
  acc.l = __fadd_rn(acc.l, __fadd_rn(r, e));
}
// acc += a b
__device__ __forceinline__ void pair_mac(DF& acc, float a, float b) {
  const float p = __fmul_rn(a, b);
  pair_acc(acc, p, fmaf(a, b, -p));
}
}  // namespace lsk
