// FP32 pairs (hi + lo), for sums and products beyond FP32 without FP64
// arithmetic.
#pragma once

namespace lbmp {

// ------------------------------------------------ FP32-pair arithmetic
// Pairs of FP32 numbers (value = hi + lo) carrying ~44 significant bits:
// exact sums (Knuth's two-sum) and exact products (fma of the product and
// its negation), the standard error-free transformations.  FP64 arithmetic
// runs at ~1/64 of the FP32 rate on this GPU; the precompute and the
// per-thread parts of the reductions use these pairs instead.
struct F2 {
  float hi, lo;
};
__device__ __forceinline__ F2 two_sum(float a, float b) {
  const float s = __fadd_rn(a, b);
  const float bb = __fsub_rn(s, a);
  const float e = __fadd_rn(__fsub_rn(a, __fsub_rn(s, bb)), __fsub_rn(b, bb));
  return {s, e};
}
__device__ __forceinline__ F2 fast_two_sum(float a, float b) {  // |a| >= |b|
  const float s = __fadd_rn(a, b);
  return {s, __fsub_rn(b, __fsub_rn(s, a))};
}
__device__ __forceinline__ F2 two_prod(float a, float b) {
  const float p = __fmul_rn(a, b);
  return {p, __fmaf_rn(a, b, -p)};
}
__device__ __forceinline__ F2 f2_add(F2 x, F2 y) {
  F2 s = two_sum(x.hi, y.hi);
  return fast_two_sum(s.hi, __fadd_rn(s.lo, __fadd_rn(x.lo, y.lo)));
}
__device__ __forceinline__ F2 f2_mul(F2 x, F2 y) {
  F2 p = two_prod(x.hi, y.hi);
  const float c = __fmaf_rn(x.hi, y.lo, __fmul_rn(x.lo, y.hi));
  return fast_two_sum(p.hi, __fadd_rn(p.lo, c));
}
// n / d from an approximate reciprocal r of d.hi (relative error e ~ 2^-23):
// q1 = n.hi r is off by ~e, the remainder n - q1 d is formed exactly enough
// (~2^-48 of n), and its quotient by the same r corrects q1 to a relative
// error of order e^2 -- one Newton step on the quotient.
__device__ __forceinline__ F2 f2_div(F2 n, F2 d) {
  const float r = rcp_approx(d.hi);
  const float q1 = __fmul_rn(n.hi, r);
  const F2 qd = f2_mul({q1, 0.0f}, d);           // q1 d
  const F2 rem = f2_add(n, {-qd.hi, -qd.lo});     // n - q1 d
  return fast_two_sum(q1, __fmul_rn(rem.hi, r));
}
// acc += x (x an FP32 value)
__device__ __forceinline__ void f2_acc(F2 &acc, float x) {
  const F2 s = two_sum(acc.hi, x);
  acc = fast_two_sum(s.hi, __fadd_rn(s.lo, acc.lo));
}

}  // namespace lbmp
