#pragma once
// Float-float arithmetic of the mixed-precision kernels: error-free transformations (Knuth's two-sum
// and the FMA product error) and the sums and products built on them.  A float-float value is the
// unevaluated sum hi + lo with |lo| <= ulp(hi) / 2, about 48 significant bits.

namespace sl {

struct ff {
  float hi, lo;
};
__device__ __forceinline__ ff two_sum(float a, float b) {
  const float s = __fadd_rn(a, b);
  const float bb = __fsub_rn(s, a);
  const float e = __fadd_rn(__fsub_rn(a, __fsub_rn(s, bb)), __fsub_rn(b, bb));
  return {s, e};
}
__device__ __forceinline__ ff fast_two_sum(float a, float b) {   // |a| >= |b| or a = 0
  const float s = __fadd_rn(a, b);
  return {s, __fsub_rn(b, __fsub_rn(s, a))};
}
__device__ __forceinline__ ff two_prod(float a, float b) {
  const float p = __fmul_rn(a, b);
  return {p, fmaf(a, b, -p)};
}
// sum of two float-float values; symmetric in its arguments bit for bit (the two-sum error term is
// exact whatever the order), so a butterfly leaves the same value in every lane
__device__ __forceinline__ ff ff_add(ff a, ff b) {
  const ff s = two_sum(a.hi, b.hi);
  return fast_two_sum(s.hi, __fadd_rn(__fadd_rn(a.lo, b.lo), s.lo));
}
__device__ __forceinline__ ff ff_neg(ff a) { return {-a.hi, -a.lo}; }
// product with a float-float weight, to about 2^-44 relative
__device__ __forceinline__ ff ff_mul(ff a, ff w) {
  const ff p = two_prod(a.hi, w.hi);
  return fast_two_sum(p.hi, fmaf(a.hi, w.lo, fmaf(a.lo, w.hi, p.lo)));
}
__device__ __forceinline__ float ff_to_f(ff a) { return __fadd_rn(a.hi, a.lo); }

// Compensated dot product sum_i (wh_i + wl_i)(hi_i + lo_i) (float-float weights and values): the
// products' high parts are added with their exact rounding errors (two-sum), everything of lower
// order goes into one float compensation.  About 2^-46 relative for sums whose terms do not cancel.
struct cdot {
  float s = 0.0f, c = 0.0f;
  __device__ __forceinline__ void add(float wh, float wl, float hi, float lo) {
    const float p = __fmul_rn(wh, hi);
    const float pe = fmaf(wh, hi, -p);
    const ff t = two_sum(s, p);
    s = t.hi;
    c = __fadd_rn(c, __fadd_rn(__fadd_rn(t.lo, pe), fmaf(wh, lo, __fmul_rn(wl, hi))));
  }
  __device__ __forceinline__ ff get() const { return fast_two_sum(s, c); }
};

// ------------------------------------------------------------------ two values at once
// The same operations on one value per lane of the paired FP32 instructions, rounded like the scalar forms
// (a - b is formed as fma(b, -1, a), the same single rounding).
struct ff2 {
  float2 hi, lo;
};
__device__ __forceinline__ float2 dup(float a) { return make_float2(a, a); }
// a stored value that is the same in both lanes
struct fdup {
  float v;
  __device__ __forceinline__ operator float2() const { return make_float2(v, v); }
};
__device__ __forceinline__ float2 neg2(float2 a) { return make_float2(-a.x, -a.y); }
__device__ __forceinline__ float2 sub2(float2 a, float2 b) { return __ffma2_rn(b, dup(-1.0f), a); }
__device__ __forceinline__ ff2 two_sum2(float2 a, float2 b) {
  const float2 s = __fadd2_rn(a, b), bb = sub2(s, a);
  return {s, __fadd2_rn(sub2(a, sub2(s, bb)), sub2(b, bb))};
}
__device__ __forceinline__ ff2 fast_two_sum2(float2 a, float2 b) {
  const float2 s = __fadd2_rn(a, b);
  return {s, sub2(b, sub2(s, a))};
}
__device__ __forceinline__ ff2 ff_add2(ff2 a, ff2 b) {
  const ff2 s = two_sum2(a.hi, b.hi);
  return fast_two_sum2(s.hi, __fadd2_rn(__fadd2_rn(a.lo, b.lo), s.lo));
}
__device__ __forceinline__ ff2 ff_mul2(ff2 a, float2 wh, float2 wl) {
  const float2 p = __fmul2_rn(a.hi, wh);
  const float2 e = __ffma2_rn(a.hi, wh, neg2(p));
  return fast_two_sum2(p, __ffma2_rn(a.hi, wl, __ffma2_rn(a.lo, wh, e)));
}
// Minus the compensated dot product of cdot, one per lane: accumulating -w v keeps every step one paired
// instruction (a negated operand would cost two integer instructions per term)
struct cdot2n {
  float2 s = {0.0f, 0.0f}, c = {0.0f, 0.0f};
  // nwh = -wh
  __device__ __forceinline__ void add(float2 wh, float2 nwh, float2 wl, float2 hi, float2 lo) {
    const float2 np = __fmul2_rn(nwh, hi);                        // -fl(wh hi)
    float2 e = __ffma2_rn(wh, hi, np);                            // wh hi - fl(wh hi), exact
    e = __ffma2_rn(wl, hi, __ffma2_rn(wh, lo, e));
    const ff2 t = two_sum2(s, np);
    s = t.hi;
    c = sub2(__fadd2_rn(c, t.lo), e);
  }
  __device__ __forceinline__ ff2 get() const { return fast_two_sum2(s, c); }
};

}  // namespace sl
