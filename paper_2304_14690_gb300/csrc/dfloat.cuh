// Double-float arithmetic: unevaluated FP32 pairs (hi + lo, struct DF) with error-free
// transformations (Knuth's TwoSum, Dekker's product through fma); the _rn intrinsics keep the
// compiler from contracting them.
#pragma once

#include "numeric.cuh"

namespace pc {

__device__ __forceinline__ DF df_of(double v) {
  DF r;
  split_f64(v, r.hi, r.lo);
  return r;
}
__device__ __forceinline__ DF df_neg(DF a) { return DF{-a.hi, -a.lo}; }
__device__ __forceinline__ DF df_add(DF a, DF b) {
  const float s = __fadd_rn(a.hi, b.hi);
  const float z = __fsub_rn(s, a.hi);
  float e = __fadd_rn(__fsub_rn(a.hi, __fsub_rn(s, z)), __fsub_rn(b.hi, z));
  e = __fadd_rn(e, __fadd_rn(a.lo, b.lo));
  const float h = __fadd_rn(s, e);
  return DF{h, __fsub_rn(e, __fsub_rn(h, s))};
}
__device__ __forceinline__ DF df_sub(DF a, DF b) { return df_add(a, df_neg(b)); }
__device__ __forceinline__ DF df_mul(DF a, DF b) {
  const float p = __fmul_rn(a.hi, b.hi);
  float e = __fmaf_rn(a.hi, b.hi, -p);
  e = __fmaf_rn(a.hi, b.lo, e);
  e = __fmaf_rn(a.lo, b.hi, e);
  const float h = __fadd_rn(p, e);
  return DF{h, __fsub_rn(e, __fsub_rn(h, p))};
}

// Sum and difference without the final renormalisation: hi is the rounded sum of the high parts, lo
// its exact error plus the low parts. lo may then exceed half an ulp of hi, which costs nothing
// where the pair is only summed further.
__device__ __forceinline__ DF df_sum(DF a, DF b) {
  const float s = __fadd_rn(a.hi, b.hi);
  const float z = __fsub_rn(s, a.hi);
  const float e = __fadd_rn(__fsub_rn(a.hi, __fsub_rn(s, z)), __fsub_rn(b.hi, z));
  return DF{s, __fadd_rn(e, __fadd_rn(a.lo, b.lo))};
}
__device__ __forceinline__ DF df_diff(DF a, DF b) { return df_sum(a, df_neg(b)); }
// (t.hi + t.lo)(h.hi + h.lo) as an unnormalised pair.
__device__ __forceinline__ DF df_scale(DF t, DF h) {
  const float p = __fmul_rn(t.hi, h.hi);
  float e = __fmaf_rn(t.hi, h.hi, -p);
  e = __fmaf_rn(t.hi, h.lo, e);
  return DF{p, __fmaf_rn(t.lo, h.hi, e)};
}

// The refinement's residual r = s - mean - L_h p of one point. acc accumulates the second
// differences axis by axis: the differences to the centre first, which cancel before any rounding
// of their sum, and which are renormalised: their low parts are then half an ulp of the small
// differences and not of p, so that summing them drops nothing of note (without that the solution
// was ten times further from the FP64 one: 2.6e-14 instead of 2.6e-15 on a 192^3 box). What
// follows is only summed, and its pairs stay unnormalised until the end: 42 FP32 operations per
// axis instead of 51.
__device__ __forceinline__ DF second_difference(DF pl, DF pc, DF pr, DF ih2) {
  return df_scale(df_sum(df_sub(pl, pc), df_sub(pr, pc)), ih2);
}
__device__ __forceinline__ DF residual_of(DF s, DF acc) {
  const DF v = df_diff(s, acc);
  const float h = __fadd_rn(v.hi, v.lo);
  return DF{h, __fsub_rn(v.lo, __fsub_rn(h, v.hi))};
}

// A stored value as a double-float pair: FP64 values are split exactly as split_f64 does, pairs
// are taken as they are.
__device__ __forceinline__ DF to_df(double v) { return df_of(v); }
__device__ __forceinline__ DF to_df(float2 v) { return DF{v.x, v.y}; }

}  // namespace pc
