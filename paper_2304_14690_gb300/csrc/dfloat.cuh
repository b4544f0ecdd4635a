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

// Two independent values per operation: the packed FP32 instructions of sm_103a, each half rounded
// as the scalar operation rounds it.
struct F2 { unsigned long long v; };
__device__ __forceinline__ F2 f2_pack(float a, float b) {
  F2 r;
  asm("mov.b64 %0, {%1, %2};" : "=l"(r.v) : "f"(a), "f"(b));
  return r;
}
__device__ __forceinline__ void f2_unpack(F2 a, float &x, float &y) { asm("mov.b64 {%0, %1}, %2;" : "=f"(x), "=f"(y) : "l"(a.v)); }
__device__ __forceinline__ F2 f2_add(F2 a, F2 b) {
  F2 r;
  asm("add.rn.f32x2 %0, %1, %2;" : "=l"(r.v) : "l"(a.v), "l"(b.v));
  return r;
}
__device__ __forceinline__ F2 f2_mul(F2 a, F2 b) {
  F2 r;
  asm("mul.rn.f32x2 %0, %1, %2;" : "=l"(r.v) : "l"(a.v), "l"(b.v));
  return r;
}
__device__ __forceinline__ F2 f2_fma(F2 a, F2 b, F2 c) {
  F2 r;
  asm("fma.rn.f32x2 %0, %1, %2, %3;" : "=l"(r.v) : "l"(a.v), "l"(b.v), "l"(c.v));
  return r;
}
// a - b as fma(b, -1, a): one rounding, the same as the subtraction's.
__device__ __forceinline__ F2 f2_sub(F2 a, F2 b) { return f2_fma(b, f2_pack(-1.0f, -1.0f), a); }
struct DF2 { F2 hi, lo; };
__device__ __forceinline__ DF2 df2_of(DF a, DF b) { return DF2{f2_pack(a.hi, b.hi), f2_pack(a.lo, b.lo)}; }
// df_sum, df_sub and second_difference on two points at a time, operation by operation.
__device__ __forceinline__ DF2 df2_sum(DF2 a, DF2 b) {
  const F2 s = f2_add(a.hi, b.hi), z = f2_sub(s, a.hi);
  const F2 e = f2_add(f2_sub(a.hi, f2_sub(s, z)), f2_sub(b.hi, z));
  return DF2{s, f2_add(e, f2_add(a.lo, b.lo))};
}
__device__ __forceinline__ DF2 df2_diff(DF2 a, DF2 b) {   // with -b in place of b: a + (-b) = a - b
  const F2 s = f2_sub(a.hi, b.hi), z = f2_sub(s, a.hi);
  const F2 e = f2_sub(f2_sub(a.hi, f2_sub(s, z)), f2_add(b.hi, z));
  return DF2{s, f2_add(e, f2_sub(a.lo, b.lo))};
}
__device__ __forceinline__ DF2 df2_norm(DF2 v) {
  const F2 h = f2_add(v.hi, v.lo);
  return DF2{h, f2_sub(v.lo, f2_sub(h, v.hi))};
}
__device__ __forceinline__ DF2 second_difference2(DF2 pl, DF2 pc, DF2 pr, DF ih2) {
  const DF2 t = df2_sum(df2_norm(df2_diff(pl, pc)), df2_norm(df2_diff(pr, pc)));
  const F2 hh = f2_pack(ih2.hi, ih2.hi), hl = f2_pack(ih2.lo, ih2.lo);
  const F2 p = f2_mul(t.hi, hh);
  F2 e = f2_fma(t.hi, hh, f2_mul(p, f2_pack(-1.0f, -1.0f)));
  e = f2_fma(t.hi, hl, e);
  return DF2{p, f2_fma(t.lo, hh, e)};
}

__device__ __forceinline__ F2 f2_neg(F2 a) { return F2{a.v ^ 0x8000000080000000ULL}; }
__device__ __forceinline__ DF2 df2_neg(DF2 a) { return DF2{f2_neg(a.hi), f2_neg(a.lo)}; }
// The ghost of an edge value: itself (Neumann) or its negative (Dirichlet).
__device__ __forceinline__ DF2 ghost(int kind, DF2 v) { return kind ? df2_neg(v) : v; }
// (last of a, first of b): the pair between two neighbouring pairs.
__device__ __forceinline__ F2 f2_mid(F2 a, F2 b) { return F2{(a.v >> 32) | (b.v << 32)}; }
__device__ __forceinline__ DF2 df2_mid(DF2 a, DF2 b) { return DF2{f2_mid(a.hi, b.hi), f2_mid(a.lo, b.lo)}; }
__device__ __forceinline__ float max_abs(float m, F2 v) {
  float x, y;
  f2_unpack(v, x, y);
  return fmaxf(m, fmaxf(fabsf(x), fabsf(y)));
}

// A stored value as a double-float pair: FP64 values are split exactly as split_f64 does, pairs
// are taken as they are.
__device__ __forceinline__ DF to_df(double v) { return df_of(v); }
__device__ __forceinline__ DF to_df(float2 v) { return DF{v.x, v.y}; }

}  // namespace pc
