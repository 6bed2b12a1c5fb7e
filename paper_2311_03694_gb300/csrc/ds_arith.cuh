// Double-single arithmetic on the FP32 pipe: a value is an unevaluated sum of
// two floats, hi = rn32(x) and lo = rn32(x - hi) (a 48-bit significand).
// GB300 issues about two FP64 FMAs per clock per SM against 128 FP32 ones,
// so FP64-tolerance contractions run in this arithmetic.  It is built from
// the error-free transformations of floating-point arithmetic: the FMA
// residual of a product (a*b - rn(a*b) is exact) and Knuth's TwoSum (the
// rounding error of a sum, exactly, in six operations), with Fast2Sum to
// renormalise a pair.  The intrinsics carry explicit rounding so that the
// compiler cannot contract or reassociate the transformations.
#pragma once

#include <cuda_runtime.h>

namespace grom {

// (S, s) += (ah + al)(bh + bl), al*bl (below 2^-48 relative) dropped.
// p = ah*bh; Knuth's TwoSum of S and p gives S1 and the exact terms
// S - (S1 - bb) and p - bb; the second and the product's rounding error
// (ah*bh - p) are folded into one residual fma(ah, bh, -bb).  The small
// terms and the cross terms ah*bl, al*bh are summed first and reach the low
// word in one addition, so each word of the accumulator carries a chain of
// one dependent operation per call.  10 FP32 operations.  The low word
// collects one rounding per call, so callers renormalise the pair
// (ds_renorm) every few terms to keep it within an ulp of the high word.
__device__ __forceinline__ void ds_mac(float ah, float al, float bh, float bl, float& S, float& s) {
  const float p = __fmul_rn(ah, bh);
  const float S1 = __fadd_rn(S, p);
  const float bb = __fsub_rn(S1, S);
  const float y = __fsub_rn(S, __fsub_rn(S1, bb));
  const float z = __fmaf_rn(ah, bh, -bb);
  float w = __fadd_rn(y, z);
  w = __fmaf_rn(al, bh, w);
  w = __fmaf_rn(ah, bl, w);
  s = __fadd_rn(s, w);
  S = S1;
}

// Two independent FP32 values in a register pair (low word first) and the
// packed operations on them: each rounds as its scalar counterpart, in one
// issue slot for both.
struct f32pair {
  unsigned long long v;
};
__device__ __forceinline__ f32pair pair_make(float x, float y) {
  f32pair r;
  asm("mov.b64 %0, {%1, %2};" : "=l"(r.v) : "f"(x), "f"(y));
  return r;
}
__device__ __forceinline__ void pair_get(f32pair a, float& x, float& y) {
  asm("mov.b64 {%0, %1}, %2;" : "=f"(x), "=f"(y) : "l"(a.v));
}
__device__ __forceinline__ f32pair pair_add(f32pair a, f32pair b) {
  f32pair r;
  asm("add.rn.f32x2 %0, %1, %2;" : "=l"(r.v) : "l"(a.v), "l"(b.v));
  return r;
}
// The product as two scalar instructions: the assembler contracts a packed
// multiplication with the addition that uses it, .rn or not, and a fused
// first sum breaks the transformation below (5e-9 instead of 1e-14 a sum).
__device__ __forceinline__ f32pair pair_mul(f32pair a, f32pair b) {
  float a0, a1, b0, b1;
  pair_get(a, a0, a1);
  pair_get(b, b0, b1);
  return pair_make(__fmul_rn(a0, b0), __fmul_rn(a1, b1));
}
__device__ __forceinline__ f32pair pair_fma(f32pair a, f32pair b, f32pair c) {
  f32pair r;
  asm("fma.rn.f32x2 %0, %1, %2, %3;" : "=l"(r.v) : "l"(a.v), "l"(b.v), "l"(c.v));
  return r;
}
__device__ __forceinline__ f32pair pair_sub(f32pair a, f32pair b) {  // a - b
  return pair_fma(b, f32pair{0xBF800000BF800000ull}, a);
}

// ds_mac for two accumulators: the same operations and roundings (-bb formed
// as S - S1), eleven issue slots for the two.
__device__ __forceinline__ void ds_mac2(f32pair ah, f32pair al, f32pair bh, f32pair bl, f32pair& S, f32pair& s) {
  const f32pair S1 = pair_add(S, pair_mul(ah, bh));
  const f32pair nb = pair_sub(S, S1);
  const f32pair y = pair_sub(S, pair_add(S1, nb));
  f32pair w = pair_add(y, pair_fma(ah, bh, nb));
  w = pair_fma(al, bh, w);
  w = pair_fma(ah, bl, w);
  s = pair_add(s, w);
  S = S1;
}
__device__ __forceinline__ void ds_renorm2(f32pair& S, f32pair& s) {
  const f32pair h = pair_add(S, s);
  s = pair_sub(s, pair_sub(h, S));
  S = h;
}

// Fast2Sum: the pair as its rounded sum and that sum's error.
__device__ __forceinline__ void ds_renorm(float& S, float& s) {
  const float h = __fadd_rn(S, s);
  s = __fsub_rn(s, __fsub_rn(h, S));
  S = h;
}

// (S, s) += (T, t): TwoSum of the leading parts, then renormalised.
__device__ __forceinline__ void ds_add(float& S, float& s, float T, float t) {
  const float S1 = __fadd_rn(S, T);
  const float bb = __fsub_rn(S1, S);
  const float err = __fadd_rn(__fsub_rn(S, __fsub_rn(S1, bb)), __fsub_rn(T, bb));
  s = __fadd_rn(__fadd_rn(s, t), err);
  S = S1;
  ds_renorm(S, s);
}

// (h, l) = (ah + al)(bh + bl), renormalised.
__device__ __forceinline__ void ds_mul(float ah, float al, float bh, float bl, float& h, float& l) {
  const float p = __fmul_rn(ah, bh);
  const float e = __fmaf_rn(ah, bh, -p);
  const float t = __fmaf_rn(ah, bl, __fmaf_rn(al, bh, e));
  h = __fadd_rn(p, t);
  l = __fsub_rn(t, __fsub_rn(h, p));
}

// (s1, s2, s3) += v: two chained TwoSums and an addition, so the unevaluated
// sum s1 + s2 + s3 keeps about 72 bits, more than an FP64 sum of the same
// FP32 terms.  13 FP32 operations a term, where the FP64 sum takes a
// conversion and an addition on a pipe 64 times narrower.
__device__ __forceinline__ void ts_add(float v, float& s1, float& s2, float& s3) {
  const float a = __fadd_rn(s1, v), ab = __fsub_rn(a, s1);
  const float e1 = __fadd_rn(__fsub_rn(s1, __fsub_rn(a, ab)), __fsub_rn(v, ab));
  const float b = __fadd_rn(s2, e1), bb = __fsub_rn(b, s2);
  const float e2 = __fadd_rn(__fsub_rn(s2, __fsub_rn(b, bb)), __fsub_rn(e1, bb));
  s1 = a;
  s2 = b;
  s3 = __fadd_rn(s3, e2);
}

// An FP32 value as FP64 and an FP64 value rounded (to nearest even) to FP32,
// on the integer pipe: a conversion instruction takes a slot of the FP64
// pipe, as long as some thirty integer operations.  Zeros, subnormals,
// infinities and NaNs, and what rounds to them, take the instruction.
__device__ __forceinline__ double f2d_int(float x) {
  const unsigned int v = (unsigned int)__float_as_int(x), mag = v & 0x7fffffffu;
  if (mag - 0x00800000u >= 0x7f000000u) return (double)x;
  return __hiloint2double((int)((v & 0x80000000u) | ((mag >> 3) + 0x38000000u)), (int)(v << 29));
}
__device__ __forceinline__ float d2f_int(double x) {
  const unsigned int hi = (unsigned int)__double2hiint(x), lo = (unsigned int)__double2loint(x);
  if (((hi >> 20) & 0x7ffu) - 897u >= 254u) return __double2float_rn(x);
  unsigned int mag = (__funnelshift_l(lo, hi, 3) - 0x40000000u) & 0x7fffffffu;  // the 29 low bits cut off
  mag += ((lo & 0x1fffffffu) + 0x0fffffffu + (mag & 1u)) >> 29;
  return __int_as_float((int)((hi & 0x80000000u) | mag));
}

// An FP64 value as a double-single pair.
__device__ __forceinline__ void ds_split(double v, float& h, float& l) {
  h = __double2float_rn(v);
  l = __double2float_rn(v - (double)h);
}

}  // namespace grom
