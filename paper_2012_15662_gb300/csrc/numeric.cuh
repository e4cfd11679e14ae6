// Small pieces of device arithmetic that stand alone: packed FP32 pairs and double-float sums on
// them, and the FP64 quotient from a reciprocal (tests/unit_numeric.cu runs them one by one).
#pragma once

namespace donof {

// Two FP32 values in one 64-bit register and the packed operations on them (each half
// rounded as the scalar operation): the epilogues work on two columns per instruction,
// since they are bound by the instructions they issue.
typedef unsigned long long f32x2;
__device__ __forceinline__ f32x2 pack2(float a, float b) {
  f32x2 r;
  asm("mov.b64 %0, {%1, %2};" : "=l"(r) : "f"(a), "f"(b));
  return r;
}
__device__ __forceinline__ void unpack2(f32x2 v, float& a, float& b) { asm("mov.b64 {%0, %1}, %2;" : "=f"(a), "=f"(b) : "l"(v)); }
__device__ __forceinline__ f32x2 both2(float a) { return pack2(a, a); }
__device__ __forceinline__ f32x2 add2(f32x2 a, f32x2 b) {
  f32x2 r;
  asm("add.rn.f32x2 %0, %1, %2;" : "=l"(r) : "l"(a), "l"(b));
  return r;
}
__device__ __forceinline__ f32x2 mul2(f32x2 a, f32x2 b) {
  f32x2 r;
  asm("mul.rn.f32x2 %0, %1, %2;" : "=l"(r) : "l"(a), "l"(b));
  return r;
}
__device__ __forceinline__ f32x2 fma2(f32x2 a, f32x2 b, f32x2 c) {
  f32x2 r;
  asm("fma.rn.f32x2 %0, %1, %2, %3;" : "=l"(r) : "l"(a), "l"(b), "l"(c));
  return r;
}
__device__ __forceinline__ f32x2 sub2(f32x2 a, f32x2 b) { return fma2(b, both2(-1.f), a); }

// s + e = a + b exactly (TwoSum).
__device__ __forceinline__ void two_sum2(f32x2 a, f32x2 b, f32x2& s, f32x2& e) {
  s = add2(a, b);
  const f32x2 bb = sub2(s, a);
  e = add2(sub2(a, sub2(s, bb)), sub2(b, bb));
}

// (sh, sl) += (ph, pl) in double-float arithmetic, renormalised after every term: the packed
// form of df_add, the same bits.  (Gathering the low parts in one word without renormalising
// saves three of the thirteen operations and lets that word grow with the number of terms, which
// no rule bounds (158 at C20H40): rms error 3.1e-14 instead of 8e-15 of a sum of 158 squares,
// 7.7e-14 instead of 1.3e-14 at 400.  No case of an iteration is faster for it.)
__device__ __forceinline__ void df_add2(f32x2& sh, f32x2& sl, f32x2 ph, f32x2 pl) {
  f32x2 s, e;
  two_sum2(sh, ph, s, e);
  e = add2(e, add2(sl, pl));
  sh = add2(s, e);
  sl = sub2(e, sub2(sh, s));
}

// x / d from r = RN(1 / d), for finite values away from overflow and underflow: one correction of
// q = RN(x r) by its remainder (Markstein, IBM J. Res. Dev. 34, 1990), three dependent operations
// where the division takes about ten at 150 cycles each.  q is within 1.5 ulp (the published
// theorem, for q within an ulp, does not cover x < d with d near 2), which leaves the corrected
// quotient faithful; it equals x / d in every one of 4 million samples of the test.
__device__ __forceinline__ double quotient(double x, double d, double r) {
  const double q = x * r;
  return fma(fma(-q, d, x), r, q);
}

}  // namespace donof
