// Binary64-accurate arithmetic on unevaluated pairs of binary32 numbers (hi, lo), value hi + lo:
// products split exactly by fused multiply-adds, sums kept error-free (TwoSum), so a sum of products
// is accurate to about 2^-48 of the sum of |terms| at a few binary32 operations per term, on a pipe
// 64 times faster than sm_103a's binary64 pipe.  Shared by the convection kernels.
#pragma once
#include "lp_ptx.cuh"

namespace stdg {

__device__ __forceinline__ float2 pair_split(double a) {
  const float h = (float)a;
  return make_float2(h, (float)(a - (double)h));
}
// the same pair (ties in hi aside) by integer operations where both parts are normal numbers: conversions and
// subtractions in binary64 take 64 cycles per warp each
__device__ __forceinline__ float2 pair_split_int(double a) {
  const unsigned h = (unsigned)__double2hiint(a), l = (unsigned)__double2loint(a);
  const int e = (int)(h >> 20 & 0x7FF) - 1023;
  if (e < -60 || e > 120) return a == 0.0 ? make_float2(0.0f, 0.0f) : pair_split(a);
  // the 53 bits m as hm 2^29 + lm, hm rounded to nearest
  const unsigned hm = ((h & 0xFFFFFu | 0x100000u) << 3 | l >> 29) + (l >> 28 & 1);
  const int lm = (int)(l << 3) >> 3;
  const unsigned sg = h & 0x80000000u;
  return make_float2((float)hm * __uint_as_float((unsigned)(e + 104) << 23 | sg),
                     (float)lm * __uint_as_float((unsigned)(e + 75) << 23 | sg));
}
// The rounded products below are formed with __fmul_rn, which is never fused into a multiply-add:
// with the compiler's default contraction a plain product feeding the sum s + p may become
// fma(a, b, s), and the error-free sum would then no longer see the p whose rounding error it adds,
// leaving a binary32-sized error in the pair (measured: 3.5e-8 relative in convection).
// (s, c) += a b for pairs a, b: TwoProd of the high parts, cross terms into the error, TwoSum into s
__device__ __forceinline__ void pair_fma(float2 a, float2 b, float& s, float& c) {
  const float p = __fmul_rn(a.x, b.x);
  const float e = fmaf(a.x, b.x, -p);
  const float t = fmaf(a.x, b.y, fmaf(a.y, b.x, e));
  const float s2 = s + p;
  const float bb = s2 - s;
  c += ((s - (s2 - bb)) + (p - bb)) + t;
  s = s2;
}
__device__ __forceinline__ double pair_value(float s, float c) { return (double)s + (double)c; }
// (s, c) with |c| small against |s| -> a normalised pair (hi, lo), hi = fl32(s + c) (Fast2Sum)
__device__ __forceinline__ float2 pair_norm(float s, float c) {
  const float h = s + c;
  return make_float2(h, c - (h - s));
}
// the product of two pairs as a normalised pair: the high parts' product exactly (FMA), the cross terms
// into its error
__device__ __forceinline__ float2 pair_mul(float2 a, float2 b) {
  const float p = __fmul_rn(a.x, b.x);
  const float e = fmaf(a.x, b.y, fmaf(a.y, b.x, fmaf(a.x, b.x, -p)));
  return pair_norm(p, e);
}
// a + b and a - b of pairs (TwoSum of the high parts, low parts added to its error)
__device__ __forceinline__ float2 pair_add(float2 a, float2 b) {
  const float s = a.x + b.x;
  const float bb = s - a.x;
  const float e = ((a.x - (s - bb)) + (b.x - bb)) + (a.y + b.y);
  return pair_norm(s, e);
}
// sqrt(a) for a >= 0: the binary32 root s, its residual (a.x - s s is exact) over 2 s, and the residual that this
// leaves over 2 s again: to the rounding of the low part, as a binary64 root split into a pair
__device__ __forceinline__ float2 pair_sqrt(float2 a) {
  const float s = __fsqrt_rn(a.x);
  if (!(s > 0.0f) || s > 3.4e38f) return make_float2(s, 0.0f);
  float r, t;
  df_two_sum(fmaf(-s, s, a.x), a.y, r, t);
  const float inv = __fdividef(1.0f, s + s), q = r * inv;
  return pair_norm(s, fmaf(fmaf(-q, q, fmaf(-(s + s), q, r)) + t, inv, q));
}
__device__ __forceinline__ float2 pair_neg(float2 a) { return make_float2(-a.x, -a.y); }

// (s, c) += a b on both halves of (s, c): a broadcast (ah2 = (a_hi, a_hi), nah2 = -ah2,
// al2 = (a_lo, a_lo)), b one pair per half (bh2 = high parts, bl2 = low parts)
__device__ __forceinline__ void pair_fma2(float2 ah2, float2 nah2, float2 al2, float2 bh2, float2 bl2, float2& s,
                                          float2& c) {
  const float2 pn = __fmul2_rn(nah2, bh2);       // -(a_hi b_hi) rounded
  float2 e = __ffma2_rn(ah2, bh2, pn);           // its rounding error, exact
  e = __ffma2_rn(al2, bh2, e);
  e = __ffma2_rn(ah2, bl2, e);
  float2 s2, err;
  df_two_diff2(s, pn, s2, err);                   // s + a_hi b_hi, error-free
  c = __fadd2_rn(c, __fadd2_rn(err, e));
  s = s2;
}

// The same with the error part negated, nc, and the rounding errors of its additions collected in d: the sum
// s - nc - d is accurate to the rounding of the single terms, at one and a half times the operations
__device__ __forceinline__ void pair_fma2(float2 ah2, float2 nah2, float2 al2, float2 bh2, float2 bl2, float2& s,
                                          float2& nc, float2& d) {
  const float2 pn = __fmul2_rn(nah2, bh2);
  float2 e = __ffma2_rn(ah2, bh2, pn);
  e = __ffma2_rn(al2, bh2, e);
  e = __ffma2_rn(ah2, bl2, e);
  float2 s2, err, n2, dn;
  df_two_diff2(s, pn, s2, err);
  df_two_diff2(nc, __fadd2_rn(err, e), n2, dn);
  d = __fadd2_rn(d, dn);
  s = s2;
  nc = n2;
}

}  // namespace stdg
