// Sums of binary64 products in 64-bit fixed point on the integer pipe.
//
// sm_103a multiplies 32 x 32 + 64 bits (IMAD.WIDE) at 16 times the rate of its binary64 FMA: 4 cycles per
// warp instruction against 64 (measured with operands from shared memory).  A matrix block and a vector are
// therefore scaled to integers by their largest exponents,
//     v = v_int 2^(e - 1022 - kFx),   |v_int| <= 2^kFx,   kFx = 61, rounded to nearest,
// and split into two limbs, v_int = h 2^31 + l with |h|, |l| <= 2^30.  A product takes three multiply-adds,
//     S0 += h_a h_x,   S1 += h_a l_x + l_a h_x
// (l_a l_x, of either sign and below 2^-62 of the full scale, is left out).  The sums of two products are
// exact in 64 bits and are added up in 96 bits each, T = S0 2^31 + S1 is formed once per row and block and
// kept to 96 bits (2^-85 of the full scale), the blocks of an output are added, aligned by their exponents,
// and the sum is rounded to binary64 once.  The multiplier binds, so the wide additions (on the other
// integer pipe) are nearly free.  Against a binary64 sum: the operands are rounded at 2^-62 of their
// largest entry instead of not at all, and the 35 to 420 roundings of the partial sums at 2^-53 of their
// size are saved.  The result does not depend on the order.
//
// The cut relative to the largest entry is harmless only if the products that matter are near the largest
// product.  The blocks of the operator grow with the polynomial degree (as the square of it) and the
// vectors fall off with it, so rows and columns are first scaled by powers of two, one per mode and the
// same for all blocks (FxScale): the operator by the square root of its diagonal, which leaves no entry
// of the symmetric positive definite blocks above about 1, and Q to match.
//
// The blocks are static, so they are stored in this form (8 bytes an entry, as binary64): the limbs and
// one exponent per block.  Exponents are the biased ones of binary64.  A block or vector whose largest
// exponent is not in [kFxMinExp, 2046] (non-finite entries, or all entries below about 1e-289) does not
// take this path: such a block is stored as binary64, and the products are then formed with binary64
// multiply-adds.  An exponent of 0 means that all entries are 0.
#pragma once
#include <cmath>
#include <cstdint>
#include <cstring>

namespace stdg {

constexpr int kFx = 61;            // bits of an entry
constexpr int kFxMinExp = 64;      // entries 2^-63 of the largest are still normal numbers
constexpr int kFxL = 31;           // bits of the lower limb

// biased exponent of v, 1 for subnormal numbers, 0 for zero
__device__ __forceinline__ int fx_exp(double v) {
  const int hi = __double2hiint(v), e = (hi >> 20) & 0x7FF;
  return e ? e : (((hi << 1) | __double2loint(v)) != 0 ? 1 : 0);
}
__device__ __forceinline__ bool fx_ok(int e) { return e == 0 || (e >= kFxMinExp && e <= 2046); }

// exponents by which the rows or columns of the blocks of an operator are scaled, one per mode
struct FxScale { signed char s[40]; };
// The blocks of an operator (len entries each): entry idx of
// block b at w[b * len + idx], divided by 2^(r.s[row] + c.s[column]), as limbs (h, l), or as binary64 where
// the block's exponent e[b] is outside the range.
struct FxBlocks { const int2* w; const uint16_t* e; FxScale r, c; };
// rounded to binary32 (sc: the scaling of its row and column): of the 61 bits at once and without the binary64
// pipe, where the value is certain to be in the normal range
__device__ __forceinline__ float fx_entry_f32(const FxBlocks& B, size_t len, size_t b, int idx, int sc) {
  const int2 w = B.w[b * len + idx];
  const int e = B.e[b], k = e - 1022 - kFx + sc;
  if (fx_ok(e) && k >= -120 && k <= 60) return __ll2float_rn((long long)w.x * (1LL << kFxL) + w.y) * __int_as_float((k + 127) << 23);
  if (!fx_ok(e)) return (float)scalbn(__hiloint2double(w.y, w.x), sc);
  return e ? (float)scalbn((double)((long long)w.x * (1LL << kFxL) + w.y), k) : 0.0f;
}
// the same on the host, for an entry copied as the 8 bytes that it is stored in
inline double fx_entry_host(double raw, int e, int sc) {
  if (e != 0 && (e < kFxMinExp || e > 2046)) return std::ldexp(raw, sc);
  int w[2];
  std::memcpy(w, &raw, sizeof w);
  return std::ldexp((double)((long long)w[0] * (1LL << kFxL) + w[1]), e - 1022 - kFx + sc);
}
__device__ __forceinline__ int2 fx_encode(double v, int e) {
  if (!fx_ok(e)) return make_int2(__double2loint(v), __double2hiint(v));
  if (!e) return make_int2(0, 0);
  const long long m = __double2ll_rn(scalbn(v, kFx + 1022 - e));
  const int h = (int)((m + (1LL << (kFxL - 1))) >> kFxL);
  return make_int2(h, (int)(m - ((long long)h << kFxL)));
}

// an integer |m| <= 2^kFx in limbs
__device__ __forceinline__ int2 fx_split(long long m) {
  const int h = (int)((m + (1LL << (kFxL - 1))) >> kFxL);
  return make_int2(h, (int)((uint32_t)m - ((uint32_t)h << kFxL)));
}
// the limbs of a vector entry, v 2^(kFx + 1022 - emax) rounded to nearest, for exponents of v up to emax,
// emax >= kFxMinExp
__device__ __forceinline__ int2 fx_limbs_x(double v, int emax) {
  const int hi = __double2hiint(v);
  const uint32_t sh = (uint32_t)(emax - ((hi >> 20) & 0x7FF));
  const uint32_t mh = ((uint32_t)hi & 0xFFFFFu) | 0x100000u, ml = (uint32_t)__double2loint(v);
  unsigned long long m = ((unsigned long long)mh << 32 | ml) << (kFx + 1 - 53);   // one bit more, to round
  asm("shr.u64 %0, %1, %2;" : "=l"(m) : "l"(m), "r"(sh));     // counts above 63 give 0
  m = (m + 1) >> 1;
  return fx_split(hi < 0 ? -(long long)m : (long long)m);
}

// T0 2^31 + T1, both in 96 bits.  The sums of two products are biased by 2^62 to be non-negative (no sign
// to extend); fx_sum takes the bias off again.
struct FxAcc { uint32_t t0[3], t1[3]; };
constexpr long long kFxBias = 1LL << 62;
__device__ __forceinline__ void fx_add64(uint32_t (&T)[3], long long S) {
  asm("add.cc.u32 %0, %0, %3;\n\taddc.cc.u32 %1, %1, %4;\n\taddc.u32 %2, %2, 0;"
      : "+r"(T[0]), "+r"(T[1]), "+r"(T[2]) : "r"((uint32_t)S), "r"((uint32_t)((unsigned long long)S >> 32)));
}
// += a0 x0 + a1 x1 (limbs (h, l); the limbs come from memory: of one that the compiler can prove
// non-negative it would form the mixed product from several instructions)
__device__ __forceinline__ void fx_mad2(int2 a0, int2 x0, int2 a1, int2 x1, FxAcc& T) {
  long long S0 = kFxBias + (long long)a0.x * x0.x;
  long long S1 = kFxBias + (long long)a0.x * x0.y;
  S0 += (long long)a1.x * x1.x;
  S1 += (long long)a0.y * x0.x;
  S1 += (long long)a1.x * x1.y;
  S1 += (long long)a1.y * x1.x;
  fx_add64(T.t0, S0);
  fx_add64(T.t1, S1);
}
__device__ __forceinline__ void fx_mad1(int2 a, int2 x, FxAcc& T) {
  const long long S0 = kFxBias + (long long)a.x * x.x;
  long long S1 = kFxBias + (long long)a.x * x.y;
  S1 += (long long)a.y * x.x;
  fx_add64(T.t0, S0);
  fx_add64(T.t1, S1);
}
// (T0 2^31 + T1) 2^-6 rounded down, in three 32-bit words (|.| < 2^91); n: the number of biases in T0, T1
struct FxSum { uint32_t a, b, c; };
__device__ __forceinline__ FxSum fx_sum(FxAcc T, int n) {
  const uint32_t b1 = (uint32_t)n << 30, b2 = (uint32_t)n >> 2;            // n 2^62
  asm("sub.cc.u32 %0, %0, %2;\n\tsubc.u32 %1, %1, %3;" : "+r"(T.t0[1]), "+r"(T.t0[2]) : "r"(b1), "r"(b2));
  asm("sub.cc.u32 %0, %0, %2;\n\tsubc.u32 %1, %1, %3;" : "+r"(T.t1[1]), "+r"(T.t1[2]) : "r"(b1), "r"(b2));
  FxSum t;
  asm("add.cc.u32 %0, %3, %6;\n\taddc.cc.u32 %1, %4, %7;\n\taddc.u32 %2, %5, %8;"
      : "=r"(t.a), "=r"(t.b), "=r"(t.c)
      : "r"(T.t0[0] << 25), "r"(__funnelshift_l(T.t0[0], T.t0[1], 25)), "r"(__funnelshift_l(T.t0[1], T.t0[2], 25)),
        "r"(__funnelshift_r(T.t1[0], T.t1[1], 6)), "r"(__funnelshift_r(T.t1[1], T.t1[2], 6)),
        "r"((uint32_t)((int)T.t1[2] >> 6)));
  return t;
}
// T += t >> d (rounded down), d >= 0
__device__ __forceinline__ void fx_add(FxSum& T, FxSum t, int d) {
  while (d >= 32) {                          // whole words first (blocks of very different scales)
    t.a = t.b; t.b = t.c; t.c = (uint32_t)((int)t.c >> 31);
    d = d >= 128 ? 96 : d - 32;              // 96 bits or more: only the sign is left
  }
  t.a = __funnelshift_r(t.a, t.b, d);
  t.b = __funnelshift_r(t.b, t.c, d);
  t.c = (uint32_t)((int)t.c >> d);
  asm("add.cc.u32 %0, %0, %3;\n\taddc.cc.u32 %1, %1, %4;\n\taddc.u32 %2, %2, %5;"
      : "+r"(T.a), "+r"(T.b), "+r"(T.c) : "r"(t.a), "r"(t.b), "r"(t.c));
}
// the unit of T is 2^fx_unit(ea, ex)
__device__ __forceinline__ int fx_unit(int ea, int ex) { return ea + ex - 2044 - 2 * kFx + kFxL + 6; }
// T 2^k rounded to binary64 (to nearest, ties to even), by integer operations: the conversion of a 64-bit
// integer to binary64 takes 64 cycles per warp, as every instruction of the binary64 pipe
__device__ __forceinline__ double fx_value(const FxSum& T, int k) {
  const uint32_t s = (uint32_t)((int)T.c >> 31);
  uint32_t a = T.a, b = T.b, c = T.c;
  if (s) asm("sub.cc.u32 %0, 0, %0;\n\tsubc.cc.u32 %1, 0, %1;\n\tsubc.u32 %2, 0, %2;" : "+r"(a), "+r"(b), "+r"(c));
  k += 1023 + 95;                            // biased exponent of 2^95 2^k
  if (c == 0) { c = b; b = a; a = 0; k -= 32; }
  if (c == 0) { c = b; b = 0; k -= 32; }
  if (c == 0) return 0.0;
  const int n = __clz((int)c);               // the leading 64 bits, top bit set; the rest only as a sticky bit
  k -= n;
  const uint32_t lo0 = __funnelshift_l(a, b, n);
  unsigned long long m = (unsigned long long)__funnelshift_l(b, c, n) << 32 | lo0 | ((a << n) != 0 ? 1u : 0u);
  const unsigned long long r = m + (0x3FFull + ((m >> 11) & 1ull));
  const unsigned long long f = (r >> 11) + (r < m ? 1ull << 53 : 0ull);      // with the leading bit: 2^52 .. 2^53
  if (k >= 1 && k <= 2045)
    return __longlong_as_double((long long)((f + ((unsigned long long)(k - 1) << 52)) | (unsigned long long)s << 63));
  const double d = scalbn(__longlong_as_double((long long)(f + (1022ull << 52))), k - 1023);
  return s ? -d : d;
}

// entry idx of block b rounded to binary64, without the binary64 pipe
__device__ __forceinline__ double fx_entry(const FxBlocks& B, size_t len, size_t b, int idx, int N) {
  const int2 w = B.w[b * len + idx];
  const int e = B.e[b], sc = B.r.s[idx / N % N] + B.c.s[idx % N];
  if (!fx_ok(e)) return scalbn(__hiloint2double(w.y, w.x), sc);
  const long long m = (long long)w.x * (1LL << kFxL) + w.y;
  return fx_value(FxSum{(uint32_t)m, (uint32_t)((unsigned long long)m >> 32), (uint32_t)(m >> 63)}, e - 1022 - kFx + sc);
}

// A small matrix (the time matrices) in limbs with one exponent; the entries as they are for the
// binary64 path.  on == 0: the identity (no mixing).
struct FxMat {
  int on, e;
  int h[25], l[25];
  double v[25];
};

}  // namespace stdg
