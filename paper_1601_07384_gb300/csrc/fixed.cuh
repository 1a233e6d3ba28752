// Sums of binary64 products in 64-bit fixed point on the integer pipe.
//
// sm_103a multiplies 32 x 32 + 64 bits (IMAD.WIDE) at 32 times the rate of its binary64 FMA: 2 cycles per
// warp instruction against 64 (measured: 18.6 T/s against 0.6 T/s).  A matrix block and a vector are
// therefore scaled to integers by their largest exponents,
//     a = a_int 2^(ea - 1022 - kFxA),  |a_int| < 2^kFxA,      x = x_int 2^(ex - 1022 - kFxX),  |x_int| < 2^kFxX
// and split into two signed 29-bit limbs, v_int = h 2^29 + l.  A product takes three multiply-adds,
//     S0 += h_a h_x,   S1 += h_a l_x + l_a h_x
// (l_a l_x, below 2^-57 of the full scale, is left out).  The sums of up to 35 products are exact in 64
// bits (|S0| < 35 2^55, |S1| < 35 1.5 2^56), and sums over several blocks are exact in 128 bits, so the
// only errors are the truncation of the operands at 2^-57 (2^-56) of their largest entry and the one
// rounding of the result to binary64: below a binary64 sum's own rounding, and independent of the order.
//
// Exponents are the biased ones of binary64.  A block or vector whose largest exponent is not in
// [kFxMinExp, 2046] (non-finite entries, or all entries below about 1e-289) does not take this path: the
// callers then form the sum with binary64 multiply-adds.  An exponent of 0 means that all entries are 0.
#pragma once
#include <cstdint>

namespace stdg {

constexpr int kFxA = 57, kFxX = 56;
constexpr int kFxMinExp = 64;      // entries 2^-63 of the largest are still normal numbers
constexpr int kFxL = 29;           // bits of the lower limb

// biased exponent of v, 1 for subnormal numbers, 0 for zero
__device__ __forceinline__ int fx_exp(double v) {
  const int hi = __double2hiint(v), e = (hi >> 20) & 0x7FF;
  return e ? e : (((hi << 1) | __double2loint(v)) != 0 ? 1 : 0);
}
__device__ __forceinline__ bool fx_ok(int e) { return e == 0 || (e >= kFxMinExp && e <= 2046); }

// h 2^29 + l = trunc(v 2^(BITS + 1022 - emax)) for exponents of v up to emax, emax >= kFxMinExp
template <int BITS>
__device__ __forceinline__ void fx_limbs(double v, int emax, int& h, int& l) {
  const int hi = __double2hiint(v);
  const uint32_t lo = (uint32_t)__double2loint(v);
  const uint32_t sh = (uint32_t)(emax - ((hi >> 20) & 0x7FF));
  unsigned long long m = ((unsigned long long)(((uint32_t)hi & 0xFFFFFu) | 0x100000u) << 32 | lo) << (BITS - 53);
  asm("shr.u64 %0, %1, %2;" : "=l"(m) : "l"(m), "r"(sh));     // counts above 63 give 0
  const int s = hi >> 31;
  const int ml = ((int)(uint32_t)m << 3) >> 3, mh = (int)((m + (1u << 28)) >> kFxL);
  l = (ml ^ s) - s;
  h = (mh ^ s) - s;
}
// the same for an integer |m| < 2^BITS
__device__ __forceinline__ int2 fx_limbs_int(long long m) {
  return make_int2((int)((m + (1 << 28)) >> kFxL), ((int)(uint32_t)m << 3) >> 3);
}
__device__ __forceinline__ void fx_mad(int ah, int al, int xh, int xl, long long& S0, long long& S1) {
  S0 += (long long)ah * xh;
  S1 += (long long)ah * xl;
  S1 += (long long)al * xh;
}
// exponent k of the unit of S0 2^29 + S1 for operand exponents ea, ex: the sum is (S0 2^29 + S1) 2^k
__device__ __forceinline__ int fx_unit(int ea, int ex) { return ea + ex - 2044 - kFxA - kFxX + kFxL; }

// T 2^k rounded to binary64
__device__ __forceinline__ double fx_value(__int128 T, int k) {
  const bool neg = T < 0;
  const unsigned __int128 m = neg ? (unsigned __int128)(-T) : (unsigned __int128)T;
  unsigned long long hi = (unsigned long long)(m >> 64), lo = (unsigned long long)m;
  if (hi) {
    const int s = 64 - __clzll((long long)hi);                 // 1..63 (|T| < 2^120)
    lo = (hi << (64 - s)) | (lo >> s) | ((lo << (64 - s)) != 0 ? 1ull : 0ull);   // sticky last bit
    k += s;
  }
  if (lo == 0) return 0.0;
  const double d = __ull2double_rn(lo);
  const int dh = __double2hiint(d), e = (dh >> 20) + k;        // d is positive and normal
  const double r = e >= 1 && e <= 2046 ? __hiloint2double(dh + (k << 20), __double2loint(d)) : scalbn(d, k);
  return neg ? -r : r;
}

// A small matrix (the time matrices) in limbs with one exponent; the entries as they are for the
// binary64 path.  on == 0: the identity (no mixing).
struct FxMat {
  int on, e;
  int h[25], l[25];
  double v[25];
};

}  // namespace stdg
