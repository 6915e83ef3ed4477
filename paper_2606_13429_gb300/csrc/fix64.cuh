// 64-bit fixed-point arithmetic for FP64 data.
//
// This GPU issues FP64 FMAs on 2 lanes per clock per SM (measured 1.98), but
// 32 x 32 + 64 bit integer multiply-adds (IMAD.WIDE) on 64 (measured 62.8) and
// 64-bit integer additions on 63. A product of a 61-bit fixed-point value
// with a 59-bit constant takes three such multiply-adds (20.6 per clock per
// SM measured), so a linear map of bounded values runs about ten times
// faster in fixed point than in FP64. The values of a block share one
// exponent: its largest entry carries 53 to 58 bits (ras_fix.cu), smaller ones
// fewer, against 53 for every entry in FP64, so errors are relative to the
// block's largest entry.
//
// A value v (|v| < 2^60) is split as v = h 2^29 + l, |l| <= 2^28; a constant
// c (|c| < 2) is stored as C = round(c 2^58) = c1 2^29 + c0, |c0| <= 2^28, c1
// in .x and c0 in .y. Then
//   c v = h c1 + 2^-29 (h c0 + l c1) + 2^-58 l c0,
// the last term (below a quarter of a unit, no bias) is dropped and the middle
// one is rounded to nearest. The middle sums of up to 8 products with
// sum |c| <= 4 stay below 2^63: 8 (2^31 2^28) + 4 (2^28 2^29).
#pragma once

#include <cstdint>

namespace dcg {

struct FxAcc {
  long long H, M;
};
__device__ __forceinline__ FxAcc fx_zero() { return FxAcc{0, 1LL << 28}; }  // rounds the middle term
struct FxVal {
  int h, l;
};
__device__ __forceinline__ FxVal fx_split(long long v) {
  const int h = (int)((v + (1LL << 28)) >> 29);
  return FxVal{h, (int)((unsigned)v - ((unsigned)h << 29))};
}
// written as the instruction: from C the compiler forms other sequences
__device__ __forceinline__ void fx_madw(long long& acc, int a, int b) {
  asm("mad.wide.s32 %0, %1, %2, %0;" : "+l"(acc) : "r"(a), "r"(b));
}
__device__ __forceinline__ void fx_mac(FxAcc& a, const FxVal& v, int c1, int c0) {
  fx_madw(a.H, v.h, c1);
  fx_madw(a.M, v.h, c0);
  fx_madw(a.M, v.l, c1);
}
__device__ __forceinline__ long long fx_value(const FxAcc& a) { return a.H + (a.M >> 29); }

// FP64 bit patterns. The exponent of a block is the exponent field of its
// largest magnitude, found on the high words (IEEE order is integer order).
constexpr unsigned kFxNonFinite = 0x7ff00000u;
__device__ __forceinline__ unsigned fx_mag(long long bits) { return (unsigned)(bits >> 32) & 0x7fffffffu; }
// A block whose largest entry lies near an end of the FP64 range (exponent
// field below 192 or from 1856) is first scaled by 2^320 or 2^-320 and its
// results back: entries then are normal numbers and no exponent below leaves
// the range. In every other block zeros and subnormals, whose significand has
// no implicit bit, lie so far below the largest entry that they vanish.
constexpr int kFxLift = 320, kFxLowest = 192;
__device__ __forceinline__ bool fx_odd(unsigned mag) { return mag - ((unsigned)kFxLowest << 20) >= 1664u << 20; }  // or not finite
__device__ __forceinline__ int fx_lift(unsigned mag) {
  return mag < (unsigned)kFxLowest << 20 ? 1 : mag >= 1856u << 20 && mag < kFxNonFinite ? -1 : 0;
}
__device__ __forceinline__ double fx_two320(int lift) {
  return lift == 0 ? 1.0 : __longlong_as_double((long long)(1023 + kFxLift * lift) << 52);
}
__device__ __forceinline__ long long fx_scaled(long long bits, double s) {
  return __double_as_longlong(__longlong_as_double(bits) * s);
}
// exponent field of a scaled block (one of subnormals counts as 2^-1022)
__device__ __forceinline__ int fx_odd_exponent(unsigned mag, int lift) {
  return max((int)(mag >> 20), 1) + kFxLift * lift;
}
// FP64 bits to fixed point with |result| <= 2^nb, rounded to nearest: the
// significand moves right by sh0 - (exponent field), sh0 = 63 - nb + (block
// exponent).
__device__ __forceinline__ long long fx_signed_significand(unsigned hi, unsigned lo) {
  const int s = (int)hi >> 31;  // one's complement: 2^-62 of the value
  const unsigned mh = __funnelshift_l(lo, (hi & 0xfffffu) | 0x100000u, 10);  // leading bit 62
  return (long long)((unsigned long long)(mh ^ (unsigned)s) << 32 | ((lo << 10) ^ (unsigned)s));
}
__device__ __forceinline__ long long fx_near(long long bits, int sh0) {
  const unsigned hi = (unsigned)(bits >> 32);
  const int sh = min(sh0 - 1 - (int)(hi << 1 >> 21), 63);
  return ((fx_signed_significand(hi, (unsigned)bits) >> sh) + 1) >> 1;
}
// v 2^(e0 - 1085) to FP64, rounded to nearest, |v| < 2^62, 63 < e0 < 0x7ff (no
// result leaves the normal range)
__device__ __forceinline__ double fx_to_double(long long v, int e0) {
  const long long s = v >> 63;
  const unsigned long long a = (unsigned long long)((v ^ s) - s);
  const int lz = __clzll((long long)a) - 1;  // 1 .. 63
  const unsigned long long sig = ((a << lz) + 0x200) >> 10;  // 2^52 .. 2^53
  const int e = e0 - lz;  // exponent field of 2^52 <= sig < 2^53
  long long bits = (long long)(((unsigned long long)(unsigned)(e - 1) << 52) + sig);
  bits = a == 0 ? 0 : bits;
  return __longlong_as_double(bits | (s & (long long)0x8000000000000000ull));
}

}  // namespace dcg
