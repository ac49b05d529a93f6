// Fixed-point arithmetic with FP64 accuracy on the integer pipe (GB300: 64 mad.wide per clock and
// SM against 2 FP64 FMAs).  A number is an integer t times a power of two common to the sums it
// takes part in, held in two limbs t = hi 2^27 + lo, |lo| <= 2^26.  A product of two numbers is
// hi hi 2^54 + (hi lo + lo hi) 2^27, two exact 64-bit sums; lo lo is left out (at most 2^52).
#pragma once

#include <cuda_runtime.h>
#include <math.h>
#include <stdint.h>

namespace qf {
namespace {

constexpr int kLimb = 27;  // bits of a low limb

// round(v 2^(bits - sx)): v in units of 2^(sx - bits); |v| < 2^(sx + 62 - bits).  Subnormal v count
// as zero.
__device__ __forceinline__ long long to_fix(double v, int sx, int bits) {
  const long long b = __double_as_longlong(v);
  const int e = (int)((b >> 52) & 0x7ff);
  if (e == 0) return 0;
  const long long m = (b & 0xfffffffffffffll) | 0x10000000000000ll;
  const int sh = e - 1075 + bits - sx;
  long long t;
  if (sh >= 0) {
    t = m << (sh > 9 ? 9 : sh);
  } else {
    const int r = -sh;
    t = r > 60 ? 0 : (m + (1ll << (r - 1))) >> r;
  }
  return b < 0 ? -t : t;
}
__device__ __forceinline__ int2 limbs(long long t) {
  const long long hi = (t + (1ll << (kLimb - 1))) >> kLimb;
  return make_int2((int)hi, (int)(t - (hi << kLimb)));
}
__device__ __forceinline__ long long unlimb(int2 w) { return ((long long)w.x << kLimb) + w.y; }
__device__ __forceinline__ void madw(long long& s, int a, int b) { s += (long long)a * b; }
// (high sum, cross sum) -> one sum in units of 2^54 products
__device__ __forceinline__ long long join(long long hh, long long xx) {
  return hh + ((xx + (1ll << (kLimb - 1))) >> kLimb);
}
// t 2^e, rounded to nearest, by field arithmetic (an int64 conversion and a multiplication hold the FP64
// pipe); results outside the normal range take ldexp
__device__ __forceinline__ double fix_value(long long t, int e) {
  const unsigned long long u = t < 0 ? 0ull - (unsigned long long)t : (unsigned long long)t;
  const int lz = __clzll((long long)u);
  const unsigned long long m = (((u << (lz & 63)) >> 10) + 1) >> 1;  // 2^52 .. 2^53
  const int ex = e + 1086 - lz;                                     // biased exponent of the leading bit
  if (t == 0) return 0.0;
  if (ex < 2 || ex > 2045) return ldexp((double)t, e);
  const unsigned long long b = ((unsigned long long)(ex - 1) << 52) + m;
  return __longlong_as_double((long long)(t < 0 ? b | 0x8000000000000000ull : b));
}
// 2^e as a double, |e| < 1022
__device__ __forceinline__ double pow2(int e) { return __longlong_as_double((long long)(e + 1023) << 52); }

// binary64 <-> binary32 by field arithmetic (a conversion holds the FP64 pipe, 64 cycles a warp): the
// float is cut off after its 23 bits.  Only for |x| in the normal FP32 range (2^-126 .. 2^127): outside it the
// exponent field wraps, so callers bound their arguments first.
__device__ __forceinline__ float cut_float(double x) {
  const unsigned hi = (unsigned)__double2hiint(x), lo = (unsigned)__double2loint(x);
  return __uint_as_float((hi & 0x80000000u) | (((hi & 0x7fffffffu) - (896u << 20)) << 3) | (lo >> 29));
}
__device__ __forceinline__ double wide(float x) {
  const unsigned u = __float_as_uint(x);
  return __hiloint2double((int)((u & 0x80000000u) | (((u & 0x7fffffffu) >> 3) + (896u << 20))), (int)(u << 29));
}
// 1 / x: FP32 reciprocal y of the cut x, off by d <= 2^-23 + 2^-24, and one Newton step (y += y (1 - x y)),
// which leaves d^2 < 2^-44; 2^-125 <= |x| <= 2^125.
__device__ __forceinline__ double recip(double x) {
  const double y = wide(__frcp_rn(cut_float(x)));
  return fma(fma(-x, y, 1.0), y, y);
}
// 1 / sqrt(x): FP32 estimate y (off by less than 2^-21) and the binomial series of (1 - e)^(-1/2), e = 1 - x y^2,
// y (1 + e / 2 + 3 e^2 / 8), whose next term 5 e^3 / 16 is below 2^-61: rounding is what is left, below
// 2^-52; 2^-125 <= x <= 2^125.
__device__ __forceinline__ double rsqrt_nr(double x) {
  const double y = wide(rsqrtf(cut_float(x)));
  const double e = fma(-x * y, y, 1.0);
  return fma(y * e, fma(0.375, e, 0.5), y);
}

}  // namespace
}  // namespace qf
