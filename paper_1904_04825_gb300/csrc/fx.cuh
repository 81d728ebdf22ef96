// FP64 sums of products on the integer units.
//
// GB300 starts 2 FP64 operations per clock and SM but 57 32 x 32 + 64-bit integer
// multiply-adds (measured).  A group of values is written as 57-bit integers with
// the group's largest exponent: x = v 2^(e - 1079), v = hi 2^28 + lo with lo a
// signed 28-bit and hi a 30-bit number.  A product then is three multiply-adds
// (hi hi, hi lo + lo hi; lo lo is below the last place kept), exact and free of
// order, and a sum of up to 32 of them is rounded once to FP64.  An operand is
// rounded to 2^-57 of its group's largest value, so a sum carries 2^-57 of
// (largest of one group) x (largest of the other) per term, where an FP64 chain
// commits 2^-53 of every partial sum: values far below their group's largest lose
// digits, and the caller scales the terms so that the groups are even (gj_fx.cuh).
// Subnormal values count as zero; an infinity or NaN gives its group the exponent
// kNonFinite, which makes the result NaN.
#pragma once

#include "device.cuh"

namespace frk {
namespace fx {

constexpr int kNonFinite = 1 << 20, kNone = -(1 << 20);  // exponents of a non-finite value and of zero

__device__ __forceinline__ int exponent(double x) { return (__double2hiint(x) >> 20) & 0x7ff; }
// the exponent of x scaled by 2^d in its group
__device__ __forceinline__ int exponent_of(double x, int d) {
  const int e = exponent(x);
  return e == 0 ? kNone : e == 2047 ? kNonFinite : e + d;
}

// x 2^d as hi 2^28 + lo for the group exponent e >= exponent_of(x, d)
__device__ __forceinline__ int2 split(double x, int d, int e) {
  const int ex = exponent(x), sh = e - ex - d;
  long long m = (__double_as_longlong(x) & 0xfffffffffffffll) | 0x10000000000000ll;
  m <<= 4;
  if (sh > 0) m = sh < 60 ? (m + (1ll << (sh - 1))) >> sh : 0;
  if (ex == 0) m = 0;
  if (__double2hiint(x) < 0) m = -m;
  const int lo = (int)((m << 36) >> 36);
  return make_int2((int)((m - lo) >> 28), lo);
}

struct Acc {
  long long hh = 0, x = 0;
};
__device__ __forceinline__ void mad(Acc& a, int2 u, int2 v) {
  asm("mad.wide.s32 %0, %1, %2, %0;" : "+l"(a.hh) : "r"(u.x), "r"(v.x));
  asm("mad.wide.s32 %0, %1, %2, %0;" : "+l"(a.x) : "r"(u.x), "r"(v.y));
  asm("mad.wide.s32 %0, %1, %2, %0;" : "+l"(a.x) : "r"(u.y), "r"(v.x));
}
// 2^(e - 1079) for e = e1 + e2 of the two groups: zero below the normal range and for
// a group of zeros, infinite above it and for a group that holds a non-finite value
__device__ __forceinline__ double scale(int e1, int e2) {
  int b = e1 + e2 - 1079;
  if (b < 1) b = 0;
  if (b > 2046 || e1 == kNonFinite || e2 == kNonFinite) b = 2047;
  return __hiloint2double(b << 20, 0);
}
// the sum, to be multiplied by scale(e1, e2)
__device__ __forceinline__ double value(const Acc& a) { return (double)(a.hh + ((a.x + (1ll << 27)) >> 28)); }

}  // namespace fx
}  // namespace frk
