// dirac_fixed.cuh -- 60-bit fixed-point arithmetic for the FP64 kernels.
//
// GB300 issues one FP64 instruction per warp and SM sub-partition every 64 to
// 76 cycles (measured: DFMA 64, DADD and DMUL 76, every conversion from or to
// FP64 64), while a 32 x 32 + 64 bit integer multiply-add (IMAD.WIDE), a
// 64-bit add or a 32-bit shift takes 2.  A product of two 60-bit numbers in
// two 32-bit limbs is three IMAD.WIDE (four with the product of the lower
// limbs), accumulated without rounding and rounded once at the end of the sum;
// converting a double by shifting its mantissa is about a dozen integer
// instructions.  So sums of products whose operands share a scale are several
// times cheaper here than on the FP64 pipe, at 5 to 7 bits more than FP64's 53
// relative to the largest operand of the group that shares the scale (and that
// many fewer for an operand so much smaller than the largest).
#pragma once
#include <cuda_runtime.h>

namespace dirac {
namespace fx {

// Exponent field ("be") of a double; |x| < 2^(be - 1022).
__device__ __forceinline__ int exp_field(double x) { return (__double2hiint(x) >> 20) & 0x7ff; }

// x 2^(F - (be - 1022)) truncated towards zero, |result| < 2^F, for an x whose
// exponent field is at most be (53 <= F <= 60).  Zero gives zero as long as
// be >= 63; so do subnormals.
template <int F>
__device__ __forceinline__ long long to_fixed(double x, int be) {
  const int hi = __double2hiint(x);
  const unsigned lo = (unsigned)__double2loint(x);
  unsigned long long m = ((unsigned long long)(unsigned)((hi & 0xfffff) | 0x100000) << 32 | lo) << (F - 53);
  m >>= min(be - ((hi >> 20) & 0x7ff), 63);
  const long long s = (long long)(hi >> 31);
  return (long long)(m ^ (unsigned long long)s) - s;
}

// v 2^e as a double (v below 2^62; one rounding), for results in the normal range
__device__ __forceinline__ double to_double(long long v, int e) {
  const double d = (double)v;
  return v ? __hiloint2double(__double2hiint(d) + (e << 20), __double2loint(d)) : 0.0;
}

// v = hi 2^32 + lo with a signed lo, so that products without lo x lo stay
// unbiased: two instructions, the words themselves
struct Limbs {
  int hi, lo;
};
__device__ __forceinline__ Limbs split(long long v) {
  Limbs l;
  l.lo = (int)(unsigned)v;
  l.hi = (int)(v >> 32) + (int)((unsigned)v >> 31);
  return l;
}

// Rows of the operator: numbers of ROW_BITS bits times coefficients of 60, summed in
// Acc and rounded to units of 2^(32 + ROW_SHIFT).  A difference of the stencil (of
// both directions, in order 4 with an eighth of the outer one: 4.5 numbers) and five
// more products stay below 2^63 in Acc's cross terms and below 2^62 in the result.
// The products' lo x lo that Acc drops are each up to 2^-57 of a number times a
// coefficient, both the largest: with 58 bits (and 55 in order 4, the outer
// difference not divided) the root mean square error of a row was 2^-57.2 (2^-54.2)
// of the sum of its terms on an even tile, now 2^-58.1 (2^-57.4); FP64's is 2^-56.8.
constexpr int ROW_BITS = 59, ROW_SHIFT = 29;

// Sum of products a b, a and b in limbs, without their lo x lo (2^62 each at most,
// of either sign): h in units of 2^64, x of 2^32 (both wrap like unsigned numbers).
struct Acc {
  unsigned long long h = 0, x = 0;
  __device__ __forceinline__ void mac(const Limbs& a, const Limbs& b) {
    h += (unsigned long long)((long long)a.hi * b.hi);
    x += (unsigned long long)((long long)a.hi * b.lo);
    x += (unsigned long long)((long long)a.lo * b.hi);
  }
  // the sum in units of 2^(32 + S), rounded
  template <int S>
  __device__ __forceinline__ long long value() const {
    return (long long)((h << (32 - S)) + (unsigned long long)((long long)(x + (1ULL << (S - 1))) >> S));
  }
};

__device__ __forceinline__ long long eighth(long long v) { return (v + 4) >> 3; }   // rounded

// Sum of squares: x holds half of the cross terms; lo x lo, never negative, is
// kept too (to 2^-29 of itself): without it the sum had a bias
struct SqAcc {
  unsigned long long h = 0, x = 0, l = 0;
  __device__ __forceinline__ void sqr(const Limbs& a) {
    h += (unsigned long long)((long long)a.hi * a.hi);
    x += (unsigned long long)((long long)a.hi * a.lo);
    const int b = a.lo >> 2;
    l += (unsigned long long)((long long)b * b);
  }
  // the sum in units of 2^60, rounded (up to 2^63)
  __device__ __forceinline__ unsigned long long value() const {
    return (h << 4) + (unsigned long long)((long long)(x + (l >> 29) + (1ULL << 26)) >> 27);
  }
};

// v / 2^s, rounded (s >= 0)
__device__ __forceinline__ long long shr_round(long long v, int s) {
  if (s <= 0) return v;
  if (s > 62) return 0;
  return (v + (1LL << (s - 1))) >> s;
}

// Sum over the warp of a number of each lane, exactly, in three pieces of 21
// and 22 bits (the top piece signed or not, as T is): t2 2^42 + t1 2^21 + t0
struct WarpSum {
  int t2, t1, t0;
};
template <class T>
__device__ __forceinline__ WarpSum warp_sum(T v) {
  WarpSum s;
  s.t2 = __reduce_add_sync(0xffffffffu, (int)(v >> 42));
  s.t1 = __reduce_add_sync(0xffffffffu, (int)(v >> 21) & 0x1fffff);
  s.t0 = __reduce_add_sync(0xffffffffu, (int)v & 0x1fffff);
  return s;
}
__device__ __forceinline__ double to_double(const WarpSum& s) {
  return fma((double)(((long long)s.t2 << 21) + s.t1), 2097152.0, (double)s.t0);
}


// d 2^e by its exponent field; scalbn only where the result leaves the normal range
__device__ __forceinline__ double scale2(double d, int e) {
  const int f = exp_field(d) + e;
  if (d == 0.0) return 0.0;
  if (f <= 0 || f >= 0x7ff) return scalbn(d, e);
  return __hiloint2double(__double2hiint(d) + (e << 20), __double2loint(d));
}

}  // namespace fx
}  // namespace dirac
