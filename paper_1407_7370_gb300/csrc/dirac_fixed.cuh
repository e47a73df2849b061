// dirac_fixed.cuh -- 60-bit fixed-point arithmetic for the FP64 kernels.
//
// GB300 issues one FP64 instruction per warp and SM sub-partition every 64 to
// 76 cycles (measured: DFMA 64, DADD and DMUL 76, every conversion from or to
// FP64 64), while a 32 x 32 + 64 bit integer multiply-add (IMAD.WIDE), a
// 64-bit add or a 32-bit shift takes 2.  A product of two 60-bit numbers in
// two 30-bit limbs is three IMAD.WIDE, accumulated exactly over a whole row of
// the operator and rounded once at its end; converting a double by shifting
// its mantissa is about a dozen integer instructions.  So sums of products
// whose operands share a scale are several times cheaper here than on the
// FP64 pipe, at 5 to 9 bits more than FP64's 53 relative to the largest
// operand of the group that shares the scale.
#pragma once
#include <cuda_runtime.h>

namespace dirac {
namespace fx {

constexpr int LIMB = 30;

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

// v = hi 2^30 + lo, lo in [-2^29, 2^29): products that drop lo x lo stay unbiased
struct Limbs {
  int hi, lo;
};
__device__ __forceinline__ Limbs split(long long v) {
  Limbs l;
  l.hi = (int)((v + (1LL << (LIMB - 1))) >> LIMB);
  l.lo = (int)((unsigned)v - ((unsigned)l.hi << LIMB));
  return l;
}
__device__ __forceinline__ Limbs neg(const Limbs& a) { return Limbs{-a.hi, -a.lo}; }

// Sum of products in units of 2^60: h exactly, x in units of 2^30.  The sums
// wrap like unsigned numbers, so a sum of squares may use all 64 bits of h.
struct Acc {
  unsigned long long h = 0, x = 0;
  __device__ __forceinline__ void mac(const Limbs& a, const Limbs& b) {
    h += (unsigned long long)((long long)a.hi * b.hi);
    x += (unsigned long long)((long long)a.hi * b.lo);
    x += (unsigned long long)((long long)a.lo * b.hi);
  }
  __device__ __forceinline__ void sqr(const Limbs& a) {   // x holds half of the cross terms
    h += (unsigned long long)((long long)a.hi * a.hi);
    x += (unsigned long long)((long long)a.hi * a.lo);
  }
  __device__ __forceinline__ long long value() const {
    return (long long)h + ((long long)(x + (1ULL << (LIMB - 1))) >> LIMB);
  }
  // the sum / 2^s, rounded (s >= 1): signed products
  __device__ __forceinline__ long long value_shr(int s) const { return (value() + (1LL << (s - 1))) >> s; }
  // the same for squares (not negative, up to 2^64)
  __device__ __forceinline__ long long value_sqr_shr(int s) const {
    const unsigned long long v = h + (unsigned long long)((long long)(x + (1ULL << (LIMB - 2))) >> (LIMB - 1));
    return (long long)((v >> s) + ((v >> (s - 1)) & 1));
  }
};

// v / 2^s, rounded (s >= 0)
__device__ __forceinline__ long long shr_round(long long v, int s) {
  if (s <= 0) return v;
  if (s > 62) return 0;
  return (v + (1LL << (s - 1))) >> s;
}

// Running sum of terms whose scale changes from tile to tile (the same for all
// threads of a warp): v in units of 2^e.  Terms of magnitude below 2^58 may be
// added 32 times between two flushes.
struct Run {
  long long v = 0;
  int e = -100000;
  __device__ __forceinline__ void add(long long t, int te) {
    if (te > e) {
      v = shr_round(v, te - e);
      e = te;
    } else {
      t = shr_round(t, e - te);
    }
    v += t;
  }
  // the sum over a warp, as a double in every lane; starts again from zero.
  // The 32 terms are added exactly, in three pieces of 21 bits.
  __device__ __forceinline__ double flush() {
    const int p2 = __reduce_add_sync(0xffffffffu, (int)(v >> 42));
    const int p1 = __reduce_add_sync(0xffffffffu, (int)(v >> 21) & 0x1fffff);
    const int p0 = __reduce_add_sync(0xffffffffu, (int)v & 0x1fffff);
    const double d = scalbn(fma((double)(((long long)p2 << 21) + p1), 2097152.0, (double)p0), e);
    v = 0;
    e = -100000;
    return d;
  }
};

}  // namespace fx
}  // namespace dirac
