// Fixed-point arithmetic in two limbs on the integer pipes, for the per-row work of the f64 tensor-core
// path.
//
// GB300 retires one FP64 warp instruction per 17 SM clocks (68 per SM sub-partition, measured) and one
// 32 x 32 + 64-bit integer multiply-add per 2.4 sub-partition clocks.  A sum of products
//   sum_i a_i b_i,  a = ah 2^L + al,  b = bh 2^L + bl  (al, bl in [-2^(L-1), 2^(L-1))),
// needs no carries when its two leading limb products are summed apart,
//   hi += ah bh,  mid += ah bl + al bh,  sum = hi 2^2L + mid 2^L + (al bl, dropped: at most 2^2L / 4 a term),
// three multiply-adds a term, a ninth of the one FP64 instruction it replaces.  The low limbs are signed and the
// conversions round to nearest so that errors have no common sign: with low limbs from 0 up every dropped product
// was positive, and with the rows kernel's floor that moved the virial, a sum over all rows, by 3.4e-15 of its
// largest element (648 atoms of water; now 3e-16).  The values are fixed
// points against a power of two that bounds them (the largest of a batch of rows; a row of the table times
// a column of dE/dT), with 56 to 61 places below it: each term's error lies below that of an f64 product
// of the bound's size.
#pragma once

#include <cuda_runtime.h>

#include <cstdint>

namespace dpc {
namespace {
namespace fx {

// v = hi 2^L + lo, -2^(L-1) <= lo < 2^(L-1), |v| < 2^(31 + L) - 2^(L-1)
struct Fix {
  int lo, hi;
};
template <int L>
__device__ __forceinline__ Fix limbs(long long v) {
  const int hi = (int)((v + (1ll << (L - 1))) >> L);
  return Fix{(int)((unsigned)v - ((unsigned)hi << L)), hi};
}
// c + a b.  As PTX: where the compiler knows that a limb is not negative it widens it by zeros and, the
// other limb being signed, multiplies 64 by 64 bits (measured: 1290 instead of 600 instructions a row).
__device__ __forceinline__ long long mad_wide(int a, int b, long long c) {
  asm("mad.wide.s32 %0, %1, %2, %0;" : "+l"(c) : "r"(a), "r"(b));
  return c;
}

template <int L>
__device__ __forceinline__ long long whole(const Fix f) {
  return mad_wide(f.hi, 1 << L, f.lo);
}

// A sum of products of fixed points: hi 2^2L + mid 2^L.  The caller's bounds keep both below 2^63.
struct Acc {
  long long hi = 0, mid = 0;
  __device__ __forceinline__ void mad(const Fix a, const Fix b) {
    hi = mad_wide(a.hi, b.hi, hi);
    mid = mad_wide(a.hi, b.lo, mid);
    mid = mad_wide(a.lo, b.hi, mid);
  }
};
// The sum over 2^2L to the nearest integer but for the dropped limb products (each at most a quarter); a sum
// of zeros is zero.
template <int L>
__device__ __forceinline__ long long over_unit(const Acc &p) {
  return p.hi + ((p.mid + (1ll << (L - 1))) >> L);
}

// a b / 2^2L as limbs: the product of a fixed point in units of 2^-2L with any other.
template <int L>
__device__ __forceinline__ long long mul(const Fix a, const Fix b) {
  Acc p;
  p.mad(a, b);
  return over_unit<L>(p);
}

// x 2^sh to the nearest integer, |x 2^sh| < 2^62 and 0 <= sh < 900, so that a zero or subnormal x still gives
// zero: the exponent moved by an integer add, one conversion on the FP64 pipe (64 sub-partition clocks that the
// integer pipes do not wait for; by integer shifts it takes them 41, measured).  A negative shift would carry a
// zero's exponent field into its sign.
__device__ __forceinline__ long long from_double(double x, int sh) {
  return __double2ll_rn(__hiloint2double(__double2hiint(x) + (sh << 20), __double2loint(x)));
}

// The same for any shift: zero where the exponent would fall below the normal range.
__device__ __forceinline__ long long from_double_any(double x, int sh) {
  const int e = ((__double2hiint(x) >> 20) & 0x7ff) + sh;
  return e > 0 ? from_double(x, sh) : 0ll;
}

// v 2^e rounded to the nearest double, for e and |v| that keep it normal (|e| <= kSafeExp): one conversion
// on the FP64 pipe.  (By 32-bit integer operations it takes the integer pipes 28 clocks; measured slower in
// every kernel here, whose FP64 pipe is idle more than a third of the time.)
constexpr int kSafeExp = 900;
__device__ __forceinline__ double to_double(long long v, int e) {
  const double d = (double)v;
  return v ? __hiloint2double(__double2hiint(d) + (e << 20), __double2loint(d)) : 0.0;
}

}  // namespace fx
}  // namespace
}  // namespace dpc
