// 64-bit fixed-point arithmetic of the residual's tensor contractions.
//
// Why: the FP64 pipe of sm_103a retires about 2 fused multiply-adds per clock
// and SM, the integer pipe about 28 32x32+64-bit multiply-adds (both measured
// with independent chains at full occupancy).  A contraction with a constant
// 1-D table needs no floating point: with the inputs of one element and
// variable scaled to their largest exponent (|x| <= 2^60) and the table to
// |sum| <= 2^62, one multiply-add is three 32-bit wide products
//     x C = xh Ch 2^64 + (xh Cl + xl Ch) 2^32 + xl Cl,
// the last of which stays below the result's unit.  A result is off by about
// one unit of 2^-60 of its bound per contraction, where FP64 rounds every
// term to 2^-53 of itself.
//
// A value is x 2^se: x the 64-bit integer, se an exponent shared by one
// (element, variable) plus the tables' own powers of two.  Infinities and NaN
// in the inputs mark the (element, variable) bad: everything converted back
// from it is NaN.
#pragma once
#include <algorithm>
#include <cstring>
#include "dg_internal.h"

// (compiled for the host too, where the tests compare it with exact integers)
#define DG_HD __host__ __device__ __forceinline__

namespace dg {

typedef long long i64;
typedef unsigned long long u64;

// Exponents below this (2^-783) count as this, so that smaller inputs become 0.
// The last conversion of M^-1 B^T W G has a scale of up to 3 x 59 + 60 powers of
// two less (every stage's input shifted up), which has to stay a normal
// double's: fix_to_double adds to the exponent field without a look at its range.
constexpr int FIX_EMIN = 240;
constexpr int FIX_EBAD = 2010;  // largest exponent held; from here on (2^987) the result is NaN

// 32 x 32 -> 64-bit product, to be accumulated with +=
DG_HD i64 mul_wide(int a, int b) {
#ifdef __CUDA_ARCH__
  i64 d;
  asm("mul.wide.s32 %0, %1, %2;" : "=l"(d) : "r"(a), "r"(b));
  return d;
#else
  return (i64)a * b;
#endif
}

// the words of a double
DG_HD int fix_hi(double v) {
#ifdef __CUDA_ARCH__
  return __double2hiint(v);
#else
  i64 b;
  std::memcpy(&b, &v, 8);
  return (int)(b >> 32);
#endif
}
DG_HD unsigned fix_lo(double v) {
#ifdef __CUDA_ARCH__
  return (unsigned)__double2loint(v);
#else
  i64 b;
  std::memcpy(&b, &v, 8);
  return (unsigned)b;
#endif
}

// half a unit of a product's result, in the middle accumulator: without it
// every contraction rounds down, and M^-1 turns the common half unit into the
// largest error of the residual
constexpr i64 FIX_HALF = 1ll << 29;

// x / 2^sh to the nearest, for any sh >= 0 and |x| < 2^61: from 62 on that is 0
// (and 2^63, twice the half unit to add at 63, is not an i64)
DG_HD i64 fix_shift(i64 x, int sh) {
  sh = std::min(sh, 62);
  return (x + ((1ll << sh) >> 1)) >> sh;
}

// biased exponent of a double (0x7ff for infinities and NaN)
DG_HD int fix_exp(double v) { return (fix_hi(v) >> 20) & 0x7ff; }

DG_HD void fix_split(i64 x, int& h, int& l) {
  l = (int)x;
  h = (int)(x >> 32) + (int)((unsigned)l >> 31);  // balanced halves: x = h 2^32 + l
}

// v as an integer below 2^nb for the largest biased exponent emax >= exponent(v)
DG_HD i64 to_fix(double v, int emax, int nb) {
  const int hi = fix_hi(v);
  const u64 m = ((u64)(unsigned)((hi & 0xfffff) | 0x100000) << 32) | fix_lo(v);
  const int d = std::min(emax - ((hi >> 20) & 0x7ff), 63);
  const i64 a = (i64)((m << (nb - 53)) >> d), s = (i64)(hi >> 31);
  return (a ^ s) - s;
}

// A positive factor rm 2^(er - 62), 2^61 <= rm < 2^62 (0: rm = 0)
struct FixMag {
  int h, l;  // balanced halves of rm
  int er;
};
// and one of either sign, kept apart: what is multiplied is a magnitude, cut
// off towards 0 on both sides (a negative rm would cut its products off towards
// -infinity and turn zeros into -1)
struct FixScale : FixMag {
  int sg;    // 0 or -1
};
DG_HD FixMag fix_mag(double r) {
  FixMag f;
  const int hi = fix_hi(r), E = (hi >> 20) & 0x7ff;
  i64 m = (i64)(((u64)(unsigned)((hi & 0xfffff) | 0x100000) << 32) | fix_lo(r)) << 9;
  if (E == 0) m = 0;
  fix_split(m, f.h, f.l);
  f.er = E == 0 ? -4000 : E - 1022;
  return f;
}
DG_HD FixScale fix_scale(double r) {
  FixScale f;
  static_cast<FixMag&>(f) = fix_mag(r);
  f.sg = fix_hi(r) >> 31;
  return f;
}
DG_HD int fix_sign(const FixMag&) { return 0; }
DG_HD int fix_sign(const FixScale& f) { return f.sg; }

// x rm / 2^62
DG_HD i64 fix_mul(i64 x, int rh, int rl) {
  int h, l;
  fix_split(x, h, l);
  const i64 mid = FIX_HALF + mul_wide(l, rh) + mul_wide(h, rl);
  return (mul_wide(h, rh) << 2) + (mid >> 30);
}

// v r as an integer below 2^nb (nb <= 60); emax >= exponent(v) + r.er
template <class R>
DG_HD i64 to_fix_mul(double v, const R& r, int emax, int nb) {
  const int hi = fix_hi(v);
  const u64 m = ((u64)(unsigned)((hi & 0xfffff) | 0x100000) << 32) | fix_lo(v);
  const int E = (hi >> 20) & 0x7ff;
  i64 a = fix_mul((i64)(m << 7), r.h, r.l);
  const int d = E == 0 ? 63 : std::min(emax - E - r.er + 60 - nb, 63);
  a >>= d;
  const i64 s = (i64)((hi >> 31) ^ fix_sign(r));
  return (a ^ s) - s;
}

// x 2^se rounded to the nearest double (|x| < 2^62); bad (0 or the high word of
// a NaN) is or-ed in
__device__ __forceinline__ double fix_to_double(i64 x, int se, int bad) {
  const i64 s = x >> 63;
  const u64 a = (u64)((x ^ s) - s);
  const int lz = __clzll((i64)a);
  // leading one at bit 62, the half below the 53rd bit added: bit 52 after the
  // shift is the leading one, which the exponent field below counts
  const u64 r = ((a << ((lz - 1) & 63)) + 0x200) >> 10;
  const int e = a ? (63 + 1022 + se - lz) << 20 : 0;
  const int hi = ((int)(r >> 32) + e) | ((int)(x >> 32) & 0x80000000) | bad;
  return __hiloint2double(hi, (int)r);
}

// shared exponent of a group of values whose largest biased exponent is e:
// the exponent used and, in *bad, the NaN mark
__device__ __forceinline__ int fix_emax(int e, int& bad) {
  bad = e >= FIX_EBAD ? 0x7ff80000 : 0;
  return max(min(e, FIX_EBAD), FIX_EMIN);
}

// one output of a contraction: sum_k x_k C_k / 2^(62 - S) (inputs as halves)
template <int K, int S = 0>
__device__ __forceinline__ i64 fix_dot(const int* xh, const int* xl, const int2* C) {
  i64 hi = 0, mid = FIX_HALF >> S;
#pragma unroll
  for (int k = 0; k < K; ++k) {
    hi += mul_wide(xh[k], C[k].x);
    mid += mul_wide(xh[k], C[k].y);
    mid += mul_wide(xl[k], C[k].x);
  }
  return (hi << (2 + S)) + (mid >> (30 - S));
}

// reads K values at stride `str` as halves
template <int K>
__device__ __forceinline__ void fix_line(const i64* p, int str, int* xh, int* xl) {
#pragma unroll
  for (int k = 0; k < K; ++k) fix_split(p[k * str], xh[k], xl[k]);
}

// The converged threads of a warp that share a key: max() raises a shared slot
// to the group's largest value with one atomic.
struct KeyGroup {
  unsigned mask;
  bool leader;
  __device__ __forceinline__ explicit KeyGroup(int key) {
    mask = __match_any_sync(__activemask(), key);
    leader = (threadIdx.x & 31) == __ffs(mask) - 1;
  }
  __device__ __forceinline__ void max(int* slot, int e) const {
    const int m = __reduce_max_sync(mask, e);
    if (leader) atomicMax(slot, m);
  }
};

}  // namespace dg
