// Fixed-point arithmetic on the integer pipes (the arithmetic of the FP64 operators).
//
// GB300 issues 32 IMAD.WIDE (32 x 32 + 64 bits) per clock and SM but only 2 FP64
// FMAs (measured: 28.5 and 1.6 per clock and SM in a register-only loop), so a product
// of two 64-bit numbers in two limbs, three IMAD.WIDE, is five times cheaper than an
// FP64 FMA.
//
// A group of numbers (the nodal values of one cell and vector) shares a power-of-two
// unit taken from its largest magnitude: value = X unit, |X| <= 2^59 (FX_F).  A
// coefficient |c| <= 1/2 of a table is C = round(c 2^64), and
//   X C 2^-64 = xh ch + (xh cl + xl ch) 2^-32 + xl cl 2^-64     (x = xh 2^32 + xl, xl signed)
// is accumulated as two exact 64-bit sums, hh and mm; only xl cl 2^-64 (at most a
// quarter of a unit of the result) is dropped, and one rounding per sum follows:
// Y = hh + round(mm 2^-32).  Limbs of 32 bits make the low limb a register of X and the
// second term a register of mm.  Against an FP64 FMA chain, which rounds every partial
// sum to 2^-53 of its size, a sum is exact to about one unit in 2^59 of the largest
// magnitude that its scales allow for.
//
// Overflow: the magnitudes of each row of a table sum to at most 1; in even/odd halves that is
// a sum of at most 1/2 on halves of at most 2^60, so a table's results are at most 2^59 where
// |X| <= 2^59, and a sum of several tables that is contracted again is scaled to that as a whole.
// With |xh| <= 2^28, sum |ch| <= 2^31 and |cl|, |xl| <= 2^31 the products of one table leave
// |hh| <= 2^59 and, for up to K = 5 of them, |mm| <= K 2^59 + 2^62 < 2^63; mm is folded into hh before
// the next table.
#pragma once

#include <cuda_runtime.h>

#include <cmath>
#include <cstdint>

namespace pawfe {

constexpr int FX_F = 59;                       // bits of a number
constexpr long long FX_HALF = 1ll << 31;       // half a unit of mm 2^-32
constexpr int FX_NONE = -100000;               // exponent of a zero coefficient
constexpr int FX_BAD = 100000;                 // exponent that marks non-finite numbers
// unit of a group whose largest exponent field is E: 2^(E - FX_BIAS)
constexpr int FX_BIAS = 1022 + FX_F;

// coefficient (h 2^32 + l) 2^-64, l signed
struct fx2 {
  int h, l;
};

// smallest s with |c| < 2^s (FX_NONE for 0)
inline int fx_scale(double c) {
  if (c == 0.0) return FX_NONE;
  int e;
  std::frexp(c, &e);
  return e;
}

// |c| < 1/2 as two limbs; in long double, so that the factors of a table keep 64 bits
inline fx2 fx_coef(long double c) {
  const long long C = std::llrint(std::ldexp(c, 64));
  return {(int)((C + FX_HALF) >> 32), (int)C};
}

#ifdef __CUDACC__
// exponent field of x as used for the common unit (zero and subnormal numbers: 1)
__device__ __forceinline__ int fx_field(double x) {
  return max((int)((unsigned)__double2hiint(x) >> 20) & 0x7ff, 1);
}

// the field that a coefficient counts with in the scale of its group: that of |x| with the carry of
// the low limb's rounding, so that fx_from<63> in the scale leaves a high limb below 2^31
__device__ __forceinline__ int fx_field_coef(double x) {
  const long long b = __double_as_longlong(x) & 0x7fffffffffffffffll;
  return max((int)((b + (1ll << 21)) >> 52), 1);
}

// x in the unit of a group with the largest exponent field E (E >= fx_field(x), finite), truncated;
// |x| < 2^(E - 1022) becomes an integer below 2^BITS (54 <= BITS <= 63)
template <int BITS = FX_F>
__device__ __forceinline__ long long fx_from(double x, int E) {
  const unsigned hi = (unsigned)__double2hiint(x), lo = (unsigned)__double2loint(x);
  const int f = (int)(hi >> 20) & 0x7ff;
  const unsigned mh = (hi & 0xfffffu) | (f ? 0x100000u : 0u);
  const unsigned long long m = ((unsigned long long)mh << 32 | lo) << (BITS - 53);
  const long long t = (long long)(m >> min(E - max(f, 1), 63));
  return (int)hi < 0 ? -t : t;
}

// the same rounded to nearest (ties away from zero), |result| <= 2^BITS (53 <= BITS <= 61)
template <int BITS>
__device__ __forceinline__ long long fx_round(double x, int E) {
  const unsigned hi = (unsigned)__double2hiint(x), lo = (unsigned)__double2loint(x);
  const int f = (int)(hi >> 20) & 0x7ff;
  const unsigned mh = (hi & 0xfffffu) | (f ? 0x100000u : 0u);
  const unsigned long long m = ((unsigned long long)mh << 32 | lo) << (BITS - 52);
  const long long t = (long long)(((m >> min(E - max(f, 1), 63)) + 1) >> 1);
  return (int)hi < 0 ? -t : t;
}

// fx_field and fx_from for FP32 numbers (fields of the equal FP64 numbers)
__device__ __forceinline__ int fx_field(float x) {
  const int f = (int)(__float_as_uint(x) >> 23) & 0xff;
  return f == 0xff ? 0x7ff : max(f, 1) + 896;
}
template <int BITS = FX_F>
__device__ __forceinline__ long long fx_from(float x, int E) {
  const unsigned b = __float_as_uint(x);
  const int f = (int)(b >> 23) & 0xff;
  const unsigned long long m = (unsigned long long)((b & 0x7fffffu) | (f ? 0x800000u : 0u)) << (BITS - 24);
  const long long t = (long long)(m >> min(E - (max(f, 1) + 896), 63));
  return (int)b < 0 ? -t : t;
}

// Y 2^e as a double (any Y and e)
static __device__ __noinline__ double fx_to_any(long long Y, int e) {
  if (Y == 0) return 0.0;
  const unsigned long long a = (unsigned long long)(Y < 0 ? -Y : Y);
  const int n = __clzll((long long)a);
  const double r = scalbn((double)(a << n), max(min(e - n, 3000), -3000));
  return Y < 0 ? -r : r;
}

// (ah 2^32 + al) 2^e with the sign bit of hi, ah != 0, f = the exponent field less one in 0 .. 2044
__device__ __forceinline__ double fx_pack(unsigned ah, unsigned al, int n, int f, unsigned hi) {
  const unsigned mh = __funnelshift_l(al, ah, n), ml = al << n;   // bit 63 set
  // 53 bits and the rounding bit; a carry moves into the exponent
  const unsigned long long q = ((unsigned long long)(mh >> 11) << 32 | __funnelshift_r(ml, mh, 11)) + ((ml >> 10) & 1u);
  const unsigned s = (hi & 0x80000000u) + ((unsigned)f << 20);
  return __longlong_as_double((long long)(q + ((unsigned long long)s << 32)));
}

// Y 2^e as a double, rounded to nearest (ties away from zero); fast for |Y| >= 2^32
__device__ __forceinline__ double fx_to(long long Y, int e) {
  const unsigned long long a = (unsigned long long)(Y < 0 ? -Y : Y);
  const unsigned ah = (unsigned)(a >> 32), al = (unsigned)a;
  const int n = __clz((int)ah), f = 1023 + 62 - n + e;
  if (ah == 0 || (unsigned)f >= 2045u) return fx_to_any(Y, e);
  return fx_pack(ah, al, n, f, (unsigned)(Y >> 32));
}

// the same, fast for small Y too
__device__ __forceinline__ double fx_to_small(long long Y, int e0) {
  int e = e0;
  const unsigned long long a = (unsigned long long)(Y < 0 ? -Y : Y);
  unsigned ah = (unsigned)(a >> 32), al = (unsigned)a;
  if (ah == 0) {
    ah = al;
    al = 0;
    e -= 32;
  }
  const int n = __clz((int)ah), f = 1023 + 62 - n + e;
  if (ah == 0) return 0.0;
  if ((unsigned)f >= 2045u) return fx_to_any(Y, e0);
  return fx_pack(ah, al, n, f, (unsigned)(Y >> 32));
}

// limbs: X = fx_hi 2^32 + fx_lo with a signed low limb
__device__ __forceinline__ int fx_lo(long long X) { return (int)X; }
__device__ __forceinline__ int fx_hi(long long X) { return (int)(X >> 32) + (int)((unsigned)X >> 31); }

// s += a b in one instruction: as a sum of products in C++ the compiler reorders the additions of a
// line, and from mad.wide it multiplies and adds separately (142k instead of 222k instructions per
// cell and vector of the local operator at degree 6)
__device__ __forceinline__ void fx_mad(long long &s, int a, int b) {
  asm("{ .reg .s64 t; mul.wide.s32 t, %1, %2; add.s64 %0, %0, t; }" : "+l"(s) : "r"(a), "r"(b));
}

// (hh, mm) += x c
__device__ __forceinline__ void fx_mac(long long &hh, long long &mm, int xh, int xl, const fx2 &c) {
  fx_mad(hh, xh, c.h);
  fx_mad(mm, xh, c.l);
  fx_mad(mm, xl, c.h);
}

// the sum of a pair of accumulators (mm started from FX_HALF)
__device__ __forceinline__ long long fx_sum(long long hh, long long mm) { return hh + (mm >> 32); }
#endif

}  // namespace pawfe
