// Block fixed-point form of FP64 vectors, and exact products in it.
//
// sm_103a executes 2 FP64 lanes per clock and SM (every DADD, DMUL, DFMA and
// conversion to or from double: 1.9 measured), but 62 lanes of IMAD.WIDE
// (32 x 32 + 64 bits).  Sums of products over FP64 vectors are therefore made
// in integers: a tile of FX_TILE consecutive points shares one binary
// exponent E (the largest of its real and imaginary parts), a value is the
// integer v = x 2^(FX_TOP + 1023 - E) rounded to nearest, |v| <= 2^54, held as
// two limbs v = hi 2^27 + lo.  A value within a factor 2 of the tile's largest
// keeps all 53 bits; a smaller one is exact to 2^-54 of the tile's largest,
// half an ulp of that value.  The limb products hi hi and hi lo are exact and
// are added exactly in 64 bits; lo lo, at most 2^-55 of the largest product
// and of mean zero, is left out (one factor's lo is symmetric about zero).
#pragma once
#include "hz_internal.h"

namespace hz {

constexpr int FX_TILE = HZ_FX_TILE;  // points that share one exponent
constexpr int FX_TOP = 53;           // bit of the leading one of a value with exponent E

__device__ __forceinline__ int fx_exp(double x) { return (__double2hiint(x) >> 20) & 0x7ff; }
__device__ __forceinline__ int fx_exp(double2 z) { return max(fx_exp(z.x), fx_exp(z.y)); }

// the smallest E that tiles use: zeros and subnormals then shift out
constexpr int FX_EMIN = 64;

// x 2^(FX_TOP + 1023 - E) to the nearest integer, E >= exponent of x and
// E >= FX_EMIN; integer operations only.  Subnormals count as zero.
__device__ __forceinline__ long long fx_from(double x, int E) {
  const int hi = __double2hiint(x);
  const unsigned lo = unsigned(__double2loint(x));
  const int sh = E - ((hi >> 20) & 0x7ff);
  const unsigned mh = unsigned((hi & 0xfffff) | 0x100000);
  unsigned long long t = static_cast<unsigned long long>(__funnelshift_l(lo, mh, 2)) << 32 | (lo << 2);
  asm("shr.u64 %0, %0, %1;" : "+l"(t) : "r"(sh));  // zero past 63
  const long long v = static_cast<long long>((t + 1) >> 1);
  const long long sg = hi >> 31;
  return (v ^ sg) - sg;
}

// limbs of v: with lo symmetric, |lo| <= 2^26, |hi| <= 2^27
__device__ __forceinline__ int fx_lo(long long v) { return int(unsigned(v) << 5) >> 5; }
__device__ __forceinline__ int fx_hi(long long v) { return int((v + (1ll << 26)) >> 27); }
// a complex value as (re hi, re lo, im hi, im lo)
__device__ __forceinline__ int4 fx_pack(double2 z, int E) {
  const long long a = fx_from(z.x, E), b = fx_from(z.y, E);
  return make_int4(fx_hi(a), fx_lo(a), fx_hi(b), fx_lo(b));
}
// the same with 0 <= lo < 2^27 (the other factor's lo is symmetric)
__device__ __forceinline__ int4 fx_pack_floor(double2 z, int E) {
  const long long a = fx_from(z.x, E), b = fx_from(z.y, E);
  return make_int4(int(a >> 27), int(unsigned(a) & 0x7ffffffu), int(b >> 27),
                   int(unsigned(b) & 0x7ffffffu));
}

__device__ __forceinline__ long long mad_w(int a, int b, long long c) {
  return static_cast<long long>(a) * b + c;
}

// hh 2^54 + x 2^27 in units of 2^54, rounded to nearest
__device__ __forceinline__ long long fx_sum(long long hh, long long x) {
  return hh + ((x + (1ll << 26)) >> 27);
}
// fx_to's k for fx_sum of products of values whose (biased) exponents add up
// to E
__device__ __forceinline__ int fx_unit(int E) { return E + 54 - 2 * FX_TOP - 2 * 1023; }

// t 2^k: zero below the normal range; above it (the operator's tiles keep
// clear of it) a wrong value
__device__ __forceinline__ double fx_to(long long t, int k) {
  const double d = static_cast<double>(t);
  const int hi = __double2hiint(d);
  const int e = ((hi >> 20) & 0x7ff) + k;
  return (t == 0 || e <= 0) ? 0.0 : __hiloint2double(hi + (k << 20), __double2loint(d));
}
// the same with infinity above the range
__device__ __forceinline__ double double_of(long long t, int k) {
  const double d = static_cast<double>(t);
  const int hi = __double2hiint(d);
  const int e = ((hi >> 20) & 0x7ff) + k;
  double r = __hiloint2double(hi + (k << 20), __double2loint(d));
  if (e >= 0x7ff) r = __hiloint2double((hi & 0x80000000) | 0x7ff00000, 0);
  return (t == 0 || e <= 0) ? 0.0 : r;
}

// Infinities and NaN have no integer form: a tile that holds one has exponent
// FX_INF, and sums over it are NaN.
constexpr int FX_INF = 0x7ff;
constexpr int FX_BAD = 1 << 14;  // above any sum of two exponents
__device__ __forceinline__ int fx_exp_sum(int e, int f) { return max(e, f) >= FX_INF ? FX_BAD : e + f; }
__device__ __forceinline__ double fx_nan() { return __longlong_as_double(0x7ff8000000000000ll); }

}  // namespace hz
