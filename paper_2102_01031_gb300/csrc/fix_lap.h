// fix_lap.h -- the sum of six neighbours minus six times the site (dx^2 times the
// seven-point Laplacian) of FP64 values in 64-bit integers; host and device code, shared
// with a CPU check.
//
// An FP64 operation holds a warp's quarter of an SM for 64 cycles on this part, an integer
// one for two on a unit of its own.  The passes with FP64 storage are bound by their FP64
// operations; this takes the Laplacian's six a field and site off them.
//
// Each value's 53-bit mantissa is shifted to the largest exponent of the seven with six
// bits below that value's own last one and summed exactly; the sum is rounded once, to the
// nearest FP64 value.  Values with smaller exponents lose what lies below those six bits
// (towards minus infinity; negative values are kept as their complement, one unit of those
// bits low): at most 12 x 2^-58 of the largest value's power of two, where the FP64 form
// rounds five sums and a fused multiply-add at 2^-53 of their own sizes (up to six times the
// largest value).  A site and six neighbours of one value give 0, as in FP64.
// Infinities, NaN and the two ends of the exponent range take the FP64 form.
#pragma once

#include "fix_fft.h"

namespace clg {

// Exponents (of the largest of the seven values, as stored) whose sums neither overflow nor
// reach the subnormal range.
constexpr uint32_t kFixLapMin = 70, kFixLapMax = 0x7f9;

// A value's mantissa with its leading bit at bit 62 (a subnormal's or a zero's leading bit
// counts as set: below every bit that is kept, as the largest exponent is at least
// kFixLapMin), its sign as a mask and its exponent field in place.
struct FixVal {
  uint64_t m;
  int64_t s;
  uint32_t e;
};
FX FixVal fix_val(double x) {
  const uint64_t b = bits_of(x);
  const uint32_t h = (uint32_t)(b >> 32);
  return FixVal{((b << 10) & 0x3fffffffffffffffull) | 0x4000000000000000ull, (int64_t)((int32_t)h >> 31), h & 0x7ff00000u};
}
// the value in units of 2^-58 of 2^(largest exponent e)
FX uint64_t fix_aligned(const FixVal& v, uint32_t e4) {
  const uint32_t n = (e4 - v.e) >> 20;
  return (v.m >> (n < 63u ? n : 63u)) ^ (uint64_t)v.s;
}
FX uint32_t fix_max(uint32_t a, uint32_t b) { return a > b ? a : b; }

FX double fix_lap(const FixVal& xl, const FixVal& xr, const FixVal& yl, const FixVal& yh, const FixVal& zl,
                  const FixVal& zh, const FixVal& c, bool* in_range) {
  const uint32_t e = fix_max(fix_max(fix_max(xl.e, xr.e), fix_max(yl.e, yh.e)), fix_max(fix_max(zl.e, zh.e), c.e));
  *in_range = e - (kFixLapMin << 20) <= ((kFixLapMax - kFixLapMin) << 20);
  const uint32_t e4 = e + (4u << 20);
  const uint64_t c1 = fix_aligned(c, e4);
  const uint64_t S = fix_aligned(xl, e4) + fix_aligned(xr, e4) + fix_aligned(yl, e4) + fix_aligned(yh, e4) +
                     fix_aligned(zl, e4) + fix_aligned(zh, e4) - (c1 << 2) - (c1 << 1);
  const uint64_t neg = (uint64_t)((int64_t)S >> 63), a = (S ^ neg) - neg;
  const int lz = leading_zeros(a | 1u);
  const uint64_t t = a << lz;
  // 53 bits, the leading one counted into the exponent; a carry out of them raises it
  const uint64_t r = ((uint64_t)(e + ((uint32_t)(4 - lz) << 20)) << 32) + (t >> 11) + ((t >> 10) & 1u);
  return a == 0 ? 0.0 : double_of(r | (neg << 63));
}

// The FP64 form: the six neighbours summed, then -6 c in one fused multiply-add.
FX double fp64_lap(double xl, double xr, double yl, double yh, double zl, double zh, double c) {
  return fma(-6.0, c, ((xl + xr) + (yl + yh)) + (zl + zh));
}

}  // namespace clg
