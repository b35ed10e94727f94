// fix_fft.h -- the arithmetic of the 1-D transforms (ic_fft.cu): 64-bit fixed point with
// one exponent per line (block floating point); host and device code, shared with a CPU
// check.  Arrays in memory stay FP64 (or the storage precision).
//
// An FP64 operation holds a warp's quarter of an SM for 64 cycles on this part, a 64-bit
// integer addition for about four, so butterflies in FP64 were what the transforms spent
// their time on (28 operations per point and axis; 256^3: 577 us for the row pairs, 994 us
// for the other two axes).  A line is scaled so that the sum of its components' sizes
// lies just below 2^62: every intermediate value of a transform is a sum of the line's
// values times factors of modulus 1, so none can overflow; sums are exact, and only the
// input's last bits and the products with the roots of unity (62 bits of fraction) round, each
// to about half a unit (FP64 rounds every sum and product at 2^-53 of its own size).  Against
// extended precision the transform's error is at most FP64's (or one unit in the last place of
// its FP64 result) over all lattice sizes and inputs from white noise to a single mode and to
// lines of a few spikes (tests/fix_fft_check.cpp).
// A line with an infinity or a NaN is NaN throughout.
//
// Measured at 256^3 from an FP32 field, before and after: row pairs 577 -> 185 us, the other two
// axes 994 -> 333 us; with the axes of a spectrum kept in fixed point 170 and 325 us (1640 to
// 2000 instructions per 4 elements, issue-bound; memory alone takes 30 and 40 us an axis).
#pragma once

#include <limits.h>
#include <math.h>
#include <stdint.h>
#include <string.h>

#if defined(__CUDACC__)
#define FX __host__ __device__ __forceinline__
#else
#define FX inline
#endif

namespace clg {

typedef long long fix;
struct alignas(16) CFix {
  fix x, y;
};

FX uint64_t bits_of(double v) {
  uint64_t b;
  memcpy(&b, &v, 8);
  return b;
}
FX uint32_t bits_of(float v) {
  uint32_t b;
  memcpy(&b, &v, 4);
  return b;
}
FX double double_of(uint64_t b) {
  double v;
  memcpy(&v, &b, 8);
  return v;
}
FX int leading_zeros(uint64_t v) {
#if defined(__CUDA_ARCH__)
  return __clzll((long long)v);
#else
  return __builtin_clzll(v);
#endif
}

// A component c of a root of unity times 2^62 as hi 2^32 + lo, both words signed (and
// lo > -2^31, so that it can be negated).
FX void root_words(double c, int& hi, int& lo) {
  const fix v = (fix)rint(c * 4611686018427387904.0);
  lo = (int)(uint32_t)(uint64_t)v;
  if (lo == INT_MIN) lo += 1;
  hi = (int)((v - lo) >> 32);
}

// The two signed words of a value, v = hi 2^32 + lo (|v| < 2^63 - 2^31).
FX void split(fix v, int& hi, int& lo) {
  lo = (int)(uint32_t)(uint64_t)v;
  hi = (int)(v >> 32) + (int)((uint32_t)lo >> 31);
}
// a (c + i s) for a root of unity given by its words (ch, cl), (sh, sl), to the nearest
// unit but for the product of the low words (half a unit rms).  Every sum below stays
// under 2^63 for |a| <= 2^62.
FX CFix cmul(const CFix& a, int ch, int cl, int sh, int sl) {
  int xh, xl, yh, yl;
  split(a.x, xh, xl);
  split(a.y, yh, yl);
  const int nsh = -sh, nsl = -sl;
  const fix half = 1ll << 29;
  const fix mr = half + (fix)xh * cl + (fix)xl * ch + (fix)yh * nsl + (fix)yl * nsh;
  const fix mi = half + (fix)xh * sl + (fix)xl * sh + (fix)yh * cl + (fix)yl * ch;
  const fix hr = (fix)xh * ch + (fix)yh * nsh, hi = (fix)xh * sh + (fix)yh * ch;
  CFix r;
  r.x = 4 * hr + (mr >> 30);
  r.y = 4 * hi + (mi >> 30);
  return r;
}
FX CFix cadd(const CFix& a, const CFix& b) {
  CFix r;
  r.x = a.x + b.x;
  r.y = a.y + b.y;
  return r;
}
FX CFix csub(const CFix& a, const CFix& b) {
  CFix r;
  r.x = a.x - b.x;
  r.y = a.y - b.y;
  return r;
}
// v sqrt(3)/2
FX fix mul_half_sqrt3(fix v) {
  const fix S3 = 3993837246235628775ll;  // sqrt(3) 2^61
  const int lo = (int)(uint32_t)(uint64_t)S3, hi = (int)((S3 - lo) >> 32);
  int vh, vl;
  split(v, vh, vl);
  const fix m = (1ll << 29) + (fix)vh * lo + (fix)vl * hi;
  return 4 * ((fix)vh * hi) + (m >> 30);
}

// v_q <- sum_r v_r exp(sign 2 pi i r q / R) in place, R = 2, 3 or 4.
template <int R>
FX void butterfly(CFix (&v)[R], int sign) {
  if (R == 2) {
    const CFix a = v[0], b = v[1];
    v[0] = cadd(a, b);
    v[1] = csub(a, b);
  } else if (R == 4) {
    const CFix t0 = cadd(v[0], v[R / 2]), t1 = csub(v[0], v[R / 2]);
    const CFix t2 = cadd(v[1], v[R - 1]), d = csub(v[1], v[R - 1]);
    CFix t3;  // (sign i)(v1 - v3)
    t3.x = sign > 0 ? -d.y : d.y;
    t3.y = sign > 0 ? d.x : -d.x;
    v[0] = cadd(t0, t2);
    v[1] = cadd(t1, t3);
    v[R / 2] = csub(t0, t2);
    v[R - 1] = csub(t1, t3);
  } else {  // R = 3: w = (-1/2, sign sqrt3/2)
    const CFix s = cadd(v[1], v[R - 1]), d = csub(v[1], v[R - 1]);
    CFix m, h;
    m.x = (2 * v[0].x - s.x) >> 1;
    m.y = (2 * v[0].y - s.y) >> 1;
    h.x = mul_half_sqrt3(sign > 0 ? -d.y : d.y);
    h.y = mul_half_sqrt3(sign > 0 ? d.x : -d.x);
    v[0] = cadd(v[0], s);
    v[1] = cadd(m, h);
    v[R - 1] = csub(m, h);
  }
}

// Storage to fixed point and back.  These run once per value beside a few operations
// per stage, so they are kept to 32-bit operations and single shifts.  A value's `top` is
// its high word without the sign; a line's exponent E is that of the largest top (1 for
// zeros and subnormals), ETOP that of infinities and NaN.
template <typename T> struct FixIO;
template <> struct FixIO<double> {
  static constexpr int MANT = 53, ETOP = 0x7ff, BIAS = 1075, EBIT = 20;
  FX static uint32_t word(double v) { return (uint32_t)(bits_of(v) >> 32); }
  FX static fix mant(double v) {  // exact
    const uint64_t b = bits_of(v);
    return (fix)((b & 0xfffffffffffffull) | ((b & 0x7ff0000000000000ull) ? 0x10000000000000ull : 0ull));
  }
  FX static uint64_t mant63(double v) {  // mantissa of a normal value with 10 bits below it
    return ((bits_of(v) & 0xfffffffffffffull) | 0x10000000000000ull) << 10;
  }
};
template <> struct FixIO<float> {
  static constexpr int MANT = 24, ETOP = 0xff, BIAS = 150, EBIT = 23;
  FX static uint32_t word(float v) { return bits_of(v); }
  FX static fix mant(float v) {
    const uint32_t b = bits_of(v);
    return (fix)((b & 0x7fffffu) | ((b & 0x7f800000u) ? 0x800000u : 0u));
  }
  FX static uint64_t mant63(float v) { return (uint64_t)((bits_of(v) & 0x7fffffu) | 0x800000u) << 39; }
};
FX int imax(int a, int b) { return a > b ? a : b; }
FX int imin(int a, int b) { return a < b ? a : b; }
template <typename T>
FX int top_of(T v) {
  return (int)(FixIO<T>::word(v) & 0x7fffffffu);
}
template <typename T>
FX int expo_of(int top) {
  return imax(top >> FixIO<T>::EBIT, 1);
}
// |v| in units of 2^(E - BIAS + MANT - 20) rounded up, at most 2^20 + 1: a line's sum of these over all components bounds every value its transform
// can take.  (A zero counts as the smallest normal: an upper bound is all that is needed.)
template <typename T>
FX int size_of(T v, int E) {
  const int top = top_of(v), e = expo_of<T>(top);
  const uint32_t m = ((uint32_t)top & ((1u << FixIO<T>::EBIT) - 1u)) | (1u << FixIO<T>::EBIT);
  return (int)((m >> (FixIO<T>::EBIT - 19)) >> imin(E - e, 31)) + 2;
}
// What a line's values are scaled by, given that sum: values are held in units of
// 2^(E - BIAS - up) with sum |components| 2^up < 2^62.
struct LineScale {
  int E, up;
  bool plain;  // exponents far from both ends of the formats: no subnormals, no overflow
};
template <typename T>
FX LineScale line_scale(int E, int sum) {
  LineScale s;
  s.E = E;
  s.up = 62 - (FixIO<T>::MANT - 20) - (64 - leading_zeros((uint64_t)(unsigned)imax(sum, 1)));
  // FP64: zeros and subnormals taken as normal values vanish in the shift, results stay normal
  s.plain = sizeof(T) == 8 ? (E > 200 && E < 1900) : E > 100;
  return s;
}
template <typename T>
FX fix to_fix(T v, const LineScale& s) {
  const int top = top_of(v), e = expo_of<T>(top);
  const fix neg = -(fix)(FixIO<T>::word(v) >> 31);  // 0 or -1
  uint64_t m;
  if (s.plain) {
    // mantissa at bit 62, shifted right (rounded) to its place; FP64 zeros: the shift takes
    // the implied 1 away as well (E > 200), FP32's E > 100
    const int rs = 62 - (FixIO<T>::MANT - 1) - s.up + (s.E - e);
    m = ((FixIO<T>::mant63(v) >> imin(rs - 1, 63)) + 1) >> 1;
    if (sizeof(T) == 4 && top == 0) m = 0;
  } else {
    const int sh = s.up - (s.E - e);
    m = (uint64_t)FixIO<T>::mant(v);
    if (sh >= 0) m <<= sh;
    else m = sh < -62 ? 0 : (m + (1ull << (-sh - 1))) >> -sh;
  }
  return ((fix)m ^ neg) - neg;
}
// v 2^q rounded to FP64; plain: the result is zero or normal (ties away from zero), else
// any (ties away; below the normal range its last bits are cut off, above it an infinity)
FX double from_fix(fix v, int q, bool plain) {
  const fix neg = v >> 63;
  const uint64_t a = (uint64_t)((v ^ neg) - neg);  // < 2^63
  const int lz = a ? leading_zeros(a) : 64;
  uint64_t m = a << ((lz - 1) & 63);     // leading 1 at bit 62
  int e = 63 - lz + q + 1023;            // its biased exponent
  const uint64_t sgn = (uint64_t)neg << 63;
  if (!plain) {
    if (a == 0) return 0.0;
    if (e <= 0) {
      const int d = 1 - e;
      return double_of(sgn | ((d > 62 ? 0ull : m >> d) >> 10));
    }
    if (e >= 0x7ff) return double_of(sgn | 0x7ff0000000000000ull);
  }
  // rounded, the leading 1 at bit 52 (a carry runs into the exponent), e - 1 above it
  m = ((m + 0x200ull) >> 10) + ((uint64_t)(uint32_t)(e - 1) << 52);
  return double_of(a ? sgn | m : 0ull);
}
// Between two axes an array stays in fixed point, each line with the exponent q of its unit
// (values v 2^q, |v| < 2^63; FIX_NAN for a line of NaN): the next axis's lines bring their
// elements' units to one.
constexpr int FIX_NAN = INT_MIN;
constexpr int FIX_TOP = 4096;  // makes a line's top positive
FX uint64_t fix_size(fix v) { return (uint64_t)(v < 0 ? -v : v); }
// FIX_TOP + q + the bits of the larger component; 0 for zeros, FIX_TOP^2 for NaN
FX int fix_top(const CFix& v, int q) {
  const uint64_t m = fix_size(v.x) | fix_size(v.y);
  return q == FIX_NAN ? FIX_TOP * FIX_TOP : (m ? FIX_TOP + q + 64 - leading_zeros(m) : 0);
}
// |v| 2^q in units of 2^(top - FIX_TOP - 20), rounded up
FX int fix_units(fix v, int q, int top) {
  const int n = top - FIX_TOP - 20 - q;
  const uint64_t a = fix_size(v);
  return (int)(n >= 0 ? a >> imin(n, 63) : a << imin(-n, 63)) + 1;
}
// The exponent of a line's unit: the sum of its sizes, `sum` of the units above, stays below 2^62.
FX int fix_line_exponent(int top, int sum) {
  if (top == FIX_TOP * FIX_TOP) return FIX_NAN;
  return top == 0 ? 0 : top - FIX_TOP - 20 - (62 - (64 - leading_zeros((uint64_t)(unsigned)imax(sum, 1))));
}
// v 2^q in units of 2^to, rounded to the nearest
FX fix fix_rescale(fix v, int q, int to) {
  const int n = to - q;
  if (n <= 0) return (fix)((uint64_t)v << imin(-n, 63));
  return ((v >> imin(n - 1, 63)) + 1) >> 1;
}
FX double fix_nan() { return double_of(0x7ff8000000000000ull); }
// x / d and x mod d by a multiplication, for 0 <= x < 2^32 / d; made on the host.
struct FastDiv {
  unsigned d, m;
  FX int div(int x) const {
    const int q = (int)(((unsigned long long)(unsigned)x * m) >> 32);
    return m ? q : x;
  }
  FX int mod(int x, int q) const { return x - q * (int)d; }
};
inline FastDiv fast_div(int n) {
  FastDiv f;
  f.d = (unsigned)n;
  f.m = n == 1 ? 0u : 0xffffffffu / (unsigned)n + 1u;
  return f;
}

}  // namespace clg
