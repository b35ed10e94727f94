// CPU check of the integer Laplacian sums (csrc/fix_lap.h) against sums in extended
// precision.  Bound, from the header: 13 units of 2^-58 of the largest of the seven
// values' power of two, and half a unit in the last place of the result; and over each
// kind of input no larger in the mean square than the FP64 form's error.
// Prints "OK <worst ratio of the two errors>" or "FAIL ...".
#include <algorithm>
#include <cmath>
#include <cstdio>
#include <limits>
#include <random>

#include "fix_lap.h"

using namespace clg;
static int fails = 0;

static double lap(const double* v, bool* ok) {
  FixVal f[7];
  for (int i = 0; i < 7; ++i) f[i] = fix_val(v[i]);
  return fix_lap(f[0], f[1], f[2], f[3], f[4], f[5], f[6], ok);
}

int main() {
  std::mt19937_64 g(7);
  std::normal_distribution<double> nd;
  std::uniform_real_distribution<double> ud(-1.0, 1.0);
  double worst = 0;
  // kinds: smooth around a mean, noise around zero, wide range of sizes, exact binades and
  // their neighbours, very large and very small values, one value far above the others,
  // zeros and subnormals among the neighbours
  for (int kind = 0; kind < 8; ++kind) {
    double fix2 = 0, ref2 = 0;
    for (int n = 0; n < 400000; ++n) {
      double v[7];
      const double sc = kind == 4 ? std::ldexp(1.0, 960) : (kind == 5 ? std::ldexp(1.0, -945) : 1.0);
      for (int i = 0; i < 7; ++i) {
        if (kind == 0) v[i] = (n & 1 ? -1.0 : 1.0) + 1e-4 * nd(g);
        else if (kind == 2) v[i] = nd(g) * std::ldexp(1.0, (int)(60 * ud(g)));
        else if (kind == 3) v[i] = std::nextafter(std::ldexp(n & 1 ? -1.0 : 1.0, (int)(3 * ud(g))), (i & 1) ? 0.0 : 4.0);
        else if (kind == 6) v[i] = nd(g) * (i == n % 7 ? std::ldexp(1.0, n % 70) : 1.0);
        else if (kind == 7) v[i] = i == (n >> 3) % 7 ? 5e-324 * (n & 7) : (i == n % 7 ? 0.0 : nd(g));
        else v[i] = sc * nd(g);
      }
      bool ok;
      const double got = lap(v, &ok);
      long double ex = 0;
      double mx = 0;
      for (int i = 0; i < 6; ++i) ex += v[i];
      ex -= 6.0L * v[6];
      for (double x : v) mx = std::max(mx, std::fabs(x));
      if (!ok) { ++fails; std::printf("FAIL range kind %d\n", kind); break; }
      const int be = std::ilogb(mx);
      const long double unit = std::ldexp(1.0L, be - 58);
      const long double err = std::fabs((long double)got - ex);
      const long double bound = 13 * unit + 0.5L * std::ldexp(1.0L, std::max(std::ilogb((double)ex == 0 ? mx : (double)ex), -1022) - 52);
      if (!(err <= bound)) {
        ++fails;
        std::printf("FAIL kind %d: %.17g exact %.21Lg bound %.3Lg\n", kind, got, ex, bound);
        break;
      }
      const long double e64 = (long double)fp64_lap(v[0], v[1], v[2], v[3], v[4], v[5], v[6]) - ex;
      fix2 += (double)((err / unit) * (err / unit));
      ref2 += (double)((e64 / unit) * (e64 / unit));
    }
    const double r = std::sqrt(fix2 / ref2);
    worst = std::max(worst, r);
    if (!(r <= 1.0)) { ++fails; std::printf("FAIL kind %d: error %.3g of FP64's\n", kind, r); }
  }
  // equal values of either sign, zero, and the values that take the FP64 form
  const double inf = std::numeric_limits<double>::infinity(), nan = std::numeric_limits<double>::quiet_NaN();
  for (double x : {1.0, -1.0, 3e-200, -7e200, 1.9999999999999998}) {
    double v[7] = {x, x, x, x, x, x, x};
    bool ok;
    const double r = lap(v, &ok);
    if (!ok || r != 0.0 || std::signbit(r)) { ++fails; std::printf("FAIL equal %g -> %g\n", x, r); }
  }
  for (double x : {inf, -inf, nan, 1e308, -1.7e308})
    for (int i = 0; i < 7; ++i) {
      double v[7] = {1, 2, 3, 4, 5, 6, 7};
      v[i] = x;
      bool ok;
      lap(v, &ok);
      if (ok) { ++fails; std::printf("FAIL %g accepted\n", x); }
    }
  for (double x : {0.0, 1e-300, 5e-324}) {
    double v[7] = {x, x, 0, 0, x, -x, x};
    bool ok;
    lap(v, &ok);
    if (ok) { ++fails; std::printf("FAIL %g accepted\n", x); }
  }
  if (!fails) std::printf("OK %.3f\n", worst);
  return fails != 0;
}
