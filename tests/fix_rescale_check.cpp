// CPU check of the exponents that lines in fixed point carry from one axis of a transform
// to the next (csrc/fix_fft.h): lines of values v 2^q with one unit 2^q per value, as the
// transforms of another axis leave them.  The rescaled line's sum of sizes is below 2^62,
// each value lies within half a unit of the line, and the unit is at most 2^-59 of the
// line's sum of sizes (62 bits, less the rounding up of the sizes and of the sum to a power of two).
#include <cmath>
#include <cstdio>
#include <random>
#include <vector>

#include "fix_fft.h"

using namespace clg;
static int fails = 0;

int main() {
  std::mt19937_64 g(3);
  for (int N : {8, 12, 64, 256, 512})
    for (int kind = 0; kind < 6; ++kind)
      for (int rep = 0; rep < 50; ++rep) {
        std::vector<CFix> v(N);
        std::vector<int> q(N);
        for (int i = 0; i < N; ++i) {
          const int bits = kind == 1 ? (int)(g() % 63) : 62;  // sizes: full, any, ...
          auto draw = [&]() { return (fix)(g() >> (64 - bits - (bits == 0))) * ((g() & 1) ? 1 : -1); };
          v[i] = CFix{draw(), draw()};
          q[i] = kind == 2 ? -900 + (int)(g() % 1800) : -40 + (kind == 3 ? (int)(g() % 3) : 0);
          if (kind == 4 && i != rep % N) v[i] = CFix{0, 0};
          if (kind == 5) v[i] = CFix{0, 0};
        }
        int top = 0;
        for (int i = 0; i < N; ++i) top = imax(top, fix_top(v[i], q[i]));
        long long sum = 0;
        for (int i = 0; i < N; ++i) sum += (long long)fix_units(v[i].x, q[i], top) + fix_units(v[i].y, q[i], top);
        if (sum >= (1ll << 31)) { ++fails; std::printf("FAIL sum\n"); }
        const int to = fix_line_exponent(top, (int)sum);
        long double size = 0, exact = 0;
        for (int i = 0; i < N; ++i)
          for (fix x : {v[i].x, v[i].y}) {
            const fix r = fix_rescale(x, q[i], to);
            const long double want = std::ldexp((long double)x, q[i] - to);
            if (!(std::fabs((long double)r - want) <= 0.5L)) {
              ++fails;
              std::printf("FAIL N %d kind %d: %lld for %.20Lg\n", N, kind, r, want);
            }
            size += std::fabs((long double)r);
            exact += std::fabs(want);
          }
        if (!(size < std::ldexp(1.0L, 62))) { ++fails; std::printf("FAIL size N %d kind %d\n", N, kind); }
        if (kind != 5 && !(exact >= std::ldexp(1.0L, 59))) { ++fails; std::printf("FAIL unit N %d kind %d %.3Lg\n", N, kind, exact); }
        if (fails > 10) return 1;
      }
  const CFix one{1, 0};
  if (fix_line_exponent(imax(fix_top(one, 0), fix_top(one, FIX_NAN)), 5) != FIX_NAN) { ++fails; std::printf("FAIL NaN\n"); }
  if (!fails) std::printf("OK\n");
  return fails != 0;
}
