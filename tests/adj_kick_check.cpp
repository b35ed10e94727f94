// CPU check of the FP64 adjoint sweep's arithmetic (csrc/adj_kick.h) against extended
// precision.  Prints "OK" or "FAIL ...".
#include <cmath>
#include <cstdio>
#include <random>

#include "adj_kick.h"

using namespace clg;
typedef long double ld;

int main() {
  const ld u = std::ldexp(1.0L, -53);
  std::mt19937_64 g(11);
  std::uniform_real_distribution<double> U(-1.0, 1.0);
  int fails = 0;
  // a kick: half a unit in the last place of the result, and two roundings of the increment
  for (int n = 0; n < 200000; ++n) {
    const double p = U(g), A1 = 0.05 * U(g), lap = 0.2 * U(g), A3 = 0.005 * U(g), d = 2.0 * U(g);
    const double got = kicked(p, A1, lap, A3, d);
    const ld t1 = (ld)A1 * lap, t2 = -(ld)A3 * d;
    int e;
    std::frexp((double)((ld)p + t1 + t2), &e);
    const ld off = std::fabs(((ld)p - (ld)got) + (t1 + t2));
    const ld tol = std::ldexp(0.5L, e - 53) + 2 * u * (std::fabs(t1) + std::fabs(t2));
    if (!(off <= tol) && ++fails < 5)
      std::printf("FAIL kick %d: off by %.3Lf units in the last place\n", n, off / std::ldexp(1.0L, e - 53));
  }
  if (!fails) std::printf("OK\n");
  return fails != 0;
}
