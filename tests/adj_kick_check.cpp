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
  // the gradient of the energy fraction, one term at a time: with dEG = 0 and J = 1 the two
  // quotients round once each; with dV = 0 and chi - J = 1 the one quotient does
  for (int n = 0; n < 200000; ++n) {
    const int N = 8 * (1 + (int)(g() % 64));
    const double V = (double)N * N * N, rho = std::exp(3.0 * U(g)), x = U(g), iV = 1.0 / V, irho = 1.0 / rho;
    const ld a = -(ld)x / V / rho, b = (ld)x / rho;
    const ld ea = std::fabs((ld)fraction_gradient<true>(0.0, 1.0, 0.0, x, V, rho, iV, irho) - a) / std::fabs(a);
    const ld eb = std::fabs((ld)fraction_gradient<true>(1.0, 0.0, x, 0.0, V, rho, iV, irho) - b) / std::fabs(b);
    if (!(ea <= 2 * u * (1 + u) && eb <= u) && ++fails < 5)
      std::printf("FAIL gradient %d: off by %.3Lf and %.3Lf of 2^-53\n", n, ea / u, eb / u);
  }
  if (!fails) std::printf("OK\n");
  return fails != 0;
}
