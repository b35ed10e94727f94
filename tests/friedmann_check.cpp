// CPU check of the kick of a' between two passes at alpha = 1 (csrc/friedmann.h) against
// extended precision: a' is rounded once, at its own size, whatever the number of terms.
// Bound, u = 2^-53: half a unit in the last place of the result, and 12 u of the terms'
// sizes (a coefficient takes at most 8 roundings: 3 for K, 3 for a^3 and the division or
// 2 for a^3 and 1 for the weights' sum, and its products; the terms' sum 3, the last one
// with the rounding of K's own factors to spare).
// A pass without a drift leaves a as it is, also where a' is no number.
// Then a homogeneous field's run: the error of a' stays that of the form that adds one
// increment to it.  Prints "OK" or "FAIL ...".
#include <cmath>
#include <cstdio>
#include <limits>
#include <random>

#include "friedmann.h"

using namespace clg;
typedef long double ld;

int main() {
  const double u = std::ldexp(1.0, -53);
  std::mt19937_64 g(7);
  std::uniform_real_distribution<double> U(0.0, 1.0);
  int fails = 0;
  for (int n = 0; n < 200000; ++n) {
    const int N = 8 * (1 + (int)(g() % 64));
    const double V = (double)N * N * N, inv_V = 1.0 / V, inv_dx2 = std::exp(6.0 * U(g) - 1.0);
    const double fm2 = std::pow(10.0, -4.0 * U(g)), K = fm2 * (1.0 / 6.0) * inv_V;
    const double a = std::exp(4.0 * U(g)), b = std::exp(4.0 * U(g) - 2.0), h = 0.02 * (U(g) - 0.3);
    const double wout = 0.5 * h, win = n % 3 ? 0.5 * h : 0.3 * h;
    const double pi2 = V * std::exp(3.0 * U(g) - 1.0) * a * a, kin = pi2 * (1.0 + 0.01 * (U(g) - 0.5));
    const double grad = V * 0.01 * U(g), pot = V * 0.25 * U(g) / (a * a * a * a);
    const double got = alpha1_b(alpha1_kick(K, inv_dx2, a, b, pi2, wout, win), kin, grad, pot);
    const ld A = a, k = (ld)fm2 / 6 * (ld)inv_V;
    const ld t[4] = {-(ld)wout * k / (A * A * A) * pi2, -(ld)win * k / (A * A * A) * kin,
                     ((ld)wout + win) * k * inv_dx2 * A * grad, 4 * ((ld)wout + win) * k * A * A * A * pot};
    const ld want = (ld)b + t[0] + t[1] + t[2] + t[3];
    // the difference without want's own rounding: b - got is exact
    const ld off = std::fabs(((ld)b - (ld)got) + ((t[0] + t[1]) + (t[2] + t[3])));
    const ld size = std::fabs(t[0]) + std::fabs(t[1]) + std::fabs(t[2]) + std::fabs(t[3]);
    int e;
    std::frexp((double)want, &e);
    const ld tol = std::ldexp(0.5L, e - 53) + 12 * (ld)u * size;
    if (!(off <= tol) && ++fails < 5)
      std::printf("FAIL case %d: off by %.3Lf units in the last place\n", n, off / std::ldexp(1.0L, e - 53));
  }
  for (double b : {1.5, std::numeric_limits<double>::infinity(), std::nan("")})
    if (alpha1_a(0.0, b, 2.5) != 2.5) {
      ++fails;
      std::printf("FAIL no drift, a' = %g: a = %g\n", b, alpha1_a(0.0, b, 2.5));
    }
  if (alpha1_a(0.01, 3.0, 2.5) != std::fma(0.01, 3.0, 2.5)) { ++fails; std::printf("FAIL drift\n"); }
  // phi^4/4 without gradients, leapfrog steps: a' against the same steps in extended precision,
  // and the form that adds the whole increment at once
  double sum_new = 0.0, sum_one = 0.0;
  const int runs = 2000, steps = 200;
  for (int r = 0; r < runs; ++r) {
    const double h = 0.005, fm2 = 0.25, K = fm2 / 6.0;
    const double f0 = 1.0 + 0.2 * U(g), p0 = 0.2 * (U(g) - 0.5);
    const double b0 = std::sqrt(fm2 / 3.0 * (0.5 * p0 * p0 + 0.25 * f0 * f0 * f0 * f0));
    struct D { double f, p, a, b; } x = {f0, p0, 1.0, b0}, y = x;
    struct { ld f, p, a, b; } z = {f0, p0, 1.0L, b0};
    for (int s = 0; s < steps; ++s) {
      for (int form = 0; form < 2; ++form) {
        D& d = form ? y : x;
        const double ab = std::fma(0.5 * h, d.b, d.a);
        d.f = std::fma(h / (ab * ab), d.p, d.f);
        d.a = std::fma(h, d.b, d.a);
        const double pn = std::fma(-h * d.a * d.a * d.a * d.a, d.f * d.f * d.f, d.p), f2 = d.f * d.f;
        const double kin0 = d.p * d.p, kin1 = pn * pn, pot = 0.25 * f2 * f2;
        if (form == 0) {
          d.b = alpha1_b(alpha1_kick(K, 1.0, d.a, d.b, kin0, 0.5 * h, 0.5 * h), kin1, 0.0, pot);
        } else {
          const double a3 = d.a * d.a * d.a, ck = 0.5 / (a3 * a3);
          const double br = std::fma(-1.0, 0.5 * h * (kin0 * ck) + 0.5 * h * (kin1 * ck), h * (2.0 * pot));
          d.b = std::fma(a3 * (fm2 / 3.0), br, d.b);
        }
        d.p = pn;
      }
      const ld ab = z.a + 0.5L * h * z.b;
      z.f += (ld)h / (ab * ab) * z.p;
      z.a += (ld)h * z.b;
      const ld a3 = z.a * z.a * z.a, pn = z.p - (ld)h * a3 * z.a * z.f * z.f * z.f;
      z.b += a3 * ((ld)fm2 / 3) * (0.5L * h) * (-(z.p * z.p + pn * pn) / (2 * a3 * a3) + z.f * z.f * z.f * z.f);
      z.p = pn;
    }
    const double en = (double)((x.b - z.b) / z.b), eo = (double)((y.b - z.b) / z.b);
    sum_new += en * en;
    sum_one += eo * eo;
  }
  const double rn = std::sqrt(sum_new / runs), ro = std::sqrt(sum_one / runs);
  std::printf("%srms error of a' after %d steps: %.3g, with one increment added at once %.3g\n",
              rn <= 1.1 * ro ? "" : "FAIL ", steps, rn, ro);
  if (!(rn <= 1.1 * ro)) ++fails;
  if (!fails) std::printf("OK\n");
  return fails != 0;
}
