// CPU check of the fixed-point transforms' arithmetic (csrc/fix_fft.h): for every lattice
// size and several kinds of line, the error of a fixed-point Stockham transform against
// an extended-precision one is at most that of the same transform in FP64, or one unit in
// the last place of the FP64 values that carry it (both as the norm of the difference over
// the norm of the result), conversions at the edges of the
// formats, and the divisions by multiplication.  Prints "OK <worst ratio>" or "FAIL ...".
#include <algorithm>
#include <cmath>
#include <complex>
#include <cstdio>
#include <limits>
#include <random>
#include <vector>

#include "fix_fft.h"

using namespace clg;
typedef long double ld;
static int fails = 0;
static void expect(bool ok, const char* what, double a, double b) {
  if (ok) return;
  ++fails;
  std::printf("FAIL %s: %.17g %.17g\n", what, a, b);
}

static std::vector<int> radices(int N) {
  std::vector<int> r;
  while (N % 4 == 0) { r.push_back(4); N /= 4; }
  while (N % 2 == 0) { r.push_back(2); N /= 2; }
  while (N % 3 == 0) { r.push_back(3); N /= 3; }
  return r;
}

// Stockham passes in a floating type (the form the transforms had in FP64)
template <typename F>
static std::vector<std::complex<F>> stockham(std::vector<std::complex<F>> a, int sign) {
  const int N = (int)a.size();
  std::vector<std::complex<F>> b(N), w(N);
  const ld pi = std::acos((ld)-1);
  for (int e = 0; e < N; ++e) w[e] = std::complex<F>((F)std::cos(2 * pi * e / N), (F)(sign * std::sin(2 * pi * e / N)));
  int Ns = 1;
  for (int R : radices(N)) {
    const int NR = N / R, L = Ns * R, ts = N / L;
    for (int j = 0; j < NR; ++j) {
      const int k = j % Ns;
      std::complex<F> v[4], o[4];
      for (int r = 0; r < R; ++r) {
        v[r] = a[j + r * NR];
        if (k && r) v[r] = std::complex<F>(v[r].real() * w[k * r * ts].real() - v[r].imag() * w[k * r * ts].imag(),
                                           v[r].real() * w[k * r * ts].imag() + v[r].imag() * w[k * r * ts].real());
      }
      const std::complex<F> I(0, sign);
      if (R == 2) {
        o[0] = v[0] + v[1];
        o[1] = v[0] - v[1];
      } else if (R == 4) {
        const std::complex<F> t0 = v[0] + v[2], t1 = v[0] - v[2], t2 = v[1] + v[3], d = v[1] - v[3];
        const std::complex<F> t3(-sign * d.imag(), sign * d.real());
        o[0] = t0 + t2; o[1] = t1 + t3; o[2] = t0 - t2; o[3] = t1 - t3;
      } else {
        const F h = (F)(std::sqrt((ld)3) / 2) * sign;
        const std::complex<F> s = v[1] + v[2], d = v[1] - v[2], m = v[0] - s * (F)0.5;
        o[0] = v[0] + s;
        o[1] = std::complex<F>(m.real() - h * d.imag(), m.imag() + h * d.real());
        o[2] = std::complex<F>(m.real() + h * d.imag(), m.imag() - h * d.real());
      }
      for (int q = 0; q < R; ++q) b[(j / Ns) * L + k + q * Ns] = o[q];
    }
    std::swap(a, b);
    Ns = L;
  }
  return a;
}

template <int R>
static void stage(const std::vector<CFix>& a, std::vector<CFix>& b, const std::vector<int>& w, int sign, int Ns) {
  const int N = (int)a.size(), NR = N / R, L = Ns * R, ts = N / L;
  for (int j = 0; j < NR; ++j) {
    const int k = j % Ns;
    CFix v[R];
    for (int r = 0; r < R; ++r) {
      v[r] = a[j + r * NR];
      const int* t = &w[4 * (k * r * ts)];
      if (Ns > 1 && r) v[r] = cmul(v[r], t[0], t[1], t[2], t[3]);
    }
    butterfly<R>(v, sign);
    for (int q = 0; q < R; ++q) b[(j / Ns) * L + k + q * Ns] = v[q];
  }
}

static std::vector<std::complex<double>> fixed(const std::vector<std::complex<double>>& x, int sign) {
  const int N = (int)x.size();
  const ld pi = std::acos((ld)-1);
  std::vector<int> w(4 * N);
  for (int e = 0; e < N; ++e) {
    root_words((double)std::cos(2 * pi * e / N), w[4 * e], w[4 * e + 1]);
    root_words((double)(sign * std::sin(2 * pi * e / N)), w[4 * e + 2], w[4 * e + 3]);
  }
  int top = 0, sum = 0;
  for (auto& v : x) top = std::max(top, std::max(top_of(v.real()), top_of(v.imag())));
  const int E = expo_of<double>(top);
  for (auto& v : x) sum += size_of(v.real(), E) + size_of(v.imag(), E);
  const LineScale sc = line_scale<double>(E, sum);
  std::vector<CFix> a(N), b(N);
  for (int i = 0; i < N; ++i) {
    a[i].x = to_fix(x[i].real(), sc);
    a[i].y = to_fix(x[i].imag(), sc);
  }
  int Ns = 1;
  for (int R : radices(N)) {
    if (R == 4) stage<4>(a, b, w, sign, Ns);
    else if (R == 2) stage<2>(a, b, w, sign, Ns);
    else stage<3>(a, b, w, sign, Ns);
    std::swap(a, b);
    Ns *= R;
  }
  std::vector<std::complex<double>> y(N);
  const int q = E - FixIO<double>::BIAS - sc.up;
  for (int i = 0; i < N; ++i) y[i] = std::complex<double>(from_fix(a[i].x, q, sc.plain), from_fix(a[i].y, q, sc.plain));
  return y;
}

int main() {
  std::mt19937_64 g(7);
  std::normal_distribution<double> n01;
  std::uniform_real_distribution<double> u01;
  double worst = 0.0;
  const char* kinds[] = {"white noise", "mean 1 and ripples", "steep spectrum", "single mode", "tiny", "huge", "constant",
                         "near a constant's bound", "one-sided"};
  for (int N : {8, 16, 24, 32, 48, 64, 72, 96, 128, 144, 192, 216, 256, 288, 384, 432, 512})
    for (int kind = 0; kind < 9; ++kind)
      for (int sign : {-1, 1}) {
        double ef = 0.0, ex = 0.0, nn = 0.0;
        for (int rep = 0; rep < 24; ++rep) {
          std::vector<std::complex<double>> x(N);
          const double ph = 6.283185307179586 * u01(g);
          const int m = 1 + (int)(u01(g) * (N / 2));
          for (int i = 0; i < N; ++i) {
            const double a = n01(g), b = n01(g);
            if (kind == 0) x[i] = {a, b};
            if (kind == 1) x[i] = {1.0 + 0.02 * a, 1.0 + 0.02 * b};
            if (kind == 2) x[i] = {std::cos(6.283185307179586 * i / N + ph) + 1e-3 * a, 1e-6 * b};
            if (kind == 3) x[i] = {std::cos(6.283185307179586 * i * m / N + ph), std::sin(6.283185307179586 * i * m / N + ph)};
            if (kind == 4) x[i] = {1e-290 * a, 1e-290 * b};
            if (kind == 5) x[i] = {1e290 * a, 1e290 * b};
            if (kind == 6) x[i] = {ph, -ph};
            if (kind == 7) x[i] = {2.0 - 1e-9 * u01(g), 2.0 - 1e-9 * u01(g)};
            if (kind == 8) x[i] = {std::exp(2.0 * a), 0.0};
          }
          std::vector<std::complex<ld>> xl(N);
          for (int i = 0; i < N; ++i) xl[i] = std::complex<ld>(x[i].real(), x[i].imag());
          const auto yl = stockham<ld>(xl, sign);
          const auto yd = stockham<double>(x, sign);
          const auto yf = fixed(x, sign);
          // scaled so that squares stay in range
          const ld sc = kind == 4 ? 1e290L : (kind == 5 ? 1e-290L : 1.0L);
          for (int i = 0; i < N; ++i) {
            const std::complex<ld> d((ld)yd[i].real() - yl[i].real(), (ld)yd[i].imag() - yl[i].imag());
            const std::complex<ld> f((ld)yf[i].real() - yl[i].real(), (ld)yf[i].imag() - yl[i].imag());
            ef += (double)std::norm(d * sc);
            ex += (double)std::norm(f * sc);
            nn += (double)std::norm(yl[i] * sc);
          }
        }
        const double rd = std::sqrt(ef / nn), rf = std::sqrt(ex / nn);
        worst = std::max(worst, rf / std::max(rd, 0x1p-52));
        if (!(rf <= std::max(rd, 0x1p-52))) {
          ++fails;
          std::printf("FAIL N %d %s sign %d: fixed %.3g FP64 %.3g\n", N, kinds[kind], sign, rf, rd);
        }
      }
  // conversions: exact at the line's scale, rounded below it, and the formats' edges
  for (double v : {1.0, -1.5, 0x1p-1022, 0x1.8p-1060, 1e300, -3.25e-17, 0.0}) {
    const LineScale sc = line_scale<double>(expo_of<double>(top_of(v)), 1 << 21);
    const double r = from_fix(to_fix(v, sc), sc.E - FixIO<double>::BIAS - sc.up, sc.plain);
    expect(r == v, "FP64 round trip", v, r);
  }
  for (float v : {1.0f, -1.5f, 1e-40f, 3e38f, -2e-3f, 0.0f}) {
    const LineScale sc = line_scale<float>(expo_of<float>(top_of(v)), 1 << 21);
    const double r = from_fix(to_fix(v, sc), sc.E - FixIO<float>::BIAS - sc.up, sc.plain);
    expect(r == (double)v, "FP32 round trip", v, r);
  }
  for (int E : {1023, 1, 2046, 210})  // values far below the line's scale, zeros among them
    for (double v : {0.0, -0.0, 0x1p-1074, std::ldexp(1.0, E - 1023 - 64)}) {
      const LineScale sc = line_scale<double>(E, 1 << 21);
      if (top_of(v) >> 20 > E) continue;
      const double want = std::nearbyint((double)std::ldexp((long double)v, FixIO<double>::BIAS - E + sc.up));
      const fix got = to_fix(v, sc);
      expect(std::fabs((double)got - want) <= 0.5, "small values", (double)got, want);
      expect(v != 0.0 || got == 0, "zero", (double)got, 0);
    }
  for (int E : {127, 101, 100, 1}) {
    const LineScale sc = line_scale<float>(E, 1 << 22);
    expect(to_fix(0.0f, sc) == 0 && to_fix(-0.0f, sc) == 0, "FP32 zero", E, 0);
    const float tiny = 1.4e-45f;  // the smallest subnormal, one unit of 2^(1 - 150)
    const double want = std::ldexp(1.0, 1 - E + sc.up);
    expect(std::fabs((double)to_fix(tiny, sc) - want) <= (sc.plain ? 0x1p-14 * std::ldexp(1.0, sc.up) : 0.5),
           "FP32 subnormal", (double)to_fix(tiny, sc), want);
  }
  expect(from_fix(1ll << 62, 1000, false) == std::numeric_limits<double>::infinity(), "overflow", 0, 0);
  expect(from_fix(-(1ll << 62), -62 - 1074, false) == -0x1p-1074, "smallest subnormal", 0, 0);
  for (int k = 0; k < 200000; ++k) {
    const fix v = (fix)(g() >> (2 + g() % 62)) * ((g() & 1) ? 1 : -1);
    const int q = (int)(g() % 200) - 100;
    const long double want = std::ldexp((long double)v, q);
    for (bool plain : {true, false}) {
      const double r = from_fix(v, q, plain);
      expect(std::fabs((double)((long double)r - want)) <= std::ldexp((double)std::fabs(want), -53), "rounding", r,
             (double)want);
      expect((r < 0) == (v < 0) && (r == 0) == (v == 0), "sign", r, (double)want);
    }
  }
  expect(expo_of<double>(top_of(std::numeric_limits<double>::quiet_NaN())) == FixIO<double>::ETOP, "NaN", 0, 0);
  expect(expo_of<float>(top_of(std::numeric_limits<float>::infinity())) == FixIO<float>::ETOP, "inf", 0, 0);
  for (int d = 1; d <= 2048; ++d) {
    const FastDiv f = fast_div(d);
    for (int x = 0; x < (1 << 20); x += 1 + x / 8192)
      if (f.div(x) != x / d || f.mod(x, f.div(x)) != x % d) {
        ++fails;
        std::printf("FAIL division %d %d\n", x, d);
        break;
      }
  }
  if (!fails) std::printf("OK worst ratio to FP64 %.3f\n", worst);
  return fails != 0;
}
