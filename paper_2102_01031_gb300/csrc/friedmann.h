// friedmann.h -- the kick of b = a' by one pass's volume sums at alpha = 1 with
// self-consistent expansion (tail.cuh); host and device code, shared with a CPU check.
//
// With K_a = (a^3/3)(f_s/m_p)^2 [-E_K + E_G + 2 E_V],  E_K = s_kin/(2 a^6 V),
// E_G = s_grad/(2 a^2 dx^2 V),  E_V = s_pot/V, the two kicks of a pass (weights wout before its
// momentum kick, win after) are a linear form of the sums, whose coefficients are
// formed before the sums are known.
#pragma once

#include "fix_fft.h"  // FX

namespace clg {

struct Alpha1Kick {
  double b, pre, c[3];  // a' before the kicks; the pre-kick kinetic part; factors of the sums
};

// K = (f_s/m_p)^2/(6 V); pi2: the pre-kick sum of pi^2
FX Alpha1Kick alpha1_kick(double K, double inv_dx2, double a, double b, double pi2, double wout, double win) {
  const double ws = wout + win, a3 = a * a * a, k3 = K / a3;
  Alpha1Kick k;
  k.b = b;
  k.pre = -wout * k3 * pi2;
  k.c[0] = -win * k3;
  k.c[1] = ws * (K * inv_dx2) * a;
  k.c[2] = 4.0 * ws * K * a3;
  return k;
}

// a' after the kicks.  The terms, each a small part of a', are added among themselves and a'
// last: it is rounded once a pass (with every term added to it in turn, four times, a run's
// a' drifted 1.7 times as far).  One dependent operation more than a chain that starts at a'.
FX double alpha1_b(const Alpha1Kick& k, double kin, double grad, double pot) {
  return k.b + fma(k.c[0], kin, fma(k.c[1], grad, fma(k.c[2], pot, k.pre)));
}

// a after the drift by dn; a pass that closes a stream (dn = 0) leaves a as it is, whatever a' is.
FX double alpha1_a(double dn, double b, double a) { return dn == 0.0 ? a : fma(dn, b, a); }

}  // namespace clg
