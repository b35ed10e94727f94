// adj_kick.h -- arithmetic of the FP64 adjoint sweep (pass_adjoint.cu, adjoint_kernels.cu) whose rounding is
// checked on the CPU; host and device code.
#pragma once

#include "fix_fft.h"  // FX

namespace clg {

// p + A1 lap - A3 d: the increment is formed first and p added last, so that p's size is rounded
// at once (two FMAs into p, one operation less on the FP64 unit, round it twice).
FX double kicked(double p, double A1, double lap, double A3, double d) { return p + fma(A1, lap, -(A3 * d)); }

// dJ/dphi of the chi energy fraction J (adjoint_kernels.cu) at one site: chi 1 for the chi field,
// dEG and dV/V the site's share in the gradient and potential energies, over rho.  Divided by V
// and rho for FP64 storage; FP32 storage, whose rounding is 2^29 times as large, multiplies by
// their reciprocals (about 20 FP64 operations a site less; 128^3 376 -> 279 us).
template <bool FP64>
FX double fraction_gradient(double chi, double J, double dEG, double dV, double V, double rho, double iV, double irho) {
  return FP64 ? (chi * dEG - J * (dEG + dV / V)) / rho : (chi * dEG - J * (dEG + dV * iV)) * irho;
}

}  // namespace clg
