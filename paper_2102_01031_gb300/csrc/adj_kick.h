// adj_kick.h -- arithmetic of the FP64 adjoint sweep (pass_adjoint.cu) whose rounding is
// checked on the CPU; host and device code.
#pragma once

#include "fix_fft.h"  // FX

namespace clg {

// p + A1 lap - A3 d: the increment is formed first and p added last, so that p's size is rounded
// at once (two FMAs into p, one operation less on the FP64 unit, round it twice).
FX double kicked(double p, double A1, double lap, double A3, double d) { return p + fma(A1, lap, -(A3 * d)); }

}  // namespace clg
