"""How the doublet passes add up a site's six hops: pairs first, so that fields near a constant
lose nothing.

Fields of 1 on the even sites and 1 + e on the odd ones (e one unit in the last place of 1),
links at the identity, no potential: the Laplacian at an even site is 6 e, and the sums
-6 + 2 (1 + e), + 2 (1 + e), + 2 (1 + e) are exact at every step, where a sum taken hop by hop
passes through -5 + e and rounds e away.  One velocity-Verlet step kicks twice by half a step
(its drift is far below e): the momenta are twice the rounded A1 6 e, A1 = h/(2 dx^2).
Tolerance 1e-6 (FP32) and 1e-14 (FP64): the rounding of A1 and of the product, two units each."""
import math

import numpy as np
import pytest

import oracle as O

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("fp32", [1, 0])
@pytest.mark.parametrize("exp", [O.EXP_SELF, O.EXP_OFF])
@pytest.mark.parametrize("model,N", [(O.MODEL_SU2U1_HIGGS, 16), (O.MODEL_LPHI4_SU2U1, 32), (O.MODEL_LPHI4_SU2U1, 48)])
def test_nearly_constant_fields(model, N, exp, fp32):
    import paper_2102_01031_gb300 as P
    kIR, h, full = 0.5, 0.01, model == O.MODEL_LPHI4_SU2U1
    kw = dict(dt=h, integrator=O.VV2, lam=0.0, v=0.0, gQ=0.6, gQB=0.8, fstar_over_omegastar=1.3, phi0=[1.0] * 4,
              dphi0=[0.0] * 4, fluct_amp2=0.0, expansion=exp, fstar_over_mp=0.5, precision=fp32)
    if full:
        kw.update(qG=0.0, qH=0.0, Qc=0.7)
    g = P.Lattice(model, N, kIR, 1.0, 1, P.make_params(**kw))
    z, y, x = np.meshgrid(*[np.arange(N)] * 3, indexing="ij")
    odd = (x + y + z) % 2
    eps = 2.0 ** (-23 if fp32 else -52)
    fields, momenta = [0, 1, 2, 3], [4, 5, 6, 7]
    if full:
        fields, momenta = fields + [35, 37, 38], momenta + [36, 39, 40]
    one, zero = np.ones((N, N, N)), np.zeros((N, N, N))
    for a in range(41 if full else 35):
        if a in fields:
            g.set_array(a, 1.0 + eps * odd)
        else:
            g.set_array(a, one if a in (14, 18, 22) else zero)  # links at the identity
    g.step(1)
    dx = 2.0 * math.pi / (N * kIR)
    want = 2.0 * (0.5 * h / dx ** 2) * 6.0 * eps
    for a in momenta:
        got = g.get_array(a)[odd == 0]
        assert np.abs(got - want).max() <= (1e-6 if fp32 else 1e-14) * want, (a, np.abs(got / want - 1.0).max())
