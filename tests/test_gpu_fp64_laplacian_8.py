"""The FP64 scalar passes' Laplacian at 8^3, where a tile is as tall as the lattice and wraps on both
sides, for each kind of field (one-field runs with expansion need noise whatever the kind, so the
kinds act on chi there).  Tolerance as in test_gpu_fp64_laplacian.py."""
import numpy as np
import pytest

import oracle as O
from tests.test_gpu_fp64_laplacian import field, reach

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("kind", ["noise", "bump", "tiny", "zero"])
@pytest.mark.parametrize("model,exp", [(O.MODEL_LPHI4_CHI, O.EXP_SELF), (O.MODEL_LPHI4, O.EXP_OFF)])
def test_fp64_scalar_pass_8(model, exp, kind):
    import paper_2102_01031_gb300 as P
    N, n, kw = 8, 3, dict(dt=0.005, q=100.0, phi0=[1.0, 0.0], fluct_amp2=0.0, fstar_over_mp=0.5, integrator=O.VV2,
                          expansion=exp)
    g = P.Lattice(model, N, 0.5, 1.0, 3, P.make_params(**kw))
    o = O.Oracle(model, N, 0.5, 1.0, 3, O.make_params(**kw))
    nf = g.nfields()
    for f in range(nf):
        for w in (0, 1):
            x = field(kind if f == nf - 1 else "noise", N, 10 * f + w)
            g.set(f, w, x)
            o.set(f, w, x)
    g.step(n)
    o.step(n)
    for f in range(nf):
        for w in (0, 1):
            ref, got = o.get(f, w), g.get(f, w)
            scale = np.maximum(reach(o.get(f, 0), n + 1), reach(o.get(f, 1), n + 1))
            assert np.all(np.abs(got - ref) <= 1e-10 * scale + 1e-318), (f, w)
    eg, eo = g.energies(), o.energies()
    for key in ("a", "b", "rho"):
        assert abs(eg[key] - eo[key]) <= 1e-10 * abs(eo[key]) + 1e-300, key
