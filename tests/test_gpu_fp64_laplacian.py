"""The FP64 scalar passes' Laplacian in integers (csrc/fix_lap.h) against the FP64 oracle:
tile heights with and without warps that have no sites, fields whose sizes differ by many
orders of magnitude from site to site, and values at the ends of the exponent range, which
take the FP64 form.

Tolerance: after n steps a site is compared with the largest value within n + 1 sites of it
(what can have reached it), 1e-10 as in the other FP64 tests."""
import numpy as np
import pytest

import oracle as O

pytestmark = pytest.mark.gpu


def reach(x, n):
    """Largest |x| within n sites along each axis (periodic)."""
    m = np.abs(x)
    for ax in range(3):
        m = np.max([np.roll(m, s, ax) for s in range(-n, n + 1)], axis=0)
    return m


def field(kind, N, seed):
    rng = np.random.default_rng(seed)
    x = 0.3 * rng.standard_normal((N, N, N))
    if kind == "bump":    # 1 down to 1e-60 across the box
        r = np.abs(np.arange(N) - N // 2)
        r2 = r[:, None, None] ** 2 + r[None, :, None] ** 2 + r[None, None, :] ** 2
        return x * np.exp(-138.0 * r2 / r2.max())
    if kind == "tiny":    # the largest exponent below the integer form's range
        return x * 1e-296
    if kind == "zero":
        return np.zeros_like(x)
    return x


@pytest.mark.parametrize("kind", ["noise", "bump", "tiny", "zero"])
@pytest.mark.parametrize("model,N,exp", [(O.MODEL_LPHI4, 8, O.EXP_SELF), (O.MODEL_LPHI4_CHI, 24, O.EXP_SELF),
                                         (O.MODEL_LPHI4_CHI, 72, O.EXP_OFF), (O.MODEL_LPHI4, 64, O.EXP_OFF)])
def test_fp64_scalar_pass(model, N, exp, kind):
    import paper_2102_01031_gb300 as P
    n, kw = 3, dict(dt=0.005, q=100.0, phi0=[1.0, 0.0], fluct_amp2=0.0, fstar_over_mp=0.5, integrator=O.VV2,
                    expansion=exp)
    g = P.Lattice(model, N, 0.5, 1.0, 3, P.make_params(**kw))
    o = O.Oracle(model, N, 0.5, 1.0, 3, O.make_params(**kw))
    nf = g.nfields()
    for f in range(nf):
        for w in (0, 1):
            # phi keeps the background's size, so that a(t) has a source, except in one-field runs without expansion
            x = field(kind if f == nf - 1 and (nf == 2 or exp == O.EXP_OFF) else "noise", N, 10 * f + w)
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
