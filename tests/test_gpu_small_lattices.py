"""Small lattices spread over the SMs (a plane or less per CTA), several lattices per CTA,
and contexts of different sizes alive at once: passes joined by each CTA's own Friedmann
update against the FP64 CPU oracle and against single-pass launches' results.

Tolerances as in the other GPU tests: FP64 storage 1e-10 (normwise, pointwise and on the
averages), FP32 1e-4 pointwise; an ensemble member and a single lattice differ only in the
order of FP64 reductions, 1e-5 in FP32."""
import numpy as np
import pytest

import oracle as O

pytestmark = pytest.mark.gpu

SC = dict(dt=0.005, q=100.0, phi0=[1.0, 0.0], fluct_amp2=1e-4, fstar_over_mp=0.5)
U1 = dict(dt=0.01, lam=1.0, v=1.0, gQ=0.5, fstar_over_omegastar=1.0, phi0=[1.0, 1.0], fluct_amp2=1e-2,
          fstar_over_mp=0.5)


@pytest.fixture(scope="module")
def P():
    import paper_2102_01031_gb300 as P
    P.build()
    P.lib()
    return P


def nrel(a, b):
    return float(np.abs(a - b).max() / max(np.abs(b).max(), 1e-300))


@pytest.mark.parametrize("model,N,integ,exp,alpha,fp32", [
    (O.MODEL_LPHI4, 8, O.VV2, O.EXP_SELF, 1.0, 0), (O.MODEL_LPHI4, 32, O.VV2, O.EXP_SELF, 0.5, 0),
    (O.MODEL_LPHI4_CHI, 24, O.VV4, O.EXP_SELF, 1.0, 0), (O.MODEL_LPHI4_CHI, 48, O.VV4, O.EXP_SELF, 1.0, 1),
    (O.MODEL_LPHI4_CHI, 16, O.LF, O.EXP_FIXED, 1.0, 0), (O.MODEL_LPHI4_CHI, 16, O.VV4, O.EXP_OFF, 1.0, 1),
    (O.MODEL_U1_HIGGS, 8, O.VV2, O.EXP_SELF, 1.0, 0), (O.MODEL_U1_HIGGS, 24, O.VV2, O.EXP_SELF, 0.0, 0),
    (O.MODEL_U1_HIGGS, 16, O.LF, O.EXP_FIXED, 1.0, 0), (O.MODEL_U1_HIGGS, 32, O.VV4, O.EXP_SELF, 1.0, 1)])
def test_small_lattice_matches_oracle(P, model, N, integ, exp, alpha, fp32):
    kw = dict(U1 if model == O.MODEL_U1_HIGGS else SC, integrator=integ, expansion=exp)
    if exp == O.EXP_FIXED:
        kw.update(omega_eos=1.0 / 3.0, H0=0.4)
    g = P.Lattice(model, N, 0.5, alpha, 3, P.make_params(precision=fp32, **kw))
    o = O.Oracle(model, N, 0.5, alpha, 3, O.make_params(**kw))
    for n in (7, 1, 12):  # several launches, one of a single pass where the integrator has one
        g.step(n)
        o.step(n)
    for f in range(g.nfields()):
        for w in (0, 1):
            assert nrel(g.get(f, w), o.get(f, w)) < (1e-4 if fp32 else 1e-10), (f, w)
    eg, eo = g.energies(), o.energies()
    for key in ("a", "b", "rho"):
        assert abs(eg[key] - eo[key]) <= (1e-5 if fp32 else 1e-10) * max(abs(eo[key]), 1e-30), key


@pytest.mark.parametrize("exp", [O.EXP_SELF, O.EXP_OFF])
def test_many_lattices_per_cta(P, exp):
    """400 lattices of 8^3 and one of 64^3: a CTA works on several lattices."""
    kw = dict(SC, integrator=O.VV4, expansion=exp, precision=P.FP32)
    Ns = [8] * 400 + [64]
    seeds = list(range(1, 402))
    E = P.Ensemble(O.MODEL_LPHI4_CHI, Ns, [0.5] * 401, 1.0, seeds, P.make_params(**kw))
    E.step(15)
    for l in (0, 1, 57, 399, 400):
        g = P.Lattice(O.MODEL_LPHI4_CHI, Ns[l], 0.5, 1.0, seeds[l], P.make_params(**kw))
        g.step(15)
        for f in range(2):
            for w in (0, 1):
                assert nrel(E.get(l, f, w), g.get(f, w)) < 1e-5, (l, f, w)
        for x, y in zip(E.scalars(l), g.scalars()):
            assert abs(x - y) <= 1e-9 * max(1.0, abs(y))
        g.close()


def test_contexts_of_other_sizes_do_not_interfere(P):
    """The kernels' shared-memory limit belongs to the function: a context of a smaller
    lattice made in between must not take it from a larger one's launches."""
    kw = dict(SC, integrator=O.VV2, expansion=O.EXP_SELF, precision=P.FP32)
    a = P.Lattice(O.MODEL_LPHI4_CHI, 96, 0.5, 1.0, 1, P.make_params(**kw))
    ref = P.Lattice(O.MODEL_LPHI4_CHI, 96, 0.5, 1.0, 1, P.make_params(**kw))
    ref.step(4)
    want = ref.get(0, 0)
    small = [P.Lattice(O.MODEL_LPHI4_CHI, n, 0.5, 1.0, 2, P.make_params(**kw)) for n in (8, 64, 24)]
    a.step(4)
    for s in small:
        s.step(3)
    assert np.array_equal(a.get(0, 0), want)
