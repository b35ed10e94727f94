"""Power spectra (row pairs, two axes in fixed point with an exponent per line, shell sums)
against the FP64 oracle over the transform's sizes: powers of two with compiled-in sizes,
mixed radices, columns that do not fill a block; rows whose sizes differ by many orders of
magnitude, rows of zeros, a NaN.  Tolerances as in the other spectrum tests: 1e-10 per bin with
FP64 storage, 1e-5 with FP32 (here the input is the same FP32 field, so 1e-10 as well)."""
import numpy as np
import pytest

import oracle as O
from tests.parity import assert_bins

pytestmark = pytest.mark.gpu

KW = dict(dt=0.005, integrator=O.VV2, q=100.0, phi0=[1.0, 0.0], fluct_amp2=0.0, fstar_over_mp=0.5,
          expansion=O.EXP_OFF)


def field(kind, N):
    x = np.random.default_rng(N).standard_normal((N, N, N))
    if kind == "rows":     # row pairs from 1e-12 to 1
        x *= 10.0 ** (-12.0 * np.random.default_rng(N + 1).random((N, N, 1)))
    elif kind == "plane":  # zeros but one plane
        x[1:] = 0.0
    return x.astype(np.float32).astype(np.float64)


@pytest.mark.parametrize("kind", ["noise", "rows", "plane"])
@pytest.mark.parametrize("N,precision", [(8, 0), (24, 1), (36 * 2, 0), (96, 1), (128, 1), (128, 0)])
def test_spectrum_matches_oracle(N, precision, kind):
    import paper_2102_01031_gb300 as P
    g = P.Lattice(O.MODEL_LPHI4_CHI, N, 0.5, 1.0, 1, P.make_params(precision=precision, **KW))
    o = O.Oracle(O.MODEL_LPHI4_CHI, N, 0.5, 1.0, 1, O.make_params(**KW))
    x = field(kind, N)
    g.set(1, 0, x)
    o.set(1, 0, x)
    kg, dg, mg = g.spectrum(1, 0)
    ko, do, mo = o.spectrum(1, 0)
    assert np.array_equal(mg, mo)
    assert_bins(dg, do, 1e-10, (N, precision, kind))


@pytest.mark.parametrize("precision", [0, 1])
def test_nan_reaches_every_bin(precision):
    import paper_2102_01031_gb300 as P
    N = 24
    g = P.Lattice(O.MODEL_LPHI4, N, 0.5, 1.0, 1, P.make_params(precision=precision, **dict(KW, phi0=[1.0])))
    x = field("noise", N)
    x[3, 5, 7] = np.nan
    g.set(0, 0, x)
    d = g.spectrum(0, 0)[1]
    assert np.all(np.isnan(d[1:])) or np.all(np.isnan(d))
