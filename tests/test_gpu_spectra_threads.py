"""Spectra of two lattice sizes from two host threads at once.  The transforms' kernels for sizes
that are not compiled in are shared, and so is their shared-memory limit: a small lattice's launch
must not lower it between another thread's setting and launch.  Results equal a single thread's
but for the order of the shells' additions (at most 2^17 positive terms a bin: 1e-11)."""
import threading

import numpy as np
import pytest

import oracle as O

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("precision", [0, 1])
def test_spectra_of_two_sizes_from_two_threads(precision):
    import paper_2102_01031_gb300 as P
    kw = dict(dt=0.005, integrator=O.VV2, q=100.0, phi0=[1.0, 0.0], fluct_amp2=1e-4, fstar_over_mp=0.5,
              expansion=O.EXP_OFF, precision=precision)
    lats = [P.Lattice(O.MODEL_LPHI4_CHI, n, 0.5, 1.0, 1, P.make_params(**kw)) for n in (24, 96)]
    want = [(g.spectrum(0, 0)[1], g.occupation(1)[1]) for g in lats]
    errors = []

    def work(k):
        try:
            for _ in range(150):
                got = (lats[k].spectrum(0, 0)[1], lats[k].occupation(1)[1])
                for a, b in zip(got, want[k]):
                    np.testing.assert_allclose(a, b, rtol=1e-11)
        except Exception as e:  # noqa: BLE001 (reported by the test below)
            errors.append(e)

    threads = [threading.Thread(target=work, args=(k,)) for k in range(2)]
    for t in threads:
        t.start()
    for t in threads:
        t.join()
    assert not errors, errors[0]
