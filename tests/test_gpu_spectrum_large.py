"""Power spectra at the sizes whose transforms are compiled in (256^3, 512^3; FP32 and FP64 rows)
against torch's FFT of the same field in FP64, binned the same way.

Tolerance as in the other spectrum tests, 1e-10 per bin: both transforms round at about 1e-15 of
their lines' sizes, a bin sums at least 6 modes of a white spectrum."""
import math

import numpy as np
import pytest

import oracle as O
from tests.parity import assert_bins

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("N,precision", [(256, 1), (256, 0), (512, 1), (512, 0)])
def test_spectrum_matches_torch_fft(N, precision):
    import torch

    import paper_2102_01031_gb300 as P
    kIR, dk = 0.5, 1.0
    g = P.Lattice(O.MODEL_LPHI4, N, kIR, 1.0, 1, P.make_params(
        dt=0.005, integrator=O.VV2, phi0=[1.0], fluct_amp2=0.0, fstar_over_mp=0.5, expansion=O.EXP_OFF,
        precision=precision))
    gen = torch.Generator(device="cuda").manual_seed(N + precision)
    # FP32 values, so that both precisions store the same field
    x = torch.randn((N, N, N), generator=gen, device="cuda", dtype=torch.float32).double()
    g.set_device(0, 0, x.data_ptr())
    torch.cuda.synchronize()
    k, d, m = g.spectrum(0, 0, dk)
    n1 = torch.fft.fftfreq(N, 1.0 / N, device="cuda", dtype=torch.float64)
    nb = len(d)
    sp, sn, ct = (torch.zeros(nb, dtype=torch.float64, device="cuda") for _ in range(3))
    F = torch.fft.fftn(x)
    del x
    for z in range(N):  # a plane at a time: the index arrays of a whole lattice are larger than it
        n2 = n1[z] ** 2 + n1[:, None] ** 2 + n1[None, :] ** 2
        n = n2.sqrt().view(-1)
        b = (n / dk).floor().long().clamp_(max=nb - 1)
        keep = n > 0
        sp.index_add_(0, b[keep], F[z].abs().square().view(-1)[keep])
        sn.index_add_(0, b[keep], n[keep])
        ct.index_add_(0, b[keep], torch.ones_like(n[keep]))
    nbar = sn / ct.clamp(min=1.0)
    kb = kIR * nbar
    dx = 2.0 * math.pi / (N * kIR)
    want = kb ** 3 / (2.0 * math.pi ** 2) * (dx / N) ** 3 * sp / (4.0 * math.pi * nbar.clamp(min=0.1) ** 2)
    want = torch.where(ct > 0, want, torch.zeros_like(want)).cpu().numpy()
    assert np.array_equal(np.asarray(m, dtype=np.float64), ct.cpu().numpy())
    assert_bins(d, want, 1e-10, (N, precision))
