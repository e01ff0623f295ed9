"""The transforms' ring sums (FFT of the belt, quarter sums of the caps) and FP32-pair
recurrences where their tiles and branches change: belts too short for the FFT, FFTs
with and without a radix-2 pass, orders at and past the ring length (l_max = 4 nside), one and
several rings a thread, more orders than one staged block.

Bounds: a radix-4 pass rounds each value about three times (3 x 2^-25 rms relative to the
sequence's rms), the passes add in quadrature (7 at most here), so 2.4e-7 rms; the largest of
up to 8e5 pixels is within 5.2 rms, 1.3e-6, and the cap sums (twiddles one ulp off per step of
an 8-step anchor) are below that: 2e-6 of the map's rms.  a_lm average over rings: 2e-6 of the
largest."""
import numpy as np
import pytest

import oracle as O
from paper_1409_4441_gb300 import inputs

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def K():
    import __graft_entry__
    __graft_entry__.build()
    from paper_1409_4441_gb300 import ksconv
    return ksconv


@pytest.mark.parametrize("nside,lmax", [(2, 8), (4, 16), (16, 64), (32, 128), (256, 300),
                                        (256, 1024), (512, 40),
                                        (512, 60)])
def test_transforms_match_oracle(K, nside, lmax):
    alm = inputs.grf_alm(lmax, inputs.cl_grf(lmax), inputs.seed_for(7, nside + lmax))
    ref = O.alm2map(nside, alm, lmax)
    d_alm = torch.tensor(alm, dtype=torch.complex128, device="cuda")
    y = torch.empty(12 * nside * nside, dtype=torch.float32, device="cuda")
    K.sht_alm2map(nside, lmax, d_alm, y)
    got = y.cpu().numpy().astype(np.float64)
    assert np.abs(got - ref).max() <= 2e-6 * np.sqrt(np.mean(ref ** 2))
    m = ref.astype(np.float32)
    back = torch.zeros_like(d_alm)
    K.sht_map2alm(nside, lmax, torch.tensor(m, device="cuda"), back)
    want = O.map2alm(nside, m.astype(np.float64), lmax)
    assert np.abs(back.cpu().numpy() - want).max() <= 2e-6 * np.abs(want).max()
