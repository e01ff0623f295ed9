"""The transforms where their shortcuts could show: memory that a call leaves unwritten, rings of unlike
brightness in the two hemispheres, coefficients and maps far from one, and the FFT lengths and the
direct sums of the largest maps."""
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


def _alm(lmax, seed):
    return torch.tensor(inputs.grf_alm(lmax, inputs.cl_grf(lmax), seed), dtype=torch.complex128, device="cuda")


@pytest.mark.parametrize("nside,lmax", [(8, 19), (64, 200), (256, 700), (512, 1201)])
def test_nothing_unwritten_is_read(K, nside, lmax):
    """Orders past a ring's limit are neither written nor read: a call whose scratch held NaN before
    (that of a larger transform of NaN, freed on the same stream) gives the bits of one that did not."""
    npix = 12 * nside * nside
    alm, bad = _alm(lmax, 5), torch.full((K.n_alm(4 * nside),), float("nan"), dtype=torch.complex128, device="cuda")
    clean, got, back, back2 = (torch.zeros(npix, device="cuda"), torch.zeros(npix, device="cuda"),
                               torch.zeros_like(alm), torch.zeros_like(alm))
    K.sht_alm2map(nside, lmax, alm, clean)
    K.sht_map2alm(nside, lmax, clean, back)
    torch.cuda.synchronize()
    K.sht_alm2map(nside, 4 * nside, bad, got)
    K.sht_alm2map(nside, lmax, alm, got)
    K.sht_alm2map(nside, 4 * nside, bad, torch.zeros(npix, device="cuda"))
    K.sht_map2alm(nside, lmax, clean, back2)
    torch.cuda.synchronize()
    assert torch.equal(got, clean) and torch.equal(back, back2)
    assert torch.isfinite(clean).all()
