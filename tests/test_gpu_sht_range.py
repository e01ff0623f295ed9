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


# belt rings through the FFT, with and without a radix-2 pass in the halves
@pytest.mark.parametrize("nside,lmax", [(512, 60), (1024, 60)])
def test_faint_rings_keep_their_digits(K, nside, lmax):
    """A broad source in one hemisphere: the other hemisphere's rings, 1e-3 of their mirrors, to 3e-6 of
    their own rms (a handful of FP32 roundings of their own values, not of their mirrors')."""
    sigma, t0 = np.radians(16.0), np.radians(118.0)  # the source's width and colatitude
    z, s, n, _, phase = O.ring_table(nside)
    ring = np.repeat(np.arange(n.size), n.astype(int))
    k = np.concatenate([np.arange(int(c)) for c in n])
    phi = (2.0 * k + phase[ring]) * np.pi / n[ring]
    cosd = z[ring] * np.cos(t0) + s[ring] * np.sin(t0) * np.cos(phi)
    alm = O.map2alm(nside, np.exp((cosd - 1.0) / sigma ** 2), lmax)
    ref = O.alm2map(nside, alm, lmax)
    y = torch.empty(12 * nside * nside, device="cuda")
    K.sht_alm2map(nside, lmax, torch.tensor(alm, device="cuda"), y)
    err = y.cpu().numpy().astype(np.float64) - ref
    r = np.flatnonzero((np.arange(n.size) > nside) & (np.arange(n.size) < 2 * nside - 1))  # northern belt
    start = np.concatenate([[0], np.cumsum(n)]).astype(int)
    rms = np.array([np.sqrt(np.mean(ref[start[i]:start[i + 1]] ** 2)) for i in r])
    bright = np.array([np.sqrt(np.mean(ref[start[j]:start[j + 1]] ** 2)) for j in n.size - 1 - r])
    worst = np.array([np.abs(err[start[i]:start[i + 1]]).max() for i in r])
    faint = rms < 0.02 * bright
    assert faint.sum() > 50
    assert (worst[faint] <= 3e-6 * rms[faint]).all()


@pytest.mark.parametrize("scale", [1e40, 1e44])
def test_coefficients_keep_the_range_of_a_double(K, scale):
    """One sectoral coefficient past FP32's range: rings where its function takes it back into that
    range, to 2e-6 of the ring's largest pixel (functions below 2^-60 count as zero: not the rings
    where less than 1e6 of that is left)."""
    nside, lmax = 64, 128
    alm = inputs.grf_alm(lmax, inputs.cl_grf(lmax), 7)
    alm[lmax * (2 * lmax + 1 - lmax) // 2 + lmax] = scale  # l = m = l_max
    ref = O.alm2map(nside, alm, lmax)
    y = torch.empty(12 * nside * nside, device="cuda")
    K.sht_alm2map(nside, lmax, torch.tensor(alm, device="cuda"), y)
    got = y.cpu().numpy().astype(np.float64)
    _, _, n, start, _ = O.ring_table(nside)
    checked = 0
    for st, c in zip(start.astype(int), n.astype(int)):
        top = np.abs(ref[st:st + c]).max()
        if 1e6 * 2.0 ** -60 * scale < top < 1e37:
            checked += 1
            assert np.abs(got[st:st + c] - ref[st:st + c]).max() <= 2e-6 * top
    assert checked >= 4


def test_analysis_of_a_map_near_the_smallest_floats(K):
    """A map of values about 1e-36: the a_lm of the same map about one, scaled, to 1e-6 of the largest."""
    nside, lmax = 64, 128
    m = torch.tensor(inputs.white_noise_map(nside, 21).astype(np.float32), device="cuda")
    one = torch.zeros(K.n_alm(lmax), dtype=torch.complex128, device="cuda")
    low = torch.zeros_like(one)
    K.sht_map2alm(nside, lmax, m, one)
    K.sht_map2alm(nside, lmax, m * 2.0 ** -119, low)
    assert (low * 2.0 ** 119 - one).abs().max() <= 1e-6 * one.abs().max()
