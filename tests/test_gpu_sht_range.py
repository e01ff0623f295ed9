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
    phi = phase[ring] + 2.0 * np.pi * k / n[ring]
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


def _lambda(lmax, z):
    """lambda_lm(z) as [l, m], no Condon-Shortley phase."""
    lam = np.zeros((lmax + 1, lmax + 1))
    s = np.sqrt((1.0 - z) * (1.0 + z))
    lam[0, 0] = np.sqrt(1.0 / (4.0 * np.pi))
    for m in range(1, lmax + 1):
        lam[m, m] = lam[m - 1, m - 1] * s * np.sqrt((2.0 * m + 1.0) / (2.0 * m))
    for m in range(lmax + 1):
        for l in range(m + 1, lmax + 1):
            a = np.sqrt((4.0 * l * l - 1.0) / (l * l - m * m))
            b = np.sqrt(((l - 1.0) ** 2 - m * m) / (4.0 * (l - 1.0) ** 2 - 1.0)) * lam[l - 2, m] if l > m + 1 else 0.0
            lam[l, m] = a * (z * lam[l - 1, m] - b)
    return lam


# FFT lengths 8192 and 16384, then belt rings too long for it
@pytest.mark.parametrize("nside", [2048, 4096, 8192])
def test_longest_rings(K, nside):
    """Synthesis on rings of every kind, and the analysis of single pixels (a_lm = 4 pi / N lambda_lm
    e^{-i m phi}), each to 2e-6 of the largest."""
    lmax, npix = 24, 12 * nside * nside
    alm = _alm(lmax, 9)
    flat = alm.cpu().numpy()
    a = np.zeros((lmax + 1, lmax + 1), complex)
    at = 0
    for m in range(lmax + 1):
        a[m:, m] = flat[at:at + lmax + 1 - m]
        at += lmax + 1 - m
    z, _, n, start, phase = O.ring_table(nside)
    y = torch.zeros(npix, device="cuda")
    K.sht_alm2map(nside, lmax, alm, y)
    ms = np.arange(lmax + 1)
    for r in (0, 5, nside // 2, nside - 2, nside - 1, nside, 2 * nside - 1, 2 * nside, 3 * nside, 4 * nside - 2):
        c = int(n[r])
        phi = phase[r] + 2.0 * np.pi * np.arange(c) / c
        g = (_lambda(lmax, z[r]) * a).sum(0) * np.where(ms > 0, 2.0, 1.0)
        want = (g[None, :] * np.exp(1j * np.outer(phi, ms))).real.sum(1)
        got = y[int(start[r]):int(start[r]) + c].cpu().numpy()
        assert np.abs(got - want).max() <= 2e-6 * np.abs(want).max()
    back = torch.zeros_like(alm)
    for r in (nside // 2, nside - 1, 2 * nside - 1, 2 * nside + 7):
        k = int(n[r]) // 3
        y.zero_()
        y[int(start[r]) + k] = 1.0
        K.sht_map2alm(nside, lmax, y, back)
        phi = phase[r] + 2.0 * np.pi * k / int(n[r])
        want = 4.0 * np.pi / npix * _lambda(lmax, z[r]) * np.exp(-1j * ms * phi)[None, :]
        want = np.concatenate([want[m:, m] for m in range(lmax + 1)])
        assert np.abs(back.cpu().numpy() - want).max() <= 2e-6 * np.abs(want).max()
