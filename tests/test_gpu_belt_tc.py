"""The tensor-core belt stage against the FP64 oracle at the edges of its tiles: ragged ring
blocks (2 nside + 1 belt rings in blocks of 16), every tile width, windows from a few
positions to many chunks, and values that its two-part FP16 split cannot carry.

Tolerance: the per-pixel parity bound of the other kernels, 1e-6 of the output rms plus the
oracle's bound on pairs whose chord lies within rounding of the cut.
"""
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


def _split(K, nside, theta_arcmin, lmax=None, **opts):
    c = inputs.gaussian_beam(lmax or 2 * nside, 3.0 * 3518.0 / nside * inputs.ARCMIN)
    tc = theta_arcmin * inputs.ARCMIN
    sp = K.make_split_real(c, nside, tc, **opts)
    return sp, tc, O.hermite_nodes(c, tc, K.split_info(sp)["n_intervals"])


def _belt_pixels(nside, n, seed):
    """Random belt pixels, with the first and last pixels of the first, last and middle rings."""
    cap, L = 2 * nside * (nside - 1), 4 * nside
    belt = (2 * nside + 1) * L
    edge = [r * L + k for r in (0, 15, 16, nside, 2 * nside - 1, 2 * nside) for k in (0, 7, 8, L - 1)]
    return np.unique(np.concatenate([edge, inputs.rng(seed).choice(belt, n, replace=False)])) + cap


# (nside, cut in arcmin): several tile widths, one chunk to many, and a window wide enough
# to be close to a whole ring
@pytest.mark.parametrize("nside,theta", [(64, 4200.0), (128, 640.0), (128, 2400.0), (256, 220.0),
                                         (256, 640.0), (512, 60.0), (1024, 40.0)])
def test_belt_parity(K, nside, theta):
    sp, tc, tab = _split(K, nside, theta)
    m = inputs.white_noise_map(nside, 77).astype(np.float32)
    x = torch.tensor(m, device="cuda")
    y = torch.full_like(x, float("nan"))
    K.conv_real(sp, x, y)
    K.device_status(sp)
    pix = _belt_pixels(nside, 1500 if nside <= 256 else 500, 5)
    ref, amb = O.brute_conv(nside, m.astype(np.float64), tc, table=tab, out_pix=pix)
    err = np.abs(y.cpu().numpy()[pix] - ref) - amb
    assert err.max() <= 1e-6 * np.sqrt(np.mean(ref ** 2))


@pytest.mark.parametrize("scale,offset", [(1.0, 50.0), (1e18, 0.0), (1e-18, 0.0), (1e-3, -4.0)])
def test_belt_scaled_and_offset_maps(K, scale, offset):
    nside = 256
    sp, tc, tab = _split(K, nside, 640.0)
    m = (inputs.white_noise_map(nside, 78) * scale + offset).astype(np.float32)
    x = torch.tensor(m, device="cuda")
    y = torch.empty_like(x)
    K.conv_real(sp, x, y)
    pix = _belt_pixels(nside, 1000, 6)
    ref, amb = O.brute_conv(nside, m.astype(np.float64), tc, table=tab, out_pix=pix)
    err = np.abs(y.cpu().numpy()[pix] - ref) - amb
    assert err.max() <= 1e-6 * np.sqrt(np.mean(ref ** 2))


@pytest.mark.parametrize("bad", [-1.6375e30, float("inf"), float("nan")])
def test_values_the_split_cannot_carry_stay_local(K, bad):
    """One masked or broken pixel: outputs whose disc does not come near it are those of the
    clean map to the parity bound; a zeroed region changes nothing about the path."""
    nside = 256
    sp, tc, tab = _split(K, nside, 640.0)
    m = inputs.white_noise_map(nside, 79).astype(np.float32)
    cap, L = 2 * nside * (nside - 1), 4 * nside
    p_bad = cap + nside * L + 300
    m[p_bad] = bad
    m[cap + 40 * L: cap + 60 * L] = 0.0
    x = torch.tensor(m, device="cuda")
    y = torch.empty_like(x)
    K.conv_real(sp, x, y)
    K.device_status(sp)
    clean = m.astype(np.float64)
    clean[p_bad] = 0.0
    pix = _belt_pixels(nside, 3000, 7)
    vec = O.pix2vec(nside)
    # past the cut and the padding of a window (26 positions of an eighth of a degree)
    far = pix[np.arccos(np.clip(vec[pix] @ vec[p_bad], -1, 1)) > tc + np.radians(12.0)]
    assert far.size > 1000
    ref, amb = O.brute_conv(nside, clean, tc, table=tab, out_pix=far)
    err = np.abs(y.cpu().numpy()[far] - ref) - amb
    assert err.max() <= 1e-6 * np.sqrt(np.mean(ref ** 2))


def test_bands_and_stacks_equal_single_maps(K):
    """Bands that start and end inside a block of rings, and the maps of a stack, bit for bit."""
    nside = 128
    sp, _, _ = _split(K, nside, 700.0)
    x = torch.tensor(np.stack([inputs.white_noise_map(nside, 80 + i) for i in range(3)]).astype(
        np.float32), device="cuda")
    y = torch.empty_like(x)
    one = torch.empty_like(x)
    K.conv_real_multimap(sp, x, y, 3)
    for i in range(3):
        K.conv_real(sp, x[i], one[i])
    assert torch.equal(y, one)
    nr = 4 * nside - 1
    z, s, n, st, _ = O.ring_table(nside)
    for lo, hi in ((nside + 5, nside + 40), (nside, nside), (3 * nside - 3, 3 * nside + 9), (1, nr)):
        part = torch.zeros_like(x[0])
        K.conv_real_rings(sp, x[0], part, lo, hi)
        a, b = int(st[lo - 1]), int(st[hi - 1] + n[hi - 1])
        assert torch.equal(part[a:b], one[0][a:b])
        assert not part[:a].any() and not part[b:].any()
