"""The tensor-core cap stage against the FP64 oracle: rings from the pole to the belt, tiles of
one and of several sectors, ring pairs that go the direct way, belt rings that reach a
cap, and values that its two-part FP16 split cannot carry.

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


def _split(K, nside, theta_arcmin, **opts):
    c = inputs.gaussian_beam(2 * nside, 3.0 * 3518.0 / nside * inputs.ARCMIN)
    tc = theta_arcmin * inputs.ARCMIN
    sp = K.make_split_real(c, nside, tc, **opts)
    return sp, tc, O.hermite_nodes(c, tc, K.split_info(sp)["n_intervals"])


def _pixels(nside, tc, n, seed):
    """Random pixels, two thirds of them in the caps, and whole runs at the poles, where the
    disc reaches the pole, and across the cap / belt boundaries."""
    cap, N = 2 * nside * (nside - 1), 12 * nside * nside
    d = int(tc * nside / 0.8165)  # rings of a disc about the pole
    g = inputs.rng(seed)
    runs = [np.arange(24), np.arange(40) + 2 * d * (d + 1) - 20, np.arange(40) + cap - 20]
    north = np.concatenate(runs + [g.choice(cap, n // 3, replace=False)])
    both = np.concatenate([north, N - 1 - north, g.choice(N, n // 3, replace=False)])
    return np.unique(both[(both >= 0) & (both < N)])


# 256: one sector a ring, wide windows (polar rings mostly direct); 512: one to three
# sectors; 1024: narrow windows
@pytest.mark.parametrize("nside,theta", [(256, 1800.0), (256, 1920.0), (256, 2700.0), (512, 640.0),
                                         (1024, 160.0), (1024, 220.0)])
def test_cap_parity(K, nside, theta):
    sp, tc, tab = _split(K, nside, theta)
    m = inputs.white_noise_map(nside, 91).astype(np.float32)
    x = torch.tensor(m, device="cuda")
    y = torch.full_like(x, float("nan"))
    K.conv_real(sp, x, y)
    K.device_status(sp)
    pix = _pixels(nside, tc, 600, 5)
    ref, amb = O.brute_conv(nside, m.astype(np.float64), tc, table=tab, out_pix=pix)
    err = np.abs(y.cpu().numpy()[pix] - ref) - amb
    assert err.max() <= 1e-6 * np.sqrt(np.mean(ref ** 2))


@pytest.mark.parametrize("scale,offset", [(1.0, 50.0), (1e18, 0.0), (1e-18, 0.0)])
def test_cap_scaled_and_offset_maps(K, scale, offset):
    nside = 256
    sp, tc, tab = _split(K, nside, 1800.0)
    m = (inputs.white_noise_map(nside, 92) * scale + offset).astype(np.float32)
    x = torch.tensor(m, device="cuda")
    y = torch.empty_like(x)
    K.conv_real(sp, x, y)
    pix = _pixels(nside, tc, 400, 6)
    ref, amb = O.brute_conv(nside, m.astype(np.float64), tc, table=tab, out_pix=pix)
    err = np.abs(y.cpu().numpy()[pix] - ref) - amb
    assert err.max() <= 1e-6 * np.sqrt(np.mean(ref ** 2))


@pytest.mark.parametrize("bad", [-1.6375e30, float("inf"), float("nan")])
def test_values_the_split_cannot_carry_stay_local(K, bad):
    """One masked or broken cap pixel: outputs whose disc does not come near it are those of
    the clean map to the parity bound."""
    nside = 512
    sp, tc, tab = _split(K, nside, 640.0)
    m = inputs.white_noise_map(nside, 93).astype(np.float32)
    p_bad = 2 * 200 * 201 + 77
    m[p_bad] = bad
    x = torch.tensor(m, device="cuda")
    y = torch.empty_like(x)
    K.conv_real(sp, x, y)
    K.device_status(sp)
    clean = m.astype(np.float64)
    clean[p_bad] = 0.0
    pix = _pixels(nside, tc, 900, 7)
    vec = O.pix2vec(nside)
    far = pix[np.arccos(np.clip(vec[pix] @ vec[p_bad], -1, 1)) > tc + np.radians(8.0)]
    assert far.size > 200
    ref, amb = O.brute_conv(nside, clean, tc, table=tab, out_pix=far)
    err = np.abs(y.cpu().numpy()[far] - ref) - amb
    assert err.max() <= 1e-6 * np.sqrt(np.mean(ref ** 2))


def test_bands_and_stacks_equal_single_maps(K):
    """Bands that start and end inside a pair of rings, and the maps of a stack, bit for bit."""
    nside = 256
    sp, _, _ = _split(K, nside, 1800.0)
    x = torch.tensor(np.stack([inputs.white_noise_map(nside, 94 + i) for i in range(2)]).astype(
        np.float32), device="cuda")
    y = torch.empty_like(x)
    one = torch.empty_like(x)
    K.conv_real_multimap(sp, x, y, 2)
    for i in range(2):
        K.conv_real(sp, x[i], one[i])
    assert torch.equal(y, one)
    _, _, n, st, _ = O.ring_table(nside)
    nr = 4 * nside - 1
    for lo, hi in ((1, 2), (7, 40), (200, nside + 20), (3 * nside - 5, nr), (100, 100)):
        part = torch.zeros_like(x[0])
        K.conv_real_rings(sp, x[0], part, lo, hi)
        a, b = int(st[lo - 1]), int(st[hi - 1] + n[hi - 1])
        assert torch.equal(part[a:b], one[0][a:b])
        assert not part[:a].any() and not part[b:].any()
