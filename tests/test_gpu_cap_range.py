"""The tensor-core cap stage where a kernel or a map is outside what its FP16 operands carry.

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


def _legendre(lmax, z):
    p = np.zeros(lmax + 1)
    p[0], p[1] = 1.0, z
    for l in range(2, lmax + 1):
        p[l] = ((2 * l - 1) * z * p[l - 1] - (l - 1) * p[l - 2]) / l
    return p


def _cap_pixels(nside, n, seed):
    cap, N = 2 * nside * (nside - 1), 12 * nside * nside
    north = np.concatenate([np.arange(24), inputs.rng(seed).choice(cap, n, replace=False)])
    return np.unique(np.concatenate([north, N - 1 - north]))


# A ring of 2.5 pixels FWHM around the cut: the kernel rises past the cut, where the edge cells'
# polynomials reach (up to 1.1e5 in units that put the largest value inside the cut at 2^13).
def test_kernel_that_rises_past_the_cut(K):
    nside, tc = 512, 640.0 * inputs.ARCMIN
    pixel = 3518.0 / nside * inputs.ARCMIN
    c = inputs.gaussian_beam(2 * nside, 2.5 * pixel) * _legendre(2 * nside, np.cos(tc + 3.5 * pixel))
    with K.make_split_real(c, nside, tc) as sp:
        m = inputs.white_noise_map(nside, 191).astype(np.float32)
        x = torch.tensor(m, device="cuda")
        y = torch.empty_like(x)
        K.conv_real(sp, x, y)
        K.device_status(sp)
        tab = O.hermite_nodes(c, tc, K.split_info(sp)["n_intervals"])
    pix = _cap_pixels(nside, 300, 5)
    ref, amb = O.brute_conv(nside, m.astype(np.float64), tc, table=tab, out_pix=pix)
    err = np.abs(y.cpu().numpy()[pix] - ref) - amb
    assert err.max() <= 1e-6 * np.sqrt(np.mean(ref ** 2))


def _far_from_ring_97(nside, tc):
    """A pixel of ring 98 (from 1) of nside 256, whose windows there are wider than any tile's, and pixels
    of the rings around it on the far side of the pole, beyond the cut."""
    z, _, n, st, _ = O.ring_table(nside)
    bad = int(st[97])
    pix = np.concatenate([np.arange(st[r] + int(0.43 * n[r]), st[r] + int(0.57 * n[r])) for r in range(85, 125)])
    vec = O.pix2vec(nside)
    return bad, pix[np.arccos(np.clip(vec[pix] @ vec[bad], -1, 1)) > tc + np.radians(2.0)]


@pytest.mark.parametrize("bad", [-1.6375e30, float("inf"), float("nan")])
def test_polar_value_past_the_cut_stays_out(K, bad):
    nside, tc = 256, 1800.0 * inputs.ARCMIN
    c = inputs.gaussian_beam(2 * nside, 3.0 * 3518.0 / nside * inputs.ARCMIN)
    p_bad, far = _far_from_ring_97(nside, tc)
    assert far.size > 500
    m = inputs.white_noise_map(nside, 193).astype(np.float32)
    clean = m.astype(np.float64)
    m[p_bad], clean[p_bad] = bad, 0.0
    with K.make_split_real(c, nside, tc) as sp:
        x = torch.tensor(m, device="cuda")
        y = torch.empty_like(x)
        K.conv_real(sp, x, y)
        K.device_status(sp)
        tab = O.hermite_nodes(c, tc, K.split_info(sp)["n_intervals"])
    ref, amb = O.brute_conv(nside, clean, tc, table=tab, out_pix=far)
    err = np.abs(y.cpu().numpy()[far] - ref) - amb
    assert err.max() <= 1e-6 * np.sqrt(np.mean(ref ** 2))


@pytest.mark.parametrize("bad", [1e8, float("nan")])
def test_polar_value_does_not_set_the_constant(K, bad):
    """A map about 50: what a tile takes off its input rings comes from those rings, not from one that
    its products leave out."""
    nside, tc = 256, 1800.0 * inputs.ARCMIN
    c = inputs.gaussian_beam(2 * nside, 3.0 * 3518.0 / nside * inputs.ARCMIN)
    p_bad, far = _far_from_ring_97(nside, tc)
    m = (inputs.white_noise_map(nside, 194) + 50.0).astype(np.float32)
    clean = m.astype(np.float64)
    m[p_bad], clean[p_bad] = bad, 0.0
    with K.make_split_real(c, nside, tc) as sp:
        x = torch.tensor(m, device="cuda")
        y = torch.empty_like(x)
        K.conv_real(sp, x, y)
        K.device_status(sp)
        tab = O.hermite_nodes(c, tc, K.split_info(sp)["n_intervals"])
    ref, amb = O.brute_conv(nside, clean, tc, table=tab, out_pix=far)
    err = np.abs(y.cpu().numpy()[far] - ref) - amb
    assert err.max() <= 1e-6 * np.sqrt(np.mean(ref ** 2))


def test_positive_map_has_no_bias(K):
    """Products of one sign and a kernel whose lobes cancel: the mean relative error of belt and of
    cap outputs stays below the FP32 spacing of the result, 2^-23 (rounding to nearest leaves a
    few tenths of it, the scale factors' own)."""
    nside, tc = 1024, 400.0 * inputs.ARCMIN
    ell = np.arange(2 * nside + 1)
    b = inputs.gaussian_beam(2 * nside, 10.0 * inputs.ARCMIN)
    z, _, n, _, _ = O.ring_table(nside)
    g = inputs.rng(195).standard_normal(12 * nside * nside)
    m = (np.exp(2.5 * np.repeat(z, n.astype(int)) + 0.3 * g) + 0.01).astype(np.float32)
    with K.make_split(b, nside, 512, tc, cl_in=1.0 / (ell + 10.0) ** 2) as sp:
        x = torch.tensor(m, device="cuda")
        y = torch.empty_like(x)
        K.conv_real(sp, x, y)
        K.device_status(sp)
        tab = O.hermite_nodes(K.split_real_coeffs(sp), tc, K.split_info(sp)["n_intervals"])
    cap, N = 2 * nside * (nside - 1), 12 * nside * nside
    for lo, hi in ((cap, N - cap), (0, cap)):
        pix = np.sort(inputs.rng(196).choice(np.arange(lo, hi), 700, replace=False))
        ref, amb = O.brute_conv(nside, m.astype(np.float64), tc, table=tab, out_pix=pix)
        d = y.cpu().numpy()[pix] - ref
        rel = np.sign(d) * np.maximum(np.abs(d) - amb, 0.0) / np.abs(ref)
        assert abs(rel.mean()) <= 2.0 ** -23


# wide windows that are mostly the stage's own, and wide ones that near the poles go the direct way
@pytest.mark.parametrize("nside,lcut,theta", [(512, 384, 480.0), (256, -1, 1800.0)])
def test_cap_pixels_are_as_accurate_as_the_gather(K, nside, lcut, theta):
    """Error rms against 64 bits over 4000 pixels of the caps, the stage and the gather with every
    weight from the chord on the same map: no larger but for the scatter of such an rms (1.1% each:
    10% is six times the two together)."""
    tc, lmax = theta * inputs.ARCMIN, (3 if lcut > 0 else 2) * nside - 1
    b = inputs.gaussian_beam(lmax, (4.4 if lcut > 0 else 3.0) * 3518.0 / nside * inputs.ARCMIN)
    ell = np.arange(lmax + 1)
    m = inputs.white_noise_map(nside, 197).astype(np.float32)
    x = torch.tensor(m, device="cuda")
    pix = _cap_pixels(nside, 2000, 8)
    rms = []
    for exact in (0, 1):
        with (K.make_split(b, nside, lcut, tc, cl_in=1.0 / (ell + 10.0) ** 2, exact_weights=exact) if lcut > 0
              else K.make_split_real(b, nside, tc, exact_weights=exact)) as sp:
            y = torch.empty_like(x)
            K.conv_real(sp, x, y)
            K.device_status(sp)
            if not exact:
                tab = O.hermite_nodes(K.split_real_coeffs(sp), tc, K.split_info(sp)["n_intervals"])
                ref, amb = O.brute_conv(nside, m.astype(np.float64), tc, table=tab, out_pix=pix)
        err = np.maximum(np.abs(y.cpu().numpy()[pix] - ref) - amb, 0.0)
        rms.append(np.sqrt(np.mean(err ** 2)))
    assert rms[0] <= 1.1 * rms[1]


def test_coefficients_leave_the_device_to_others(K):
    """The stage's coefficients take at most an eighth of the free memory: beside a program that leaves
    less, the split is made without them and gives the same outputs, to 1e-6 of their rms in the rms
    (single pixels have pairs whose chord lies within rounding of the cut)."""
    nside, tc = 1024, 400.0 * inputs.ARCMIN
    c = inputs.gaussian_beam(2 * nside, 3.0 * 3518.0 / nside * inputs.ARCMIN)
    x = torch.tensor(inputs.white_noise_map(nside, 198).astype(np.float32), device="cuda")
    y, z = torch.empty_like(x), torch.empty_like(x)

    def used():
        torch.cuda.synchronize()
        free, total = torch.cuda.mem_get_info()
        return total - free

    before = used()
    with K.make_split_real(c, nside, tc) as sp:
        assert K.split_stages(sp)["cap_stage"] == 1
        size = used() - before
        K.conv_real(sp, x, y)
    torch.cuda.empty_cache()
    hold = torch.empty(torch.cuda.mem_get_info()[0] - 4 * size, dtype=torch.uint8, device="cuda")
    with K.make_split_real(c, nside, tc) as sp:
        assert K.split_stages(sp)["cap_stage"] == 0
        K.conv_real(sp, x, z)
        K.device_status(sp)
    del hold
    torch.cuda.empty_cache()
    assert size > 1 << 28
    assert (y - z).double().square().mean().sqrt() <= 1e-6 * z.double().square().mean().sqrt()
