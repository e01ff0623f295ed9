"""Which kernels a split runs, and the tensor-core stages against the FP64 oracle at sizes that are
known to be theirs: every tile width of the belt stage, ragged ring blocks, bands and stacks.

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
    return K.make_split_real(c, nside, theta_arcmin * inputs.ARCMIN, **opts), c


def _launched(K, sp, x, y):
    """Kernels of one ksc_conv_real, by name."""
    from torch.profiler import ProfilerActivity, profile
    for _ in range(2):  # (the first profile of a process may record nothing)
        with profile(activities=[ProfilerActivity.CUDA]) as p:
            K.conv_real(sp, x, y)
            torch.cuda.synchronize()
    return [e.name for e in p.events() if "kernel" in e.name]


# (nside, cut in arcmin): neither stage, the belt's, both
@pytest.mark.parametrize("nside,theta", [(64, 360.0), (512, 240.0), (512, 640.0)])
def test_reported_kernels_are_the_ones_that_run(K, nside, theta):
    sp, _ = _split(K, nside, theta)
    x = torch.tensor(inputs.white_noise_map(nside, 11).astype(np.float32), device="cuda")
    with sp:
        names = _launched(K, sp, x, torch.empty_like(x))
        st = K.split_stages(sp)
    assert len(names) == st["n_launches"], names
    assert any("conv_belt_tc_kernel" in n for n in names) == (st["belt_columns"] > 0)
    assert any("conv_cap_tc_kernel" in n for n in names) == (st["cap_stage"] == 1)


def _legendre(lmax, z):
    p = np.zeros(lmax + 1)
    p[0], p[1] = 1.0, z
    for l in range(2, lmax + 1):
        p[l] = ((2 * l - 1) * z * p[l - 1] - (l - 1) * p[l - 2]) / l
    return p


def test_cap_stage_takes_kernels_that_its_polynomials_carry(K):
    """At one nside and cut: a beam of three pixels with l_max = 2 nside; the same with l_max =
    3 nside, whose sixth-order coefficients are above the 2^-12 of the peak that one FP16 part may
    leave; a ring of 2.5 pixels FWHM five pixels past the cut, of which the interpolation keeps
    5e-6 of what lies within."""
    nside, tc = 512, 640.0 * inputs.ARCMIN
    pixel = 3518.0 / nside * inputs.ARCMIN
    ring = inputs.gaussian_beam(2 * nside, 2.5 * pixel) * _legendre(2 * nside, np.cos(tc + 5.0 * pixel))
    for c, want in ((inputs.gaussian_beam(2 * nside, 3.0 * pixel), 1),
                    (inputs.gaussian_beam(3 * nside - 1, 3.0 * pixel), 0), (ring, 0)):
        with K.make_split_real(c, nside, tc) as sp:
            assert K.split_stages(sp)["cap_stage"] == want


# (nside, cut in arcmin, whether the stage was measured to be the faster one)
@pytest.mark.parametrize("nside,theta,want", [(256, 1800.0, 1), (512, 660.0, 1), (2048, 110.0, 1),
                                              (2048, 28.0, 0), (2048, 55.0, 0), (256, 7040.0, 0)])
def test_cap_stage_is_taken_where_it_is_faster(K, nside, theta, want):
    """Narrow windows, of which a tile costs as much as of wide ones, and cuts whose cap ring pairs
    all go the direct way, are the gather's (2048, 28': 6.9 against 5.2 ms; 256, 7040': 214
    against 153 ms)."""
    sp, _ = _split(K, nside, theta)
    with sp:
        assert K.split_stages(sp)["cap_stage"] == want
