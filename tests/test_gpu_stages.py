"""Which kernels a split runs, and the tensor-core stages against the FP64 oracle at sizes that are
known to be theirs: every tile width of the belt stage, ragged ring blocks, bands and stacks.

Tolerance: the per-pixel parity bound of the other kernels, 1e-6 of the output rms plus the
oracle's bound on pairs whose chord lies within rounding of the cut.
"""
import json
import os
import subprocess
import sys

import numpy as np
import pytest

import oracle as O
from paper_1409_4441_gb300 import inputs

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu
ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))


@pytest.fixture(scope="module")
def K():
    import __graft_entry__
    __graft_entry__.build()
    from paper_1409_4441_gb300 import ksconv
    return ksconv


def _split(K, nside, theta_arcmin, **opts):
    c = inputs.gaussian_beam(2 * nside, 3.0 * 3518.0 / nside * inputs.ARCMIN)
    return K.make_split_real(c, nside, theta_arcmin * inputs.ARCMIN, **opts), c


# Kernels by name of calls on splits of this file's beam, from a process of its own (a profiler in
# this one would stay under the graphs that other tests replay).
PROBE = """
import json, sys
import torch
from torch.profiler import ProfilerActivity, profile
from paper_1409_4441_gb300 import inputs, ksconv as K
out = []
for nside, theta, tensor, n_maps, lo, hi in json.loads(sys.argv[1]):
    c = inputs.gaussian_beam(2 * nside, 3.0 * 3518.0 / nside * inputs.ARCMIN)
    sp = K.make_split_real(c, nside, theta * inputs.ARCMIN, tensor=tensor)
    x = torch.randn((n_maps, 12 * nside * nside), device="cuda")
    y = torch.empty_like(x)
    for _ in range(2):  # (the first profile of a process may record nothing)
        with profile(activities=[ProfilerActivity.CUDA]) as p:
            if hi:
                K.conv_real_rings(sp, x[0], y[0], lo, hi)
            elif n_maps > 1:
                K.conv_real_multimap(sp, x, y, n_maps)
            else:
                K.conv_real(sp, x[0], y[0])
            torch.cuda.synchronize()
    out.append({"names": [e.name for e in p.events() if "kernel" in e.name], "stages": K.split_stages(sp)})
    sp.close()
print(json.dumps(out))
"""


def _launched(cases):
    run = subprocess.run([sys.executable, "-c", PROBE, json.dumps(cases)], capture_output=True, text=True,
                         timeout=300, cwd=ROOT)
    assert run.returncode == 0, run.stderr[-2000:]
    return json.loads(run.stdout.splitlines()[-1])


def test_reported_kernels_are_the_ones_that_run(K):
    """Neither stage, the belt's, both."""
    for r in _launched([(64, 360.0, 0, 1, 0, 0), (512, 240.0, 0, 1, 0, 0), (512, 640.0, 0, 1, 0, 0)]):
        names, st = r["names"], r["stages"]
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
    """At one nside and cut: a beam of three pixels with l_max = 2 nside and 3 nside; one of 2.2
    pixels with l_max = 3 nside, whose sixth-order coefficients are above the 2^-10.5 of the peak
    that one FP16 part may serve; a ring of 2.5 pixels FWHM five pixels past the cut, of which the interpolation keeps
    5e-6 of what lies within."""
    nside, tc = 512, 640.0 * inputs.ARCMIN
    pixel = 3518.0 / nside * inputs.ARCMIN
    ring = inputs.gaussian_beam(2 * nside, 2.5 * pixel) * _legendre(2 * nside, np.cos(tc + 5.0 * pixel))
    for c, want in ((inputs.gaussian_beam(2 * nside, 3.0 * pixel), 1),
                    (inputs.gaussian_beam(3 * nside - 1, 3.0 * pixel), 1),
                    (inputs.gaussian_beam(3 * nside - 1, 2.2 * pixel), 0), (ring, 0)):
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


def test_calls_take_only_what_their_stages_need(K):
    """A cap band of a split with a belt stage, and a stack whose stages are both the TF32 kernels: no
    block maxima.  A belt band: one launch of them."""
    cap, belt, stack = _launched([(256, 900.0, 0, 1, 100, 140), (256, 900.0, 0, 1, 500, 540),
                                  (256, 900.0, 2, 16, 0, 0)])
    assert cap["stages"]["belt_columns"] > 0 and not cap["stages"]["cap_stage"]
    assert not any("block_max" in n for n in cap["names"])
    assert sum("block_max" in n for n in belt["names"]) == 1
    assert any("conv_belt_mma" in n for n in stack["names"])
    assert not any("block_max" in n for n in stack["names"])


@pytest.mark.parametrize("nside,theta", [(256, 900.0), (512, 700.0)])
def test_bands_of_the_stages_equal_the_whole_map(K, nside, theta):
    """Bit for bit, for bands that start and end inside a block of 16 belt rings, of one ring, across
    the equator and both cap boundaries, at both poles; the rest of the output untouched."""
    sp, _ = _split(K, nside, theta)
    m = inputs.white_noise_map(nside, 13).astype(np.float32)
    m[: 6 * nside * nside] += np.float32(3.0)  # a constant is taken off northern rings
    x = torch.tensor(m, device="cuda")
    one = torch.empty_like(x)
    _, _, n, st, _ = O.ring_table(nside)
    with sp:
        assert K.split_stages(sp)["belt_columns"] > 0
        K.conv_real(sp, x, one)
        for lo, hi in ((nside + 5, nside + 40), (2 * nside, 2 * nside), (2 * nside - 9, 2 * nside + 3),
                       (nside - 7, nside + 1), (3 * nside - 3, 3 * nside + 9), (1, 9),
                       (4 * nside - 30, 4 * nside - 1), (nside // 2, 3 * nside)):
            part = torch.zeros_like(x)
            K.conv_real_rings(sp, x, part, lo, hi)
            a, b = int(st[lo - 1]), int(st[hi - 1] + n[hi - 1])
            assert torch.equal(part[a:b], one[a:b]), (lo, hi)
            assert not part[:a].any() and not part[b:].any()


# (nside, cut in arcmin, whether the belt stage takes at most 0.7 of the FFMA kernel's time)
@pytest.mark.parametrize("nside,theta,want", [(256, 440.0, 0), (256, 660.0, 1), (512, 110.0, 0), (512, 165.0, 1),
                                              (2048, 7.0, 0), (2048, 28.0, 1), (2048, 240.0, 1)])
def test_belt_stage_is_taken_where_it_is_faster(K, nside, theta, want):
    sp, _ = _split(K, nside, theta)
    with sp:
        assert (K.split_stages(sp)["belt_columns"] > 0) == want


@pytest.mark.parametrize("nside,theta", [(256, 660.0), (512, 700.0)])
def test_captured_calls_hold_their_scratch(K, nside, theta):
    """A call captured into a graph, replayed on other values, and a call on another stream between."""
    sp, _ = _split(K, nside, theta)
    x = torch.tensor(inputs.white_noise_map(nside, 15).astype(np.float32), device="cuda")
    y, z, one = torch.zeros_like(x), torch.zeros_like(x), torch.zeros_like(x)
    with sp:
        K.conv_real(sp, x, y)
        torch.cuda.synchronize()
        g = torch.cuda.CUDAGraph()
        with torch.cuda.graph(g):
            K.conv_real(sp, x, y, stream=torch.cuda.current_stream())
        side = torch.cuda.Stream()
        for k in range(3):
            x.copy_(torch.tensor(inputs.white_noise_map(nside, 16 + k).astype(np.float32)))
            torch.cuda.synchronize()
            g.replay()
            K.conv_real(sp, x, z, stream=side)
            torch.cuda.synchronize()
            K.conv_real(sp, x, one)
            torch.cuda.synchronize()
            assert torch.equal(y, one) and torch.equal(z, one)
        K.device_status(sp)
        del g


def test_batch_gather_tile_suits_all_entries(K):
    """One tile a group of one nside: small tables where those of every split fit and there are
    items enough, whichever entry comes first."""
    fits, wide, tiny = _split(K, 512, 440.0)[0], _split(K, 512, 660.0)[0], _split(K, 64, 360.0)[0]
    assert K.split_stages(fits)["gather_variant"] == 1 and K.split_stages(wide)["gather_variant"] == 2
    for splits, want in (([fits, fits], [1]), ([fits, wide], [2]), ([wide, fits], [2]), ([tiny, fits], [2, 1])):
        with K.Batch(splits) as b:
            assert [g["sym_variant"] for g in b.info()["groups"]] == want
    for sp in (fits, wide, tiny):
        sp.close()


def test_calls_share_the_scratch_of_a_split(K):
    """More calls at once than a split has scratch for, from two threads and six streams, single maps,
    bands and a stack: bit for bit the outputs of calls one after the other."""
    import threading
    nside = 256
    sp, _ = _split(K, nside, 900.0)
    xs = torch.stack([torch.tensor(inputs.white_noise_map(nside, 20 + k).astype(np.float32)) for k in range(6)]).cuda()
    want = torch.empty_like(xs)
    with sp:
        for k in range(6):
            K.conv_real(sp, xs[k], want[k])
        torch.cuda.synchronize()
        got = torch.zeros_like(xs)
        stack = torch.zeros_like(xs)
        streams = [torch.cuda.Stream() for _ in range(6)]

        def work(ks):
            for _ in range(20):
                for k in ks:
                    K.conv_real(sp, xs[k], got[k], stream=streams[k])
                    K.conv_real_rings(sp, xs[k], got[k], 2 * nside - 4, 2 * nside + 9, stream=streams[k])

        threads = [threading.Thread(target=work, args=(ks,)) for ks in ((0, 1, 2), (3, 4, 5))]
        for t in threads:
            t.start()
        K.conv_real_multimap(sp, xs, stack, 6)
        for t in threads:
            t.join()
        torch.cuda.synchronize()
        K.device_status(sp)
        assert torch.equal(got, want) and torch.equal(stack, want)


# (nside, cut in arcmin, columns of the belt tiles, cap stage): each width that a plan takes, short and
# long windows
@pytest.mark.parametrize("nside,theta,columns,cap", [(128, 2400.0, 32, 0), (256, 660.0, 32, 0), (256, 1800.0, 32, 1),
                                                     (512, 240.0, 128, 0), (512, 640.0, 128, 1),
                                                     (1024, 60.0, 256, 0), (1024, 400.0, 256, 1)])
def test_stages_match_the_oracle(K, nside, theta, columns, cap):
    """First and last pixels of the first, sixteenth, seventeenth and last belt rings, the poles, both
    sides of the cap boundaries, and random pixels."""
    sp, c = _split(K, nside, theta)
    tc = theta * inputs.ARCMIN
    m = inputs.white_noise_map(nside, 17).astype(np.float32)
    x = torch.tensor(m, device="cuda")
    y = torch.full_like(x, float("nan"))
    with sp:
        st = K.split_stages(sp)
        assert (st["belt_columns"], st["cap_stage"]) == (columns, cap)
        K.conv_real(sp, x, y)
        K.device_status(sp)
        tab = O.hermite_nodes(c, tc, K.split_info(sp)["n_intervals"])
    first, L, N = 2 * nside * (nside - 1), 4 * nside, 12 * nside * nside
    edge = [first + r * L + k for r in (0, 15, 16, nside, 2 * nside - 1, 2 * nside) for k in (0, 7, 8, L - 1)]
    pix = np.unique(np.concatenate([edge, np.arange(24), N - 1 - np.arange(24), np.arange(40) + first - 20,
                                    inputs.rng(18).choice(N, 500, replace=False)]))
    ref, amb = O.brute_conv(nside, m.astype(np.float64), tc, table=tab, out_pix=pix)
    err = np.abs(y.cpu().numpy()[pix] - ref) - amb
    assert err.max() <= 1e-6 * np.sqrt(np.mean(ref ** 2))


# Kernels whose sums build up over many MMAs: wide beams cut far out, or ringing to the cut.  Error
# rms of FP32 sums with one rounding of the weights, 1.0 to 1.2e-7 of the output's, and a tenth.
@pytest.mark.parametrize("nside,lmax,pixels,lcut,theta", [(512, 1308, 7.73, 516, 1168.0), (512, 1024, 2.5, 512, 640.0),
                                                          (256, 522, 7.12, 235, 1800.0)])
def test_stages_are_left_out_where_their_cuts_add_up(K, nside, lmax, pixels, lcut, theta):
    l = np.arange(lmax + 1)
    b = inputs.gaussian_beam(lmax, pixels * 3518.0 / nside * inputs.ARCMIN)
    m = inputs.white_noise_map(nside, 197).astype(np.float32)
    with K.make_split(b, nside, lcut, theta * inputs.ARCMIN, cl_in=1.0 / (l + 10.0) ** 2) as sp:
        st = K.split_stages(sp)
        x = torch.tensor(m, device="cuda")
        y = torch.empty_like(x)
        K.conv_real(sp, x, y)
        K.device_status(sp)
        tab = O.hermite_nodes(K.split_real_coeffs(sp), theta * inputs.ARCMIN, K.split_info(sp)["n_intervals"])
    assert st["belt_columns"] == 0 and not st["cap_stage"]
    cap, N = 2 * nside * (nside - 1), 12 * nside * nside
    g = inputs.rng(11)
    for pix in (g.choice(cap, 800, replace=False), cap + g.choice(N - 2 * cap, 800, replace=False)):
        ref, amb = O.brute_conv(nside, m.astype(np.float64), theta * inputs.ARCMIN, table=tab, out_pix=pix)
        err = np.maximum(np.abs(y.cpu().numpy()[pix] - ref) - amb, 0.0)
        assert np.sqrt(np.mean(err ** 2)) <= 1.3e-7 * np.sqrt(np.mean(ref ** 2))
