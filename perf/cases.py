"""The work that programs have this library do, as cases that can be timed and compared.

A case is a dict of plain values.  Its `kind` names the entry point:

  conv       ksc_conv_real on one device map
  rings      ksc_conv_real_rings: one latitude band of a map
  stack      ksc_conv_real_multimap: maps that share one split
  batch      ksc_batch_run: maps with splits of their own, of several nside
  host       ksc_conv_real_host: pinned host map in, host map out
  harmonic   ksc_conv_harmonic: the harmonic half of a split (analysis, then synthesis)
  synthesis  ksc_sht_alm2map

Maps are white noise (the paper's test map, and a value at every scale), beams are
Gaussian, splits are weighted with C_l = 1 / (l + 10)^2.  A case with l_cut >= 0 fits
the split in its preparation; l_cut = -1 convolves with the beam itself, truncated
where it has fallen to nothing.
"""
import math

import numpy as np
import torch

from paper_1409_4441_gb300 import ksconv as K

ARCMIN = math.pi / 180.0 / 60.0


def listed():
    return [
        # The smallest call: a low-resolution map smoothed with a 2 degree beam, whole.
        dict(name="conv_nside64", kind="conv", nside=64, lmax=191, fwhm=120.0, l_cut=-1, theta=360.0),
        # An ordinary map: 40' beam, split at l_cut 128, cut at 16 beams.
        dict(name="conv_nside256", kind="conv", nside=256, lmax=512, fwhm=40.0, l_cut=128, theta=640.0),
        # A 20' beam at nside 512, cut at 60': many short windows.
        dict(name="conv_nside512", kind="conv", nside=512, lmax=1535, fwhm=20.0, l_cut=-1, theta=60.0),
        # The Planck-size map of the paper: 5' beam, l_max 4096, l_cut 1024, cut at 240'.
        dict(name="conv_nside2048", kind="conv", nside=2048, lmax=4096, fwhm=5.0, l_cut=1024, theta=240.0),
        # One of eight latitude bands of that map, at the 120' cut that meets 1e-5.
        dict(name="rings_nside2048", kind="rings", nside=2048, lmax=4096, fwhm=5.0, l_cut=1024, theta=120.0,
             ring_lo=1025, ring_hi=2047),
        # Simulations: sixteen maps under one split.
        dict(name="stack_nside512", kind="stack", nside=512, lmax=1535, fwhm=30.0, l_cut=384, theta=480.0,
             n_maps=16, tensor=0),
        # The same with the cap ring pairs on the tensor cores, as the option offers.
        dict(name="stack_nside512_tensor", kind="stack", nside=512, lmax=1535, fwhm=30.0, l_cut=384,
             theta=480.0, n_maps=16, tensor=1),
        # Detectors of unlike resolution in one replayed batch.
        dict(name="batch_ragged", kind="batch", n256=8, n512=4, n1024=1, graph=True),
        # A program that has its map in host memory.
        dict(name="host_nside1024", kind="host", nside=1024, lmax=2048, fwhm=10.0, l_cut=512, theta=160.0),
        # The other half of the split at the paper's size.
        dict(name="harmonic_nside2048", kind="harmonic", nside=2048, lmax=4096, fwhm=5.0, l_cut=1024,
             theta=120.0, add=True),
        # The other half for a small map, where launches count.
        dict(name="harmonic_nside128", kind="harmonic", nside=128, lmax=256, fwhm=80.0, l_cut=64,
             theta=640.0, add=False),
        # Making a map from its coefficients up to l_max = 2 nside.
        dict(name="synthesis_nside512", kind="synthesis", nside=512, lmax=1024),
    ]


def _log(rng, lo, hi):
    return math.exp(rng.uniform(math.log(lo), math.log(hi)))


def _draw_split(rng, nside, whole):
    """A beam of 2.5 to 8 pixels and a cut that costs no more than the Planck-size map's."""
    pixel = 3518.0 / nside  # arcmin
    fwhm = round(rng.uniform(2.5, 8.0) * pixel, 2)
    lmax = rng.randint(3 * nside // 2, 3 * nside - 1)
    if whole:
        return dict(nside=nside, lmax=lmax, fwhm=fwhm, l_cut=-1, theta=round(3.0 * fwhm, 2))
    theta = min(_log(rng, 12.0, 64.0) * fwhm, 1800.0, 9.0e8 / nside**2)
    return dict(nside=nside, lmax=lmax, fwhm=fwhm, l_cut=rng.randint(lmax // 8, lmax // 2), theta=round(theta, 2))


def draw(rng):
    kind = rng.choice(["conv", "conv", "conv", "conv", "rings", "stack", "batch", "host", "harmonic", "synthesis"])
    if kind == "conv":
        nside = 2 ** rng.randint(6, 11)
        return dict(kind=kind, **_draw_split(rng, nside, rng.random() < 0.3))
    if kind == "rings":
        nside = 2 ** rng.randint(8, 11)
        lo = rng.randint(1, 4 * nside - 2)
        hi = min(4 * nside - 1, lo + int(_log(rng, 8, nside)))
        return dict(kind=kind, **_draw_split(rng, nside, rng.random() < 0.3), ring_lo=lo, ring_hi=hi)
    if kind == "stack":
        nside = 2 ** rng.randint(6, 9)
        c = dict(kind=kind, **_draw_split(rng, nside, rng.random() < 0.3))
        c["theta"] = min(c["theta"], 600.0)
        return dict(c, n_maps=int(_log(rng, 2, 24)), tensor=rng.choice([0, 1]))
    if kind == "batch":
        return dict(kind=kind, n256=rng.randint(1, 16), n512=rng.randint(0, 6), n1024=rng.randint(0, 2),
                    graph=rng.random() < 0.5)
    if kind == "host":
        nside = 2 ** rng.randint(6, 11)
        return dict(kind=kind, **_draw_split(rng, nside, rng.random() < 0.3))
    nside = 2 ** rng.randint(6, 10)
    if kind == "harmonic":
        lmax = 2 * nside
        return dict(kind=kind, nside=nside, lmax=lmax, fwhm=round(_log(rng, 2.5, 8.0) * 3518.0 / nside, 2),
                    l_cut=rng.randint(lmax // 8, lmax // 2 + 1), theta=round(_log(rng, 20.0, 60.0) * 3518.0 / nside, 2),
                    add=rng.random() < 0.5)
    return dict(kind=kind, nside=nside, lmax=rng.randint(nside // 2, min(1024, 2 * nside)))


# ---- what a program has before the call -----------------------------------

def _beam(lmax, fwhm):
    ell = np.arange(lmax + 1)
    sigma = fwhm * ARCMIN / math.sqrt(8.0 * math.log(2.0))
    return np.exp(-ell * (ell + 1) * sigma * sigma / 2.0)


def _split(c, **opts):
    b, theta = _beam(c["lmax"], c["fwhm"]), c["theta"] * ARCMIN
    if c["l_cut"] < 0:
        return K.make_split_real(b, c["nside"], theta, **opts)
    cl = 1.0 / (np.arange(c["lmax"] + 1) + 10.0) ** 2
    return K.make_split(b, c["nside"], c["l_cut"], theta, cl_in=cl, **opts)


def _noise(shape, seed, k=0):
    g = torch.Generator(device="cuda").manual_seed(1409 + 1000003 * seed + k)
    return torch.randn(shape, generator=g, device="cuda", dtype=torch.float32)


def _npix(nside):
    return 12 * nside * nside


def _batch_entries(c):
    """(nside, beam) of each map: beams of 40', 20' and 10', cuts at 16 beams."""
    return [(256, 40.0)] * c["n256"] + [(512, 20.0)] * c["n512"] + [(1024, 10.0)] * c["n1024"]


def prepare(case, seed):
    kind = case["kind"]
    s = {"case": case, "kind": kind}
    if kind == "batch":
        entries = _batch_entries(case)
        own = {ns: _split(dict(nside=ns, lmax=2 * ns, fwhm=fw, l_cut=ns // 2, theta=16.0 * fw))
               for ns, fw in dict.fromkeys(entries)}
        s["batch"] = K.Batch([own[ns] for ns, _ in entries], use_graph=case["graph"])
        s["x"] = [_noise((_npix(ns),), seed, k) for k, (ns, _) in enumerate(entries)]
        s["y"] = [torch.zeros_like(t) for t in s["x"]]
        return s
    if kind == "synthesis":
        lmax = case["lmax"]
        ell = torch.cat([torch.arange(m, lmax + 1, device="cuda") for m in range(lmax + 1)])
        a = _noise((2, K.n_alm(lmax)), seed).double() / (ell + 10.0) / math.sqrt(2.0)
        a[0, : lmax + 1] *= math.sqrt(2.0)
        a[1, : lmax + 1] = 0.0  # the field is real
        s["alm"] = torch.complex(a[0], a[1])
        s["y"] = torch.zeros(_npix(case["nside"]), device="cuda")
        return s
    if kind == "harmonic":
        b = _beam(case["lmax"], case["fwhm"])
        s["split"] = K.make_split(b, case["nside"], case["l_cut"], case["theta"] * ARCMIN, mode="sharp")
        s["x"] = _noise((_npix(case["nside"]),), seed)
        # what the real-space half wrote before, where the harmonic half is added to it
        s["real"] = _noise((_npix(case["nside"]),), seed, 1) if case["add"] else None
        s["y"] = torch.zeros_like(s["x"])
        return s
    s["split"] = _split(case, tensor=case.get("tensor", 0))
    n = _npix(case["nside"])
    if kind == "host":
        s["x"] = _noise((n,), seed).cpu().pin_memory()
        s["y"] = torch.zeros(n).pin_memory()
        return s
    s["x"] = _noise((case["n_maps"], n) if kind == "stack" else (n,), seed)
    s["y"] = torch.zeros_like(s["x"])
    return s


def run(state):
    kind, c, y = state["kind"], state["case"], state["y"]
    if kind == "conv":
        K.conv_real(state["split"], state["x"], y)
    elif kind == "rings":
        K.conv_real_rings(state["split"], state["x"], y, c["ring_lo"], c["ring_hi"])
    elif kind == "stack":
        K.conv_real_multimap(state["split"], state["x"], y, c["n_maps"])
    elif kind == "batch":
        state["batch"].run(state["x"], y)
    elif kind == "host":
        K.conv_real_host(state["split"], state["x"], y)
    elif kind == "harmonic":
        if c["add"]:
            y.copy_(state["real"])
        K.conv_harmonic(state["split"], state["x"], y, add=c["add"])
    else:
        K.sht_alm2map(c["nside"], c["lmax"], state["alm"], y)
    return y


# ---- what a pass cannot do without ------------------------------------------

def _pairs(nside, theta):
    return _npix(nside) ** 2 * (1.0 - math.cos(theta * ARCMIN)) / 2.0


def work(case):
    kind = case["kind"]
    if kind == "batch":
        e = _batch_entries(case)
        return {"bytes": sum(8.0 * _npix(ns) for ns, _ in e), "flops": sum(2.0 * _pairs(ns, 16.0 * fw) for ns, fw in e)}
    n = float(_npix(case["nside"]))
    if kind in ("harmonic", "synthesis"):
        # Legendre sums: a recurrence step (3) and the even or odd complex sum (4) for each
        # order, degree and northern ring; ring sums by FFT, 2.5 n log2(ring length).
        way = 2 if kind == "harmonic" else 1
        l = case["l_cut"] if kind == "harmonic" else case["lmax"]
        rings = 2.0 * case["nside"]
        legendre = 7.0 * rings * (l + 1) * (l + 2) / 2.0
        fft = 2.5 * n * math.log2(4.0 * case["nside"])
        maps = (3 if case.get("add") else 2) if kind == "harmonic" else 1
        alm = 16.0 * (l + 1) * (l + 2) / 2.0 if kind == "synthesis" else 0.0
        return {"bytes": 4.0 * n * maps + alm, "flops": way * (legendre + fft)}
    pairs = _pairs(case["nside"], case["theta"])
    if kind == "rings":
        share = (case["ring_hi"] - case["ring_lo"] + 1) / (4.0 * case["nside"] - 1.0)
        reach = min(1.0, share + 2.0 * case["theta"] * ARCMIN / math.pi)
        return {"bytes": 4.0 * n * (share + reach), "flops": 2.0 * pairs * share}
    maps = case.get("n_maps", 1)
    return {"bytes": 8.0 * n * maps, "flops": 2.0 * pairs * maps}


# ---- the same in 64 bits, from the definition ---------------------------------

def _rings64(nside):
    """z, sin(theta), length, first pixel and phase flag of every RING-order ring."""
    i = np.arange(1, 4 * nside, dtype=np.int64)
    north, south = i < nside, i > 3 * nside
    ip = np.where(north, i, 4 * nside - i)
    cap = ip.astype(float) ** 2 / (3.0 * nside * nside)
    belt = (4.0 * nside - 2.0 * i) / (3.0 * nside)
    z = np.where(north, 1.0 - cap, np.where(south, cap - 1.0, belt))
    s = np.where(north | south, np.sqrt(cap * (2.0 - cap)), np.sqrt((1.0 - belt) * (1.0 + belt)))
    length = np.where(north | south, 4 * ip, 4 * nside)
    start = np.concatenate([[0], np.cumsum(length)[:-1]])
    phase = np.where(north | south, 1, ((i - nside) % 2 == 0).astype(np.int64))
    return z, s, length, start, phase


def _exact_conv(c, x):
    """All pairs within the cut of each map x[k], pixel by pixel of the window."""
    ns, lmax, cut = c["nside"], c["lmax"], 2.0 * math.sin(0.5 * c["theta"] * ARCMIN)
    dev = x.device
    # the kernel at nodes uniform in chord, values and slopes of its Legendre sum
    n = 32768
    d = torch.linspace(0.0, cut, n + 1, dtype=torch.float64, device=dev)
    z = 1.0 - 0.5 * d * d
    b = _beam(lmax, c["fwhm"])
    p0, p1 = torch.ones_like(z), z.clone()
    q0, q1 = torch.zeros_like(z), torch.ones_like(z)  # derivatives in z
    val = (b[0] * p0 + 3.0 * b[1] * p1) / (4.0 * math.pi)
    slope = 3.0 * b[1] * q1 / (4.0 * math.pi)
    for l in range(2, lmax + 1):
        p0, p1 = p1, ((2 * l - 1) * z * p1 - (l - 1) * p0) / l
        q0, q1 = q1, q0 + (2 * l - 1) * p0
        w = (2 * l + 1) * b[l] / (4.0 * math.pi)
        val += w * p1
        slope += w * q1
    h = cut / n
    slope = slope * -d * h  # per node spacing in chord
    zr, sr, length, start, phase = (torch.from_numpy(a).to(dev) for a in _rings64(ns))
    ring = torch.repeat_interleave(torch.arange(4 * ns - 1, device=dev), length)
    k = torch.arange(_npix(ns), device=dev) - start[ring]
    phi = (2.0 * k + phase[ring]) * math.pi / length[ring]
    theta = torch.atan2(sr, zr)
    out = torch.zeros_like(x, dtype=torch.float64)
    x = x.double()
    for dr in range(-(4 * ns - 2), 4 * ns - 1):
        q_all = torch.arange(4 * ns - 1, device=dev) + dr
        ok = (q_all >= 0) & (q_all < 4 * ns - 1)
        qc = q_all.clamp(0, 4 * ns - 2)
        ok &= (theta[qc] - theta).abs() <= c["theta"] * ARCMIN + 1e-9
        if not bool(ok.any()):
            continue
        sel = torch.nonzero(ok[ring]).squeeze(1)
        q = qc[ring[sel]]
        lq = length[q]
        a = (zr[ring[sel]] - zr[q]) ** 2 + (sr[ring[sel]] - sr[q]) ** 2
        bb = 4.0 * sr[ring[sel]] * sr[q]
        near = torch.round((phi[sel] * lq / math.pi - phase[q]) / 2.0).long()
        # half window in input pixels, at most the whole ring once
        sx = ((cut * cut - a) / bb).clamp(0.0, 1.0)
        half = torch.asin(torch.sqrt(sx)) * lq / math.pi + 2.0
        lo = torch.maximum(-half.long(), -(lq // 2))
        hi = torch.minimum(half.long(), lq - lq // 2 - 1)
        for j in range(int(lo.min()), int(hi.max()) + 1):
            live = torch.nonzero((lo <= j) & (j <= hi)).squeeze(1)
            g, ql = sel[live], q[live]
            kk = near[live] + j
            half_dphi = 0.5 * (phi[g] - (2.0 * kk + phase[ql]) * math.pi / lq[live])
            dist = torch.sqrt(a[live] + bb[live] * torch.sin(half_dphi) ** 2)
            u = (dist / h).clamp(max=float(n))
            t = u.long().clamp(max=n - 1)
            f = u - t
            w = ((1 + 2 * f) * (1 - f) ** 2 * val[t] + f * f * (3 - 2 * f) * val[t + 1]
                 + f * (1 - f) ** 2 * slope[t] + f * f * (f - 1) * slope[t + 1])
            w = torch.where(dist <= cut, w, torch.zeros_like(w))
            out[:, g] += w * x[:, start[ql] + kk % lq[live]]
    return out * (4.0 * math.pi / _npix(ns))


def _exact_cost(c, maps):
    """Seconds _exact_conv takes, about."""
    steps = 15.0 * (c["theta"] * ARCMIN * c["nside"]) ** 2 + 60.0 * c["theta"] * ARCMIN * c["nside"]
    return steps * 30 * (10e-6 + 3e-12 * _npix(c["nside"]) * 2 * maps)


def _legendre64(nside, lmax, dev):
    """lambda_lm for l = 0, 1, ...: tensors [northern ring, m] with zeros where l < m.  Starting
    values that leave the range of a double belong to functions that stay below 1e-60."""
    z, s, _, _, _ = _rings64(nside)
    z = torch.from_numpy(z[: 2 * nside]).to(dev)[:, None]
    m = torch.arange(lmax + 1, dtype=torch.float64, device=dev)[None, :]
    logmm = 0.5 * torch.log((2 * m + 1) / (4 * math.pi)) + 0.5 * (
        torch.lgamma(2 * m + 1) - 2 * torch.lgamma(m + 1) - 2 * m * math.log(2.0)) + m * torch.log(
            torch.from_numpy(s[: 2 * nside]).to(dev)[:, None])
    start = torch.exp(logmm)
    prev, cur = torch.zeros_like(start), torch.zeros_like(start)
    for l in range(lmax + 1):
        new = torch.zeros_like(cur)
        if l:
            al = torch.sqrt((4.0 * l * l - 1.0) / (l * l - m[:, :l] ** 2))
            new[:, :l] = al * z * cur[:, :l]
            if l > 1:
                k = l - 1
                bl = torch.sqrt((k * k - m[:, :k] ** 2) / (4.0 * k * k - 1.0))
                new[:, :k] -= al[:, :k] * bl * prev[:, :k]
        new[:, l] = start[:, l]
        prev, cur = cur, new
        yield l, cur


def _exact_synthesis(nside, lmax, alm):
    """alm: complex128 [l, m] -> map, float64."""
    dev, nr = alm.device, 4 * nside - 1
    g = torch.zeros((nr, lmax + 1), dtype=torch.complex128, device=dev)
    m = torch.arange(lmax + 1, device=dev)
    for l, lam in _legendre64(nside, lmax, dev):
        t = lam * alm[l][None, :]
        g[: 2 * nside] += t
        g[2 * nside:] += (t * (1 - 2 * ((l + m) % 2)))[: 2 * nside - 1].flip(0)
    g[:, 1:] *= 2.0
    _, _, length, _, phase = _rings64(nside)
    g = g * torch.exp(1j * math.pi * m[None, :] * torch.from_numpy(phase / length).to(dev)[:, None])
    out = []
    for r in range(nr):
        f = torch.zeros(int(length[r]), dtype=torch.complex128, device=dev)
        f.index_add_(0, m % int(length[r]), g[r])
        out.append(torch.fft.ifft(f).real * int(length[r]))
    return torch.cat(out)


def _exact_harmonic(c, x):
    nside, lmax, dev = c["nside"], c["l_cut"], x.device
    z, s, length, start, phase = _rings64(nside)
    m = torch.arange(lmax + 1, device=dev)
    f = []
    for r in range(4 * nside - 1):
        t = torch.fft.fft(x[int(start[r]): int(start[r]) + int(length[r])].double())
        f.append(t[m % int(length[r])])
    f = torch.stack(f)
    f = f * torch.exp(-1j * math.pi * m[None, :] * torch.from_numpy(phase / length).to(dev)[:, None])
    north, south = f[: 2 * nside], torch.zeros_like(f[: 2 * nside])
    south[: 2 * nside - 1] = f[2 * nside:].flip(0)
    b = _beam(c["lmax"], c["fwhm"])
    alm = torch.zeros((lmax + 1, lmax + 1), dtype=torch.complex128, device=dev)
    for l, lam in _legendre64(nside, lmax, dev):
        sign = (1 - 2 * ((l + m) % 2))[None, :]
        alm[l] = (lam * (north + sign * south)).sum(0) * (4.0 * math.pi / _npix(nside) * b[l])
    return _exact_synthesis(nside, lmax, alm)


def exact(case, seed):
    kind = case["kind"]
    if kind == "batch":
        return None
    if kind == "synthesis":
        lmax = case["lmax"]
        flat = prepare(case, seed)["alm"]
        alm = torch.zeros((lmax + 1, lmax + 1), dtype=torch.complex128, device=flat.device)
        at = 0
        for m in range(lmax + 1):
            alm[m:, m] = flat[at: at + lmax + 1 - m]
            at += lmax + 1 - m
        return _exact_synthesis(case["nside"], lmax, alm)
    n = _npix(case["nside"])
    if kind == "harmonic":
        y = _exact_harmonic(case, _noise((n,), seed))
        return y + _noise((n,), seed, 1).double() if case["add"] else y
    maps = case.get("n_maps", 1)
    if case["l_cut"] >= 0 or kind == "rings" or _exact_cost(case, maps) > 15.0:
        return None
    x = _noise((maps, n) if kind == "stack" else (n,), seed)
    y = _exact_conv(case, x.reshape(maps, n))
    y = y.reshape(x.shape)
    return y.cpu() if kind == "host" else y
