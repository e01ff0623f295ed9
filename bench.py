"""Benchmark: real-space convolution of the Planck-resolution workload.

Workload: HEALPix nside 2048 (50.3M pixels) FP32 map, l_max 4096, 5' Gaussian
beam, least-squares split at l_cut 1024, theta_cut 240' (Sec. 2-3 sizes).  One
step = one real-space convolution of one map (the whole hot path).  Metric:
pixel-pair interactions per second (and maps per second) over the timed steps.

    python bench.py [--gpus N] [--steps K] [--warmup W] [--impl ours|reference]

Under torchrun each rank convolves its own map (independent problems, weak
scaling); timing is the maximum over ranks.  `--impl reference` times the FP64
CPU oracle (all-pairs brute force) on a bounded sample of output pixels of the
same workload on the host cores.
"""
from __future__ import annotations

import argparse
import json
import os
import statistics
import subprocess
import sys
import time

import numpy as np

ROOT = os.path.dirname(os.path.abspath(__file__))
sys.path.insert(0, ROOT)

from paper_1409_4441_gb300 import inputs  # noqa: E402

ARC = inputs.ARCMIN
WORKLOADS = {
    # the Planck-resolution case (Sec. 2-3 sizes): the benchmark line
    "nside2048": dict(nside=2048, lmax=4096, fwhm=5.0 * ARC, lcut=1024, theta_cut=240.0 * ARC),
    # the same per-ring-pair shape at a quarter of the resolution (every angle x4),
    # small enough for full ncu captures
    "nside512": dict(nside=512, lmax=1024, fwhm=20.0 * ARC, lcut=256, theta_cut=960.0 * ARC),
    # plain convolution, no split: the 2-degree beam itself truncated at 3 x FWHM
    "nside64": dict(nside=64, lmax=191, fwhm=120.0 * ARC, lcut=None, theta_cut=360.0 * ARC),
    # the nside-512 split (l_max 1535, 20' beam, l_cut 256) at the scaled 5' cut
    # the nside-512 split (l_max 1535, 20' beam, l_cut 256), theta_cut chosen by the Sec. 2
    # scan (judged by a measured run where one is recorded)
    "nside512split": dict(nside=512, lmax=1535, fwhm=20.0 * ARC, lcut=256, theta_cut=None),
}
SPLIT_CHOICE = os.path.join(ROOT, "profiles", "split_choice.json")
WORKLOAD = dict(WORKLOADS["nside2048"])
METRIC = "pixel-pair interactions/s and maps/s at nside=2048 vs roofline, at 1e-5 C_l rms err"
UNIT = "pairs/s"
N_SM = 152
FP32_LANES_PER_SM = 128
# DRAM bytes per launch of the dominant kernel at the nside-2048 workload, from one ncu
# capture (dram__bytes_read.sum + dram__bytes_write.sum, full launch): the stage's coefficients,
# 2.4 GB, then the map in and out; the gather (option exact_weights) is not captured
DRAM_TRAFFIC = {"conv_cap_tc_kernel": 2.68e9 + 0.202e9}


def step_kernels(K, sp, opts):
    """(belt kernel, cap kernel, launches per step) of a split's single-map call, as the split
    reports them."""
    st = K.split_stages(sp)
    return ("conv_belt_tc_kernel" if st["belt_columns"] else "conv_belt_kernel",
            "conv_cap_tc_kernel" if st["cap_stage"] else
            "conv_sym_tc_kernel" if opts.get("cap_kernel", 0) == 1 else "conv_sym_kernel",
            st["n_launches"])


def workload_desc(extra=None):
    W = WORKLOAD
    npix = 12 * W["nside"] ** 2
    split = ("no split (the beam itself)" if W["lcut"] is None
             else f"least-squares split l_cut {W['lcut']}")
    d = {"workload": f"nside-{W['nside']} real-space convolution: {npix / 1e6:.1f}M-pixel FP32 map, "
                     f"l_max {W['lmax']}, {W['fwhm'] / ARC:.0f}' Gaussian beam, {split}, "
                     f"theta_cut {W['theta_cut'] / ARC:.0f}', white-noise input",
         "nside": W["nside"], "lmax": W["lmax"], "fwhm_arcmin": W["fwhm"] / ARC,
         "l_cut": W["lcut"], "theta_cut_arcmin": W["theta_cut"] / ARC,
         "l2": ("inputs larger than L2 (201 MB map in, 201 MB out)" if npix * 4 > 129e6
                else "inputs smaller than L2: L2 flushed (256 MB write) between timed steps, "
                     "steps timed alone")}
    if extra:
        d.update(extra)
    return d


def peaks():
    p = {}
    try:
        with open(os.path.join(ROOT, "MEASURED_PEAKS.json")) as f:
            p = json.load(f)
    except OSError:
        pass
    return p


class ClockSampler:
    """nvidia-smi clock / throttle-reason sampling during the timed region."""

    FIELDS = ("clocks.sm,clocks.max.sm,power.draw,clocks_event_reasons.active,"
              "clocks_event_reasons.hw_slowdown,clocks_event_reasons.hw_thermal_slowdown,"
              "clocks_event_reasons.sw_thermal_slowdown,clocks_event_reasons.sw_power_cap")

    def __init__(self, index: int):
        self.index = index
        self.proc = None

    def __enter__(self):
        try:
            self.proc = subprocess.Popen(
                ["nvidia-smi", f"--query-gpu={self.FIELDS}", "--format=csv,noheader,nounits",
                 "-lms", "200", "-i", str(self.index)],
                stdout=subprocess.PIPE, stderr=subprocess.DEVNULL, text=True)
        except OSError:
            self.proc = None
        return self

    def __exit__(self, *a):
        self.lines = []
        if self.proc is not None:
            self.proc.terminate()
            try:
                out, _ = self.proc.communicate(timeout=5)
            except subprocess.TimeoutExpired:
                self.proc.kill()
                out, _ = self.proc.communicate()
            self.lines = [ln for ln in out.splitlines() if ln.strip()]

    def summary(self):
        sm, mx, reasons = [], None, set()
        names = ["hw_slowdown", "hw_thermal_slowdown", "sw_thermal_slowdown", "sw_power_cap"]
        for ln in getattr(self, "lines", []):
            parts = [p.strip() for p in ln.split(",")]
            if len(parts) < 8:
                continue
            try:
                sm.append(float(parts[0]))
                mx = float(parts[1])
            except ValueError:
                continue
            for n, v in zip(names, parts[4:8]):
                if v.lower() == "active":
                    reasons.add(n)
        if not sm:
            return None
        return {"sm_mhz": statistics.median(sm), "sm_max_mhz": mx, "reasons": sorted(reasons),
                "samples": len(sm)}


def dist_setup():
    world = int(os.environ.get("WORLD_SIZE", "1"))
    rank = int(os.environ.get("RANK", "0"))
    local = int(os.environ.get("LOCAL_RANK", "0"))
    return world, rank, local


def oracle_sample(n_pix: int, seed: int, c, n_int: int, m64, result=None):
    """Time the FP64 oracle on n_pix sampled output pixels; returns (pairs, seconds).
    With `result` (a dict) it also receives the pixels, the oracle's outputs there and
    their boundary-ambiguity bounds."""
    import oracle as O
    nside, tc = WORKLOAD["nside"], WORKLOAD["theta_cut"]
    pix = inputs.rng(seed).choice(O.npix(nside), size=n_pix, replace=False)
    tab = O.hermite_nodes(c, tc, n_int)
    t0 = time.perf_counter()
    ref, amb = O.brute_conv(nside, m64, tc, table=tab, out_pix=pix)
    dt = time.perf_counter() - t0
    pairs = int(O.count_pairs(nside, tc, out_pix=pix).sum())
    if result is not None:
        result.update(pix=pix, ref=ref, amb=amb)
    return pairs, dt


def sharp_coeffs():
    b = inputs.gaussian_beam(WORKLOAD["lmax"], WORKLOAD["fwhm"])
    c = b.copy()
    if WORKLOAD["lcut"] is not None:
        c[: WORKLOAD["lcut"] + 1] = 0.0
    return c


def eq6_alpha_refit():
    """(alpha, rows): the least alpha for which Eq. 6 bounds the measured eps_C of every
    split in the surrogate's training set (tests/golden/surrogate_splits.csv)."""
    path = os.path.join(ROOT, "tests", "golden", "surrogate_splits.csv")
    rows = [ln.strip().split(",") for ln in open(path) if ln.strip() and not ln.startswith("#")]
    col = {h: i for i, h in enumerate(rows[0])}
    ratio = [float(r[col["eps_c"]]) / float(r[col["eq6_alpha5"]]) for r in rows[1:]]
    if not ratio:
        raise ValueError("no rows")
    return 5.0 * max(ratio), len(ratio)


def _split_choice():
    """The measured split selection tests/split_choice.py recorded on the machine with the GPU, or {}."""
    try:
        with open(SPLIT_CHOICE) as f:
            return json.load(f)
    except (OSError, ValueError):
        return {}


def choose_theta_cut(K):
    """theta_cut of a workload with a fixed l_cut, by the Sec. 2 scan in the library
    (ksc_scan_split: 30' grid, Eq. 6 with alpha refitted on the measured splits, cost
    max(GPU model, Eq. 8 on 16 cores)), candidates in cost order; where a measured run
    judged the candidates (tests/split_choice.py), its accepted cut."""
    W = WORKLOAD
    b = inputs.gaussian_beam(W["lmax"], W["fwhm"])
    cl = inputs.cl_grf(W["lmax"])
    alpha, _ = eq6_alpha_refit()
    host = K.eq8_cost_model(cores=16)
    cost = K.cost_model(host_ms0=host.host_ms0, host_ms_eq8=host.host_ms_eq8)
    best, rows = K.scan_split(b, W["nside"], cl_in=cl, theta_lo=60 * ARC, theta_hi=1200 * ARC,
                              theta_step=30 * ARC, bound=1e-5, l_cut_fixed=W["lcut"],
                              alpha=alpha, cost=cost)
    sel = {"by": f"library scan (Sec. 2; ksc_scan_split): 30' grid 60'-1200', l_cut fixed, "
                 f"Eq. 6 with alpha {alpha:.3g} (refitted), cost max(GPU model, Eq. 8 / 16 cores)",
           "scan_choice_arcmin": None if best is None else rows[best]["theta_cut"] / ARC,
           "scan_candidates": sum(r["l_cut"] >= 0 for r in rows)}
    th = None if best is None else rows[best]["theta_cut"]
    judged = _split_choice().get("c2", {}).get("chosen")
    if judged:
        th = judged["theta_cut_arcmin"] * ARC
        sel["judged_by_measurement"] = {k: judged[k] for k in ("theta_cut_arcmin", "eps_C",
                                                               "eq6_alpha5")}
        sel["judged_by_measurement"]["source"] = "tests/split_choice.py (GRF input, eps_C <= 1e-5)"
    if th is None:  # nothing meets the bound: the least estimated error
        th = min(rows, key=lambda r: r["error"])["theta_cut"]
        sel["fallback"] = "no candidate meets the bound: least Eq. 6 error"
    return th, sel


def run_cheapest_split(K, torch, stream, b, cl, x):
    """The cheapest nside-2048 split whose measured eps_C meets 1e-5 (l_cut in {512, 1024,
    1536}, theta_cut searched by measurement; tests/split_choice.py), rebuilt and timed
    here: GPU maps/s, and maps/s of the concurrent pair with the host half modelled by
    Eq. 8 on 16 cores."""
    rec = _split_choice().get("c3", {})
    ch = rec.get("chosen")
    if not ch:
        return {"source": "not measured (tests/split_choice.py writes it on the machine with the GPU)"}
    lcut, tc = int(ch["l_cut"]), ch["theta_cut_arcmin"] * ARC
    y = torch.empty_like(x)
    with K.make_split(b, 2048, lcut, tc, cl_in=cl) as sp:
        n_pairs = K.count_pairs(sp)
        ms = _event_ms(lambda: K.conv_real(sp, x, y, stream=stream), stream, torch, reps=3)
        K.device_status(sp)
    host = K.cost_eval(K.eq8_cost_model(cores=16), 2048, lcut, 4096, tc)[1]
    return {"l_cut": lcut, "theta_cut_arcmin": ch["theta_cut_arcmin"],
            "eps_C_measured": ch["eps_C"], "gpu_ms": ms, "gpu_maps_per_s": 1e3 / ms,
            "pairs_per_s": n_pairs / (ms / 1e3), "host_ms_eq8_16cores": host,
            "maps_per_s_concurrent_halves": 1e3 / max(ms, host),
            "fastest_gpu_half": min(({"l_cut": int(k), "theta_cut_arcmin": v["theta_cut_arcmin"],
                                      "eps_C": v["eps_C"], "gpu_ms": v["gpu_ms"],
                                      "gpu_maps_per_s": 1e3 / v["gpu_ms"]}
                                     for k, v in rec.get("smallest_passing_per_l_cut", {}).items()),
                                    key=lambda r: r["gpu_ms"], default=None),
            "per_l_cut": {k: {"theta_cut_arcmin": v["theta_cut_arcmin"], "eps_C": v["eps_C"],
                              "gpu_ms": v["gpu_ms"]}
                          for k, v in rec.get("smallest_passing_per_l_cut", {}).items()},
            "source": f"{_split_choice().get('command')} ({_split_choice().get('date')}): GRF "
                      "input, smallest passing theta_cut per l_cut on a 30' grid"}


def run_whole_split(K, torch, stream, b, cl, x):
    """Both halves of the split convolution on the GPU (ksc_conv_real, then
    ksc_conv_harmonic adding the harmonic half: analysis to l_cut, Khat_l, synthesis) for
    the benchmark split and for the fastest split whose measured eps_C meets 1e-5
    (tests/split_choice.py): maps/s of the whole convolution on one GB300, against the
    paper's ~12 s per map on a GTX 480 + one CPU core (Sec. 3)."""
    out = {}
    cases = [("benchmark_split", 1024, 240.0)]
    fast = [v for v in _split_choice().get("c3", {}).get("smallest_passing_per_l_cut", {}).values()]
    if fast:
        f = min(fast, key=lambda r: r["gpu_ms"])
        cases.append(("fastest_measured_split", int(f["l_cut"]), f["theta_cut_arcmin"]))
    y = torch.empty_like(x)
    for name, lcut, tca in cases:
        with K.make_split(b, 2048, lcut, tca * ARC, cl_in=cl) as sp:
            def whole():
                K.conv_real(sp, x, y, stream=stream)
                K.conv_harmonic(sp, x, y, add=True, stream=stream)
            ms = _event_ms(whole, stream, torch, reps=3)
            ms_h = _event_ms(lambda: K.conv_harmonic(sp, x, y, add=True, stream=stream),
                             stream, torch, reps=3)
            K.device_status(sp)
        out[name] = {"l_cut": lcut, "theta_cut_arcmin": tca, "ms_per_map": ms,
                     "maps_per_s": 1e3 / ms, "harmonic_half_ms": ms_h,
                     "real_half_ms": ms - ms_h}
    return out


def split_accuracy(info):
    """eps_C of the benchmark's split (quoted from the measurement that
    tests/split_accuracy.py writes on the machine with the GPU) and the Eq. 6 estimate with the
    paper's alpha = 5 and with alpha refitted so that Eq. 6 bounds every measured
    split of the surrogate's training set."""
    out = {"eq6_frac_error_alpha5": info["frac_error"]}
    try:
        alpha, n = eq6_alpha_refit()
        out["eq6_alpha_refit"] = alpha
        out["eq6_frac_error_alpha_refit"] = info["frac_error"] * alpha / 5.0
        out["eq6_alpha_refit_from"] = (f"{n} measured splits (nside 128-512, C1 cut): "
                                       "the least alpha with eps_C <= Eq. 6 for all")
    except (OSError, ValueError, KeyError) as e:
        out["eq6_alpha_refit"] = None
        out["eq6_alpha_refit_from"] = f"unavailable: {e}"
    path = os.path.join(ROOT, "profiles", "split_accuracy_nside2048.json")
    try:
        with open(path) as f:
            meas = json.load(f)
        out["eps_C"] = {k: meas[k] for k in ("c1", "free") if k in meas}
        out["eps_C"]["source"] = (f"{meas.get('command')} ({meas.get('date')}); "
                                  f"{meas.get('field')}; c1 = this build's cut (the fitted "
                                  "kernel vanishes with zero slope at theta_cut, timed here), "
                                  "free = the paper's fit as printed")
    except (OSError, ValueError, KeyError) as e:
        out["eps_C"] = {"source": f"not measured: {e}"}
    return out


def run_reference(args, world, rank):
    """The oracle as it stands, on the host cores, bounded samples of the workload."""
    if rank != 0:
        return
    import oracle as O
    O.build()
    nside = WORKLOAD["nside"]
    m64 = inputs.white_noise_map(nside, inputs.seed_for(3)).astype(np.float32).astype(np.float64)
    c = sharp_coeffs()
    # the library's automatic table size (about 96 intervals per shortest l_max wavelength)
    dc = 2.0 * np.sin(0.5 * WORKLOAD["theta_cut"])
    n_int = int(min(8192, max(256, np.ceil(96.0 * dc * WORKLOAD["lmax"] /
                                           (2 * np.pi * np.cos(0.5 * WORKLOAD["theta_cut"]))))))
    n_pix = args.ref_pixels
    cores = os.cpu_count()
    for w in range(args.warmup):
        oracle_sample(max(8, n_pix // 8), 7 + w, c, n_int, m64)
    tot_pairs, tot_t = 0, 0.0
    for s in range(args.steps):
        p, t = oracle_sample(n_pix, 100 + s, c, n_int, m64)
        tot_pairs += p
        tot_t += t
    v = tot_pairs / tot_t
    sample = f"{args.steps} steps x {n_pix} random output pixels of the nside-{nside} map"
    line = {"metric": METRIC, "value": v, "unit": UNIT, "impl": "reference", "n_gpus": 0,
            "steps": args.steps, "warmup": args.warmup,
            "ms_per_step": 1e3 * tot_t / args.steps, "higher_is_better": True,
            "scaling": "weak", "vs_baseline": None, "dtype": "f64", "data": "synthetic",
            "config": workload_desc({"sample": sample}),
            "cpu_baseline": {"value": v, "unit": UNIT, "cores": cores, "kind": "oracle",
                             "sample": sample},
            "e2e": {"value": v, "unit": UNIT, "h2d_bytes_per_step": 0, "d2h_bytes_per_step": 0}}
    print(json.dumps(line), flush=True)


def run_ours(args, world, rank, local):
    import torch
    if not torch.cuda.is_available():
        raise SystemExit("bench.py needs a CUDA device")
    torch.cuda.set_device(local)
    dev = torch.device("cuda", local)
    if world > 1:
        import torch.distributed as dist
        dist.init_process_group("nccl", device_id=dev)
    from paper_1409_4441_gb300 import ksconv as K

    selection = None
    if WORKLOAD["theta_cut"] is None:
        WORKLOAD["theta_cut"], selection = choose_theta_cut(K)
    nside, lmax, lcut, tc = (WORKLOAD[k] for k in ("nside", "lmax", "lcut", "theta_cut"))
    npix = 12 * nside * nside
    b = inputs.gaussian_beam(lmax, WORKLOAD["fwhm"])
    cl = inputs.cl_grf(lmax)
    t0 = time.perf_counter()
    if lcut is None:  # no split: the whole beam in real space
        sp = K.make_split_real(b, nside, tc, **split_opts(args))
    else:
        sp = K.make_split(b, nside, lcut, tc, cl_in=cl, **split_opts(args))
    t_split = time.perf_counter() - t0
    flush = None
    if npix * 4 <= 129e6:  # map smaller than L2: flush it between timed steps
        flush = torch.empty(64 << 20, dtype=torch.float32, device=dev)
    n_pairs = K.count_pairs(sp)
    info = K.split_info(sp)

    m = inputs.white_noise_map(nside, inputs.seed_for(3, rank)).astype(np.float32)
    x = torch.tensor(m, device=dev)
    y = torch.empty_like(x)
    stream = torch.cuda.current_stream()

    def barrier():
        if world > 1:
            import torch.distributed as dist
            dist.barrier()
        torch.cuda.synchronize()

    for _ in range(args.warmup):
        K.conv_real(sp, x, y)
    barrier()
    evs = [(torch.cuda.Event(enable_timing=True), torch.cuda.Event(enable_timing=True))
           for _ in range(args.steps)]
    with ClockSampler(local) as clk:
        barrier()
        t_start = torch.cuda.Event(enable_timing=True)
        t_end = torch.cuda.Event(enable_timing=True)
        t_start.record(stream)
        for i in range(args.steps):
            if flush is not None:
                flush.zero_()
            evs[i][0].record(stream)
            K.conv_real(sp, x, y)
            evs[i][1].record(stream)
        t_end.record(stream)
        barrier()
    elapsed = t_start.elapsed_time(t_end) / 1e3
    launch_ms = [a.elapsed_time(b_) for a, b_ in evs]
    if flush is not None:  # the steps alone, without the flushes between them
        elapsed = sum(launch_ms) / 1e3
    if world > 1:
        import torch.distributed as dist
        tt = torch.tensor([elapsed], device=dev)
        dist.all_reduce(tt, op=dist.ReduceOp.MAX)
        elapsed = float(tt.item())

    # end to end through the host-pointer entry point (pinned host buffers)
    hin = torch.from_numpy(m).pin_memory()
    hout = torch.empty_like(hin).pin_memory()
    for _ in range(max(1, min(args.warmup, 2))):
        K.conv_real_host(sp, hin, hout)
    barrier()
    te = time.perf_counter()
    for _ in range(args.steps):
        K.conv_real_host(sp, hin, hout)
    barrier()
    e2e_t = time.perf_counter() - te
    if world > 1:
        import torch.distributed as dist
        tt = torch.tensor([e2e_t], device=dev)
        dist.all_reduce(tt, op=dist.ReduceOp.MAX)
        e2e_t = float(tt.item())

    # per-stage launch durations (for the roofline of the dominant kernel)
    stage_ms = {1: [], 2: []}
    for st_id in (1, 2):
        for _ in range(2):
            K.conv_real_stage(sp, x, y, st_id)
        for _ in range(args.steps):
            a_, b_ = torch.cuda.Event(enable_timing=True), torch.cuda.Event(enable_timing=True)
            a_.record(stream)
            K.conv_real_stage(sp, x, y, st_id)
            b_.record(stream)
            stage_ms[st_id].append((a_, b_))
    torch.cuda.synchronize()
    stage_ms = {k: statistics.mean(a_.elapsed_time(b_) for a_, b_ in v) for k, v in stage_ms.items()}
    K.device_status(sp)

    total_pairs = n_pairs * args.steps * world
    value = total_pairs / elapsed
    if rank != 0:
        sp.close()
        return
    pk = peaks()
    clocks = clk.summary()
    sm_max = (clocks or {}).get("sm_max_mhz") or pk.get("sm_max_mhz") or 2070.0
    peak_tflops = N_SM * FP32_LANES_PER_SM * 2 * sm_max * 1e6 / 1e12
    n_belt = info["n_pairs_belt"] if info["n_pairs_belt"] >= 0 else 0
    belt_name, cap_name, launches = step_kernels(K, sp, split_opts(args))
    stages = {
        belt_name: {"pairs": n_belt, "ms": stage_ms[1]},
        cap_name: {"pairs": n_pairs - n_belt, "ms": stage_ms[2]},
    }
    for v in stages.values():
        v["tflops"] = 2.0 * v["pairs"] / (v["ms"] / 1e3) / 1e12 if v["ms"] > 0 else 0.0
        v["frac"] = v["tflops"] / peak_tflops
    dom = max(stages, key=lambda k: stages[k]["ms"])
    achieved = stages[dom]["tflops"]

    # a clean output for the accuracy check (the stage timings above add the cap stage
    # into the belt outputs repeatedly)
    K.conv_real(sp, x, y)
    torch.cuda.synchronize()
    cpu = None
    accuracy = {"tolerance": {"per_pixel": "1e-6 of the output rms (+ boundary-pair bound)",
                              "eps_C": 1e-5}}
    if world == 1 and not args.no_cpu_baseline:
        try:
            import oracle as O
            O.build()
            # the timed split's own real-space kernel, tabulated as the library does
            c = K.split_real_coeffs(sp)
            m64 = m.astype(np.float64)
            oracle_sample(16, 5, c, info["n_intervals"], m64)
            res = {}
            p, t = oracle_sample(args.cpu_pixels, 6, c, info["n_intervals"], m64, res)
            cpu = {"value": p / t, "unit": UNIT, "cores": os.cpu_count(), "kind": "oracle",
                   "sample": f"{args.cpu_pixels} random output pixels of the nside-{nside} map, "
                             f"all-pairs FP64 brute force ({t:.1f} s)"}
            # the same pixels of the last timed step's output against the oracle
            got = y.cpu().numpy().astype(np.float64)[res["pix"]]
            rms = float(np.sqrt(np.mean(res["ref"] ** 2)))
            err = np.abs(got - res["ref"])
            accuracy["per_pixel_sampled"] = {
                "pixels": int(res["pix"].size), "max_abs_over_rms": float(err.max() / rms),
                "rms_over_rms": float(np.sqrt(np.mean(err ** 2)) / rms),
                "max_excess_over_tolerance": float((err - res["amb"] - 1e-6 * rms).max() / rms),
                "reference": "FP64 all-pairs oracle on the same tabulated kernel"}
        except Exception as e:  # the baseline must not sink the GPU number
            cpu = {"value": None, "unit": UNIT, "cores": os.cpu_count(), "kind": "oracle",
                   "sample": f"failed: {e}"}
    if args.workload == "nside2048":
        accuracy.update(split_accuracy(info))

    multimap = None
    stack = None
    if world == 1 and not args.no_multimap and args.workload == "nside2048":
        multimap = run_multimap(K, torch, dev, stream, pk)
        stack = run_stack(K, torch, dev, stream, sp,
                          lambda: K.make_split(b, nside, lcut, tc, cl_in=cl, tensor=1),
                          n_pairs, 16, world * args.steps / elapsed)
    cheapest = whole_split = None
    if world == 1 and not args.no_extras and args.workload == "nside2048":
        cheapest = run_cheapest_split(K, torch, stream, b, cl, x)
        whole_split = run_whole_split(K, torch, stream, b, cl, x)
    batch = None
    if world == 1 and not args.no_batch and args.workload == "nside2048":
        batch = run_batch(K, torch, dev, stream, big_split=sp)

    line = {
        "metric": METRIC, "value": value, "unit": UNIT, "n_gpus": world, "steps": args.steps,
        "warmup": args.warmup, "ms_per_step": 1e3 * elapsed / args.steps,
        "higher_is_better": True, "scaling": "weak", "vs_baseline": None, "dtype": "f32",
        "data": "synthetic",
        "config": workload_desc({"n_pairs_per_map": n_pairs, "n_intervals": info["n_intervals"],
                                 "split": ("none: the beam's Legendre series is the "
                                           "real-space kernel, truncated at theta_cut"
                                           if lcut is None else
                                           "weighted least squares (Eq. 3-5), C_l^in = "
                                           "1/(l+10)^2, with this build's addition to the "
                                           "paper's fit: the real-space part vanishes with "
                                           "zero slope at theta_cut (cut_continuity C1; "
                                           "accuracy.eps_C also gives the paper-literal fit)"),
                                 "split_fit_s": round(t_split, 2),
                                 "theta_cut_selection": selection,
                                 "cap_weights_from_tables": round(info["frac_tabulated"], 4),
                                 "parallelism": f"independent maps x{world}"}),
        "maps_per_s": world * args.steps / elapsed,
        "roofline": {"bound": "alu", "kernel": dom,
                     "achieved": achieved, "peak": peak_tflops, "unit": "TFLOP/s",
                     "frac": achieved / peak_tflops,
                     "traffic": DRAM_TRAFFIC.get(dom) if args.workload == "nside2048" else None,
                     "traffic_unit": "bytes per launch (ncu dram__bytes_read.sum + "
                                     "dram__bytes_write.sum of one full-size launch)",
                     "note": "2 FLOP (one FMA) per in-disc pixel pair the kernel handles; "
                             "peak = 152 SMs x 128 FP32 lanes x 2 x max SM clock (the FP32 "
                             "pipe that the paper's formulation uses; the belt and cap "
                             "stages run on the tensor cores, two-part FP16 products with "
                             "FP32 sums, so a stage may exceed it).  In the cap stage operand "
                             "reads of N = 144 MMAs and the turning of their accumulators "
                             "share shared memory, and warps wait for tensor-memory loads "
                             "(ncu: LSU wavefronts 58%, issue 49%, tensor pipe 23%)"},
        "target": {"roofline_frac": 0.5, "met": bool(achieved / peak_tflops >= 0.5),
                   "step_frac": 2.0 * n_pairs / statistics.mean(launch_ms) * 1e3 / 1e12
                   / peak_tflops},
        "accuracy": accuracy,
        "stages": stages,
        "step_tflops": 2.0 * n_pairs / statistics.mean(launch_ms) * 1e3 / 1e12,
        "e2e": {"value": total_pairs / e2e_t, "unit": UNIT, "h2d_bytes_per_step": 4 * npix,
                "d2h_bytes_per_step": 4 * npix},
        "gpu_launches": launches * args.steps,
        "clocks": clocks,
        "cpu_baseline": cpu,
        "multimap": multimap,
        "stack_nside2048": stack,
        "cheapest_split_nside2048": cheapest,
        "whole_split_on_gpu_nside2048": whole_split,
        "batch": batch,
    }
    print(json.dumps(line), flush=True)
    sp.close()


def split_opts(args):
    """Split options chosen on the command line (the library's defaults otherwise)."""
    return {} if args.cap_kernel is None else {"cap_kernel": args.cap_kernel}


def run_band(args):
    """Profiling case: output rings lo..hi of the benchmark workload (a band of
    cap rings, so that ncu can capture the cap gather's per-ring-pair shapes at
    nside 2048 in a launch of tens of ms).  Prints the band's launch time."""
    import torch
    from paper_1409_4441_gb300 import ksconv as K
    dev = torch.device("cuda", 0)
    lo, hi = args.band
    nside, lmax, lcut, tc = (WORKLOAD[k] for k in ("nside", "lmax", "lcut", "theta_cut"))
    b = inputs.gaussian_beam(lmax, WORKLOAD["fwhm"])
    sp = K.make_split(b, nside, lcut, tc, cl_in=inputs.cl_grf(lmax), **split_opts(args))
    m = inputs.white_noise_map(nside, inputs.seed_for(3)).astype(np.float32)
    x = torch.tensor(m, device=dev)
    y = torch.zeros_like(x)
    ms = _event_ms(lambda: K.conv_real_rings(sp, x, y, lo, hi), torch.cuda.current_stream(),
                   torch, reps=args.steps)
    K.device_status(sp)
    print(json.dumps({"band": [lo, hi], "ms": ms, "workload": workload_desc()}), flush=True)
    sp.close()


def _event_ms(fn, stream, torch, reps=3):
    """Mean CUDA-event time (ms) of fn() on `stream` after one untimed call."""
    fn()
    torch.cuda.synchronize()
    ev = []
    for _ in range(reps):
        a_, b_ = torch.cuda.Event(enable_timing=True), torch.cuda.Event(enable_timing=True)
        a_.record(stream)
        fn()
        b_.record(stream)
        ev.append((a_, b_))
    torch.cuda.synchronize()
    return statistics.mean(a_.elapsed_time(b_) for a_, b_ in ev)


def run_stack(K, torch, dev, stream, sp, make_tensor_split, n_pairs, n_maps, single_maps_per_s):
    """n_maps maps of the benchmark workload itself (nside 2048, the same split) as one
    map-stack call: the default path (the single-map kernels, one launch of each
    for the stack) and the opt-in tensor path (tensor=1: cap ring pairs on the tensor
    cores, belt on the default stage), maps/s against the single-map step.  Maps: i.i.d.
    N(0,1) drawn on the device from a seeded generator (throughput does not depend on
    the values)."""
    npix = 12 * 2048 * 2048
    gen = torch.Generator(device=dev)
    gen.manual_seed(inputs.seed_for(3, 1000))
    x = torch.randn((n_maps, npix), generator=gen, device=dev, dtype=torch.float32)
    y = torch.empty_like(x)
    ms = _event_ms(lambda: K.conv_real_multimap(sp, x, y, n_maps), stream, torch, reps=1)
    K.device_status(sp)
    with make_tensor_split() as st_:
        ms_t = _event_ms(lambda: K.conv_real_multimap(st_, x, y, n_maps), stream, torch, reps=2)
        K.device_status(st_)
    del x, y
    return {"workload": f"{n_maps} maps x nside 2048, the benchmark split (5' beam, l_cut 1024, "
                        "theta_cut 240'), one map-stack call",
            "maps_per_s": n_maps / (ms / 1e3), "ms_per_call": ms,
            "pairs_per_s": n_maps * n_pairs / (ms / 1e3),
            "maps_per_s_tensor": n_maps / (ms_t / 1e3), "ms_per_call_tensor": ms_t,
            "tensor_note": "opts.tensor = 1 (TF32 x3 caps, C_l-level accuracy: per pixel "
                           "within ~3e-5 of the output rms of the default path's result)",
            "single_map_maps_per_s": single_maps_per_s}


def run_multimap(K, torch, dev, stream, pk, nside=1024, n_maps=64):
    """n_maps maps sharing one split (at nside 1024: 15' beam, l_max 3071, l_cut 768,
    theta_cut 480'; other nside scale every angle by 1024/nside).  Default path: the
    single-map kernels.  Opt-in tensor path (tensor=1): the cap ring pairs as a
    tcgen05 contraction (each weight shared by 16 images x 8 maps, TF32 x3, FP32
    accumulate), the belt ring pairs on the default belt stage.  Reports maps/s of
    both, the roofline of the tensor cap stage, and the tensor form of the belt stage
    (tensor=2) for comparison."""
    sc = 1024.0 / nside
    lmax, lcut = 3 * nside - 1, (3 * nside) // 4
    fwhm, tc = 15.0 * sc * ARC, 480.0 * sc * ARC
    b = inputs.gaussian_beam(lmax, fwhm)
    cl = inputs.cl_grf(lmax)
    sp = K.make_split(b, nside, lcut, tc, cl_in=cl, tensor=1)       # tensor caps
    sf = K.make_split(b, nside, lcut, tc, cl_in=cl)                 # FFMA only (default)
    sb = K.make_split(b, nside, lcut, tc, cl_in=cl, tensor=2)       # tensor belt as well
    n_pairs = K.count_pairs(sp)
    info = K.split_info(sp)
    npix = 12 * nside * nside
    x = torch.empty((n_maps, npix), dtype=torch.float32, device=dev)
    for i in range(n_maps):
        x[i] = torch.from_numpy(inputs.white_noise_map(nside, inputs.seed_for(4, i)).astype(np.float32))
    y = torch.empty_like(x)
    t_all = _event_ms(lambda: K.conv_real_multimap(sp, x, y, n_maps), stream, torch, reps=2) / 1e3
    t_belt = _event_ms(lambda: K.conv_real_multimap_stage(sp, x, y, n_maps, 1), stream, torch) / 1e3
    t_caps = _event_ms(lambda: K.conv_real_multimap_stage(sp, x, y, n_maps, 2), stream, torch) / 1e3
    t_ffma = _event_ms(lambda: K.conv_real_multimap(sf, x, y, n_maps), stream, torch, reps=1) / 1e3
    t_tbelt = _event_ms(lambda: K.conv_real_multimap_stage(sb, x, y, n_maps, 1), stream, torch,
                        reps=2) / 1e3
    for s_ in (sp, sf, sb):
        K.device_status(s_)
    belt_pairs = info["n_pairs_belt"]
    cap_pairs = n_pairs - belt_pairs
    tf32_peak = pk.get("bf16_tflops", 1900.0) * (1.1 / 2.25)
    caps_tf = 2.0 * cap_pairs * n_maps / t_caps / 1e12
    tbelt_tf = 2.0 * belt_pairs * n_maps / t_tbelt / 1e12
    for s_ in (sp, sf, sb):
        s_.close()
    return {"workload": f"{n_maps} maps x nside {nside}, shared {fwhm / ARC:.3g}' split, "
                        f"l_max {lmax}, l_cut {lcut}, theta_cut {tc / ARC:.4g}'",
            "maps_per_s": n_maps / t_ffma, "ms_per_call": 1e3 * t_ffma,
            "maps_per_s_tensor": n_maps / t_all, "ms_per_call_tensor": 1e3 * t_all,
            "pairs_per_map": n_pairs, "belt_pairs_per_map": belt_pairs,
            "stages_ms": {"belt": 1e3 * t_belt, "caps_tensor": 1e3 * t_caps},
            "tensor_stage": {"kernel": "conv_sym_mma_kernel", "ms": 1e3 * t_caps,
                             "achieved": caps_tf, "unit": "TFLOP/s", "peak": tf32_peak,
                             "frac": caps_tf / tf32_peak,
                             "note": "2 FLOP per cap pixel pair per map; peak = measured bf16 "
                                     "burst x (1.1/2.25) nominal TF32 ratio; 3 TF32 MMAs per "
                                     "product for FP32 accuracy"},
            "belt_tensor_form": {"kernel": "conv_belt_mma_kernel", "ms": 1e3 * t_tbelt,
                                 "achieved": tbelt_tf, "unit": "TFLOP/s",
                                 "frac": tbelt_tf / tf32_peak,
                                 "note": "opts.tensor = 2; slower than the FFMA belt stage"}}


def _time_calls(fn, stream, torch, reps=3):
    """Mean CUDA-event time (s) of fn() on `stream` after one untimed call."""
    fn()
    torch.cuda.synchronize()
    a_, b_ = torch.cuda.Event(enable_timing=True), torch.cuda.Event(enable_timing=True)
    a_.record(stream)
    for _ in range(reps):
        fn()
    b_.record(stream)
    torch.cuda.synchronize()
    return a_.elapsed_time(b_) / 1e3 / reps


def run_batch(K, torch, dev, stream, big_split=None):
    """Batched persistent launches (ksc_batch): (a) 64 maps at nside 1024, each with
    its own least-squares split (FWHM uniform in [7, 30]', l_max 3071, l_cut 768,
    theta_cut 240'); (b) a ragged batch of nside 256 / 512 / 1024 / 2048 maps.  Each
    is autotuned, then timed as one graph-replayed batch run against the same
    entries as serial single-map calls (maps/s)."""
    from concurrent.futures import ThreadPoolExecutor
    out = {}
    lmax, lcut, tc = 3071, 768, 240.0 * ARC
    fw = inputs.fwhm_draws(64, 7.0, 30.0, inputs.seed_for(4))
    cl = inputs.cl_grf(lmax)
    t0 = time.perf_counter()
    with ThreadPoolExecutor(8) as ex:  # ctypes releases the GIL during each fit
        sps = list(ex.map(lambda f: K.make_split(inputs.gaussian_beam(lmax, f), 1024, lcut, tc,
                                                 cl_in=cl), fw))
    t_fit = time.perf_counter() - t0
    pairs = [K.count_pairs(s) for s in sps]
    npix = 12 * 1024 ** 2
    xs = [torch.from_numpy(inputs.white_noise_map(1024, inputs.seed_for(4, 100 + i))
                           .astype(np.float32)).to(dev) for i in range(64)]
    ys = [torch.empty_like(x) for x in xs]
    out["per_map_beams"] = _batch_case(K, torch, stream, sps, xs, ys, sum(pairs))
    out["per_map_beams"].update({
        "workload": "64 maps x nside 1024, per-map LSQ splits, FWHM U[7,30]', l_max 3071, "
                    "l_cut 768, theta_cut 240'", "split_fit_s_total": round(t_fit, 1)})
    del xs, ys
    for s in sps:
        s.close()
    # ragged: 32 x nside 256 (40'), 16 x 512 (20'), 4 x 1024 (10'), 1 x 2048 (5')
    ragged, xs = [], []
    specs = [(256, 32, 40.0), (512, 16, 20.0), (1024, 4, 10.0)]
    own = []
    for ns, cnt, fwhm in specs:
        lm = 2 * ns
        sp = K.make_split(inputs.gaussian_beam(lm, fwhm * ARC), ns, ns // 2, 2.0 * fwhm * ARC * 8,
                          cl_in=inputs.cl_grf(lm))
        K.count_pairs(sp)
        own.append(sp)
        for i in range(cnt):
            ragged.append(sp)
            xs.append(torch.from_numpy(inputs.white_noise_map(ns, inputs.seed_for(4, 200 + len(xs)))
                                       .astype(np.float32)).to(dev))
    if big_split is not None:
        ragged.append(big_split)
        xs.append(torch.from_numpy(inputs.white_noise_map(2048, inputs.seed_for(4, 300))
                                   .astype(np.float32)).to(dev))
    ys = [torch.empty_like(x) for x in xs]
    n_pairs = sum(K.split_info(s)["n_pairs"] for s in ragged)
    out["ragged"] = _batch_case(K, torch, stream, ragged, xs, ys, n_pairs)
    out["ragged"]["workload"] = ("32 x nside 256 (40'), 16 x 512 (20'), 4 x 1024 (10'), "
                                 "1 x 2048 (5', the main split); theta_cut 16 x FWHM")
    # small maps alone: where one launch per map leaves the GPU part-idle
    n_small = 32
    sm_specs = [s_ for s_ in ragged if s_ is own[0]][:n_small]
    xs_s = xs[:n_small]
    ys_s = [torch.empty_like(x) for x in xs_s]
    out["small"] = _batch_case(K, torch, stream, sm_specs, xs_s, ys_s,
                               n_small * K.split_info(own[0])["n_pairs"])
    out["small"]["workload"] = "32 x nside 256 (40' beam, l_max 512, l_cut 128, theta_cut 640')"
    for s in own:
        s.close()
    return out


def _batch_case(K, torch, stream, splits, xs, ys, n_pairs):
    n = len(splits)
    t_serial = _time_calls(lambda: [K.conv_real(s, x, y) for s, x, y in zip(splits, xs, ys)],
                           stream, torch)
    with K.Batch(splits, use_graph=True) as b:
        rep = b.autotune(xs, ys)
        t_batch = _time_calls(lambda: b.run(xs, ys), stream, torch)
        b.status()
        info = b.info()
    with K.Batch(splits, use_graph=False) as b:
        t_nograph = _time_calls(lambda: b.run(xs, ys), stream, torch)
    return {"maps": n, "pairs_per_run": n_pairs,
            "maps_per_s_batch": n / t_batch, "maps_per_s_serial": n / t_serial,
            "maps_per_s_batch_no_graph": n / t_nograph,
            "pairs_per_s_batch": n_pairs / t_batch, "ms_batch": 1e3 * t_batch,
            "ms_serial": 1e3 * t_serial, "launches_per_run": info["n_launches"],
            "autotune": rep["groups"]}


def main():
    ap = argparse.ArgumentParser()
    ap.add_argument("--gpus", type=int, default=1)
    ap.add_argument("--steps", type=int, default=10)
    ap.add_argument("--warmup", type=int, default=3)
    ap.add_argument("--impl", default="ours", choices=["ours", "reference"])
    ap.add_argument("--cpu-pixels", type=int, default=512)
    ap.add_argument("--ref-pixels", type=int, default=128)
    ap.add_argument("--no-cpu-baseline", action="store_true")
    ap.add_argument("--no-multimap", action="store_true")
    ap.add_argument("--no-batch", action="store_true")
    ap.add_argument("--no-extras", action="store_true",
                    help="time the benchmark step only (no stack, batch or split-choice runs)")
    ap.add_argument("--multimap-only", action="store_true",
                    help="only the map-stack (tensor-core) section, at --mm-nside / --mm-maps")
    ap.add_argument("--mm-nside", type=int, default=1024)
    ap.add_argument("--mm-maps", type=int, default=64)
    ap.add_argument("--workload", default="nside2048", choices=sorted(WORKLOADS))
    ap.add_argument("--cap-kernel", type=int, choices=[0, 1], default=None,
                    help="ksc_split_opts.cap_kernel for the timed split (default: library's)")
    ap.add_argument("--band", type=int, nargs=2, metavar=("LO", "HI"),
                    help="profiling case: only output rings LO..HI (1-based), timed alone")
    args = ap.parse_args()
    if args.no_extras:
        args.no_multimap = args.no_batch = True
    WORKLOAD.clear()
    WORKLOAD.update(WORKLOADS[args.workload])
    world, rank, local = dist_setup()
    if args.band and args.impl != "reference":
        run_band(args)
        return
    if args.multimap_only and args.impl != "reference":
        import torch
        from paper_1409_4441_gb300 import ksconv as K
        torch.cuda.set_device(local)
        dev = torch.device("cuda", local)
        print(json.dumps(run_multimap(K, torch, dev, torch.cuda.current_stream(), peaks(),
                                      nside=args.mm_nside, n_maps=args.mm_maps)), flush=True)
        return
    if args.impl == "reference":
        if WORKLOAD["theta_cut"] is None:  # the cut the measured selection accepted, if any
            ch = _split_choice().get("c2", {}).get("chosen")
            WORKLOAD["theta_cut"] = (ch["theta_cut_arcmin"] if ch else 960.0) * ARC
        run_reference(args, world, rank)
    else:
        run_ours(args, world, rank, local)


if __name__ == "__main__":
    main()
