"""Throughput benchmark of the D3Q19 central-moment LBM step on GB300.

Workload: body-force-driven periodic flow on a 512^3 grid (uniform g = 1e-6
along x, initial u = seeded uniform noise of amplitude 1e-3, rho = 1,
tau = 0.6), FP32 population storage.  One benchmark "step" is one full LBM
time step of the whole grid (stream + moments + CM collision with forcing +
back-transform + store), i.e. 512^3 lattice updates.  The state (2 x 10.2 GB)
is far larger than L2, so no flush is needed between steps.

Prints one JSON line (rank 0).  Under torchrun each rank runs an independent
replica of the workload on its own GPU (weak scaling; the single-domain step
has no data-parallel exchange in this build).

``--impl reference`` times the FP64 CPU oracle (the slow, obviously-correct
implementation written from the paper) on a bounded sample of the same
workload on the host cores.
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

from paper_2010_01628_gb300 import inputs  # noqa: E402
from paper_2010_01628_gb300.ranks import Ranks, partition_domains  # noqa: E402

METRIC = "D3Q19 CM-LBM MLUPS & % HBM roofline; time to 1e-6 residual, warm vs cold"
N = 512
TAU = 0.6
G = (1e-6, 0.0, 0.0)
BYTES_PER_VALUE = {"fp64": 8, "fp32": 4, "fp16": 2, "bf16": 2}
DTYPE_NAME = {"fp64": "f64", "fp32": "f32", "fp16": "f16 storage / f32 math", "bf16": "bf16 storage / f32 math"}


def workload_config(n, precision):
    return {"workload": f"periodic body-force flow {n}^3, g=1e-6 x, u noise 1e-3 (seed 1), tau=0.6",
            "grid": [n, n, n], "precision": precision, "lattice": "D3Q19", "streaming": "pull A-B",
            "l2": "state larger than L2 (no flush needed)", "synthetic": True}


def algorithmic_bytes(n, precision):
    """19 populations read + 19 written per lattice update (no coupled fields)."""
    return 19 * 2 * BYTES_PER_VALUE[precision] * n ** 3


def measured_peaks():
    path = os.path.join(ROOT, "MEASURED_PEAKS.json")
    try:
        with open(path) as fh:
            d = json.load(fh)
        return float(d["hbm_gbs"]), "measured"
    except Exception:
        return 6800.0, "fallback"


def committed_traffic(kernel_key, group="fluid"):
    """DRAM bytes per launch from the committed ncu summary, if it was taken on
    the current kernel source (matched by hash); else None."""
    path = os.path.join(ROOT, "profiles", "traffic.json")
    try:
        with open(path) as fh:
            d = json.load(fh)
        ent = d[kernel_key]
    except Exception:
        return None
    try:
        from paper_2010_01628_gb300 import build
        if ent.get("source_sha") != build.source_hash(group):
            return None
    except Exception:
        return None
    return ent.get("dram_bytes_per_launch")


class ClockSampler:
    """nvidia-smi clock/throttle sampling during the timed region."""

    QUERY = ("index,clocks.sm,clocks.max.sm,power.draw,clocks_event_reasons.active,"
             "clocks_event_reasons.hw_slowdown,clocks_event_reasons.hw_thermal_slowdown,"
             "clocks_event_reasons.sw_thermal_slowdown,clocks_event_reasons.sw_power_cap")

    def __init__(self, device_id):
        self.proc = None
        self.device_id = device_id

    def __enter__(self):
        try:
            self.proc = subprocess.Popen(["nvidia-smi", f"--query-gpu={self.QUERY}", "--format=csv,noheader,nounits",
                                          "-lms", "200", "-i", str(self.device_id)], stdout=subprocess.PIPE,
                                         stderr=subprocess.DEVNULL, text=True)
        except Exception:
            self.proc = None
        time.sleep(0.3)
        return self

    def __exit__(self, *a):
        self.lines = []
        if self.proc is not None:
            self.proc.terminate()
            try:
                out, _ = self.proc.communicate(timeout=5)
            except Exception:
                self.proc.kill()
                out = ""
            self.lines = [l for l in out.splitlines() if l.strip()]

    def summary(self):
        sm, mx, reasons = [], None, set()
        names = ["hw_slowdown", "hw_thermal_slowdown", "sw_thermal_slowdown", "sw_power_cap"]
        for l in getattr(self, "lines", []):
            p = [x.strip() for x in l.split(",")]
            if len(p) < 9:
                continue
            try:
                sm.append(float(p[1]))
                mx = float(p[2])
            except ValueError:
                continue
            for k, name in enumerate(names):
                if p[5 + k].lower().startswith("active"):
                    reasons.add(name)
        if not sm:
            return {"sm_mhz": None, "sm_max_mhz": None, "reasons": ["unsampled"]}
        return {"sm_mhz": statistics.median(sm), "sm_max_mhz": mx, "reasons": sorted(reasons), "samples": len(sm)}


def smi_device_id(torch):
    try:
        props = torch.cuda.get_device_properties(torch.cuda.current_device())
        uuid = str(getattr(props, "uuid", "") or "")
        if uuid:
            return uuid if uuid.startswith("GPU-") else "GPU-" + uuid
    except Exception:
        pass
    vis = os.environ.get("CUDA_VISIBLE_DEVICES", "")
    return vis.split(",")[0] if vis else "0"


def cpu_baseline_sample(seconds=15.0, n_full=N):
    """Time the FP64 oracle (closed form, all host threads) on a bounded cubic
    sample of the workload; returns a cpu_baseline dict (MLUPS)."""
    import oracle as O
    cores = O.max_threads()
    rho, u = inputs.noise_box((64, 64, 64), amp=1e-3, seed=1)
    d = O.Domain((64, 64, 64), 1 / TAU, g=G)
    d.init(rho, u)
    t = time.perf_counter()
    d.step(2)
    rate = 64 ** 3 * 2 / (time.perf_counter() - t)  # cell updates / s
    n = 96
    steps = max(3, int(seconds * rate / n ** 3))
    rho, u = inputs.noise_box((n, n, n), amp=1e-3, seed=1)
    d = O.Domain((n, n, n), 1 / TAU, g=G)
    d.init(rho, u)
    t = time.perf_counter()
    d.step(steps)
    dt = time.perf_counter() - t
    return {"value": n ** 3 * steps / dt / 1e6, "unit": "MLUPS", "cores": cores, "kind": "oracle",
            "sample": f"{n}^3 periodic sample of the {n_full}^3 body-force workload, {steps} FP64 steps "
                      f"(closed-form oracle, OpenMP), {dt:.1f} s"}


def run_reference(args):
    """The oracle as the reference arm: each step is one oracle step on a
    bounded cubic sample of the workload, sized so the run takes minutes."""
    rank = int(os.environ.get("RANK", "0"))
    if rank != 0:
        return 0
    import oracle as O
    cores = O.max_threads()
    rho, u = inputs.noise_box((48, 48, 48), amp=1e-3, seed=1)
    d = O.Domain((48, 48, 48), 1 / TAU, g=G)
    d.init(rho, u)
    t = time.perf_counter()
    d.step(1)
    rate = 48 ** 3 / (time.perf_counter() - t)
    budget = 90.0 / max(1, args.steps + args.warmup)  # seconds per step
    n = int(max(16, min(256, round((rate * budget) ** (1 / 3) / 8) * 8)))
    rho, u = inputs.noise_box((n, n, n), amp=1e-3, seed=1)
    d = O.Domain((n, n, n), 1 / TAU, g=G)
    d.init(rho, u)
    d.step(args.warmup)
    t = time.perf_counter()
    d.step(args.steps)
    dt = time.perf_counter() - t
    value = n ** 3 * args.steps / dt / 1e6
    line = {"impl": "reference", "metric": METRIC, "value": value, "unit": "MLUPS", "n_gpus": args.gpus,
            "steps": args.steps, "warmup": args.warmup, "ms_per_step": dt / args.steps * 1e3,
            "higher_is_better": True, "scaling": "weak", "vs_baseline": None, "dtype": "f64", "data": "synthetic",
            "config": workload_config(N, "fp32") | {"sample": f"{n}^3",
                                                     "oracle": "FP64 closed-form oracle on the sample (dtype f64)"},
            "cpu_baseline": {"value": value, "unit": "MLUPS", "cores": cores, "kind": "oracle",
                             "sample": f"{n}^3 periodic sample of the {N}^3 workload per step"},
            "e2e": {"value": value, "unit": "MLUPS", "h2d_bytes_per_step": 0, "d2h_bytes_per_step": 0}}
    print(json.dumps(line), flush=True)
    return 0


def extra_workloads(L, torch, stream, steps, peak, only=None, domains=64, n_cgm=256, tune_cache="tmp", n_only=None,
                    ranks=None, launch="auto"):
    """Throughput of the other configurations of the method, each with its own
    algorithmic bytes per lattice update (populations read + written plus the
    coupled fields).  ``only`` restricts the run to one of them (profiling)."""
    out = {}

    def timed(fn, n):
        a = torch.cuda.Event(enable_timing=True)
        b = torch.cuda.Event(enable_timing=True)
        a.record(stream)
        fn(n)
        b.record(stream)
        b.synchronize()
        return a.elapsed_time(b) / 1e3

    if only in (None, "tg32"):
        out.update(_tg32(L, timed))
    if only in (None, "mhd_batch"):
        out.update(_mhd_batch(L, timed, steps, peak, domains, tune_cache, ranks))
    if only in (None, "cgm"):
        out.update(_cgm(L, timed, steps, peak, n_cgm, launch))
    if only in (None, "cgm_batch"):
        out.update(_cgm_batch(L, timed, steps, peak, domains, tune_cache))
    if only in (None, "sc_batch"):
        out.update(_sc_batch(L, timed, steps, peak, domains, tune_cache))
    if only in (None, "sc"):
        out.update(_sc(L, timed, steps, peak, (n_only,) if n_only else (100, 256), launch))
    if only in (None, "rt"):
        out.update(_rt(L, timed, steps, peak, launch))
    if only in (None, "appd"):
        out.update(_appd(L, timed, steps, n_only or 256))
    if only in (None, "channel"):
        out.update(_channel(L, timed, steps, peak, n_only or 512))
    if only in (None, "cnn"):
        out.update(_cnn(L, torch, timed, n_only or 128))
    return out


# Tensor-core work of the warm-start network per voxel, with the channel
# padding the kernels compute (16-32-32-32-16): forward 2 x 27 x 3072,
# backward data (layers 4..2) 2 x 27 x 2560, weight gradients 2 x 27 x 3072.
CNN_FLOP_FWD = 2 * 27 * 3072
CNN_FLOP_TRAIN = 2 * 27 * (3072 + 2560 + 3072)


def bf16_peak():
    try:
        with open(os.path.join(ROOT, "MEASURED_PEAKS.json")) as fh:
            d = json.load(fh)
        return float(d["bf16_tflops"]), float(d["bf16_tflops_sustained"]), "measured"
    except Exception:
        return 1900.0, 1700.0, "fallback"


def _cnn(L, torch, timed, n=128, steps=20):
    """Warm-start network at n^3: one Adam step (forward, loss, backward data,
    weight gradients, Adam) and one inference (forward), CUDA-event timed;
    TFLOP/s of the tensor-core work against the measured BF16 peaks."""
    P = n ** 3
    rng = np.random.default_rng(11)
    rho = torch.from_numpy(1.0 + 0.01 * rng.standard_normal((n, n, n))).cuda()
    u = torch.from_numpy(0.05 * rng.standard_normal((3, n, n, n))).cuda()
    net = L.lbm_cnn_create((n, n, n))
    try:
        L.lbm_cnn_set_input(net, 550.0)
        for _ in range(3):
            L.lbm_cnn_train_step(net, rho, u, 1e-4)
        t_train = timed(lambda k: [L.lbm_cnn_train_step(net, rho, u, 1e-4) for _ in range(k)], steps) / steps
        t_fwd = timed(lambda k: [L.lbm_cnn_forward(net) for _ in range(k)], steps) / steps
    finally:
        L.lbm_cnn_destroy(net)
    burst, sustained, kind = bf16_peak()
    tf_train = CNN_FLOP_TRAIN * P / t_train / 1e12
    tf_fwd = CNN_FLOP_FWD * P / t_fwd / 1e12
    return {f"cnn_warmstart_{n}": {
        "train_step_ms": t_train * 1e3, "train_TFLOPs": tf_train, "train_frac_of_bf16_sustained": tf_train / sustained,
        "forward_ms": t_fwd * 1e3, "forward_TFLOPs": tf_fwd, "forward_frac_of_bf16_burst": tf_fwd / burst,
        "peak_kind": kind, "steps": steps,
        "note": "tcgen05 BF16 MMAs (TMEM accumulators, bulk-copy row staging); FLOPs with padded channels "
                "16-32-32-32-16; the train step includes the loss, Adam and weight packing; each call synchronises"}}


def _tg32(L, timed):
    # C1: 3D Taylor-Green vortex 32^3, FP64, 200 steps.  32,768 nodes are a
    # fraction of one wave; a step's 10 M FP64 operations take ~16 us at the
    # FP64 pipes' rate, close to the measured step time.
    out = {}
    rho, u = inputs.taylor_green_3d(32, u0=0.05)
    c = L.lbm_create((32, 32, 32), 1 / 0.53, precision="fp64")
    L.lbm_init_fields(c, rho, u)
    L.lbm_autotune(c, None)
    L.lbm_step(c, 5)
    t = timed(lambda n: L.lbm_step(c, n), 200)
    shape = L.lbm_get_launch_shape(c)
    L.lbm_destroy(c)
    out["taylor_green_32_fp64"] = {"MLUPS": 32 ** 3 * 200 / t / 1e6, "steps": 200, "bytes_per_lup": 304,
                                   "launch": shape,
                                   "note": "small domain, one kernel per step: FP64-pipe bound"}
    return out


def _mhd_batch(L, timed, steps, peak, domains, tune_cache="tmp", ranks=None):
    import tempfile
    out = {}

    # C3: Hartmann channels (64 by default), sizes {32,48,64,96}^3, Ha in [1,20], FP32 MHD,
    # one launch per step over all domains, replayed from captured graphs.  With several ranks the sweep's
    # domains are partitioned by node count (no exchange between ranks): strong scaling of the fixed sweep.
    full = inputs.hartmann_batch(domains, seed=2)
    world = ranks.world if ranks else 1
    mine = partition_domains([n ** 3 for n, _ in full], world)[ranks.rank if ranks else 0]
    sweep = [full[i] for i in mine]
    nu = 0.1
    shapes = [(n, n, n) for n, _ in sweep]
    b0s = [2 * ha * nu / n for n, ha in sweep]
    batch = L.lbm_batch_create(shapes, 1 / (nu / (1 / 3) + 0.5), periodic=(True, False, True), physics="mhd",
                               precision="fp32", tau_m=0.5 + nu / 0.25,
                               g=[(8 * nu * 0.01 / n ** 2, 0.0, 0.0) for n, _ in sweep],
                               b_wall=[(0.0, b, 0.0) for b in b0s])
    cells = sum(n ** 3 for n, _ in full)
    for k, (n, _) in enumerate(sweep):
        r, uu, B = inputs.hartmann(n, b0s[k], nx=n, nz=n)
        L.lbm_init_fields(L.lbm_batch_domain(batch, k), r, uu, B=B)
    cache = os.path.join(tempfile.gettempdir(), "lbm_tune_cache.json") if tune_cache == "tmp" else None
    tuned = L.lbm_autotune(batch, cache)  # no cache: every run times the candidates
    L.lbm_batch_step(batch, 4)
    n_b = max(20, steps)
    if ranks:
        ranks.barrier()
    t = timed(lambda n: L.lbm_batch_step(batch, n), n_b)
    L.lbm_sync(batch)
    if ranks:
        t = ranks.max_over_ranks(t)
    info = L.lbm_batch_info(batch)
    L.lbm_destroy(batch)
    ach = 320 * cells * n_b / t / 1e9
    out[f"mhd_batch_{domains}"] = {"MLUPS": cells * n_b / t / 1e6, "cells": cells, "steps": n_b, "bytes_per_lup": 320,
                           "achieved_GBps": ach, "frac_of_hbm_peak": ach / peak, "launch": info,
                           "autotune_MLUPS": tuned, "launches_per_step": 1, "ranks": world,
                           "domains_on_rank0": len(mine)}
    return out


# Colour-gradient state: 19 total populations plus the red fraction, the 3-vector of the recolouring term and the
# red rest population per node, read and written once, and phi and rho_r written and read once per step.
CGM_BYTES = 24 * 2 * 4 + 2 * 2 * 4


def _cgm_batch(L, timed, steps, peak, domains=64, tune_cache="tmp"):
    """Density-ratio sweep: `domains` periodic droplet boxes, sizes {32,48,64,96}^3, density ratio U[2, 10]
    (seed 5), sigma = 1e-4, tau = 0.8, beta = 0.7, FP32, as one batch (two launches per step over all domains,
    replayed from captured graphs)."""
    import tempfile
    sweep = inputs.droplet_sweep(domains, seed=5)
    shapes = [(n, n, n) for n, _ in sweep]
    tau, sigma, alpha_b = 0.8, 1e-4, 1.0 / 3.0
    om = 1.0 / tau
    batch = L.lbm_batch_create(shapes, om, physics="cgm", precision="fp32", alpha_b=alpha_b,
                               alpha_r=[1.0 - (1.0 - alpha_b) / r for _, r in sweep], A=9.0 * sigma * om / 4.0,
                               beta=0.7)
    cells = sum(n ** 3 for n, _ in sweep)
    for k, (n, ratio) in enumerate(sweep):
        rho, u, ph = inputs.sweep_droplets(n, ratio, k)
        L.lbm_init_fields(L.lbm_batch_domain(batch, k), rho, u, phase=ph)
    cache = os.path.join(tempfile.gettempdir(), "lbm_tune_cache.json") if tune_cache == "tmp" else None
    tuned = L.lbm_autotune(batch, cache)
    L.lbm_batch_step(batch, 4)
    n_b = max(20, steps)
    t = timed(lambda n: L.lbm_batch_step(batch, n), n_b)
    L.lbm_sync(batch)
    info = L.lbm_batch_info(batch)
    L.lbm_destroy(batch)
    ach = CGM_BYTES * cells * n_b / t / 1e9
    return {f"cgm_batch_{domains}": {
        "MLUPS": cells * n_b / t / 1e6, "cells": cells, "steps": n_b, "bytes_per_lup": CGM_BYTES,
        "moved_bytes_per_lup": 284, "achieved_GBps": ach, "frac_of_hbm_peak": ach / peak, "launch": info,
        "autotune_MLUPS": tuned, "launches_per_step": 2,
        "note": "colour-gradient density-ratio sweep (ratio U[2,10]) stepped as one batch; "
                + CGM_NOTE}}
CGM_NOTE = ("two passes per step (phi and rho_r, then collide); 24 stored values per node (total populations, red "
            "fraction, recolouring vector, red rest), 208 B/LUP algorithmic; pass 1 and pass 2 both read the totals "
            "(284 B moved). The two colour distributions stored separately would be 312 B/LUP.")


def _cgm(L, timed, steps, peak, n, launch="auto"):
    out = {}
    # C4: colour-gradient droplets n^3 (10% volume, R in [8,24]), FP32, autotuned block size.
    rho, u, phase, spheres, frac = inputs.droplets(n, seed=3)
    sigma, tau = 1e-4, 0.8
    alpha_b = 1 / 3
    alpha_r = 1 - (1 - alpha_b) * 1.0 / 10.0
    c = L.lbm_create((n, n, n), 1 / tau, physics="cgm", precision="fp32", alpha_r=alpha_r, alpha_b=alpha_b,
                     A=9 * sigma / tau / 4, beta=0.7)
    L.lbm_init_fields(c, rho, u, phase=phase)
    tuned = L.lbm_autotune(c, None) if launch == "auto" else apply_launch(L, c, launch, None)
    shape = L.lbm_get_launch_shape(c)
    L.lbm_step(c, 3)
    n_c = max(20, steps // 2)
    t = timed(lambda k: L.lbm_step(c, k), n_c)
    L.lbm_reduce(c)
    L.lbm_destroy(c)
    ach = CGM_BYTES * n ** 3 * n_c / t / 1e9
    out[f"cgm_droplets_{n}"] = {"MLUPS": n ** 3 * n_c / t / 1e6, "steps": n_c, "droplets": len(spheres),
                               "volume_fraction": frac, "bytes_per_lup": CGM_BYTES, "moved_bytes_per_lup": 284,
                               "launch": shape, "autotune_MLUPS": tuned, "achieved_GBps": ach,
                               "frac_of_hbm_peak": ach / peak, "note": CGM_NOTE}
    return out


def _sc_batch(L, timed, steps, peak, domains=64, tune_cache="tmp"):
    """Interaction-strength sweep: `domains` periodic static-bubble boxes, sizes {32,48,64,96}^3, G U[-5.5, -4.5]
    (seed 6; the coexistence densities, hence the density ratio, follow G), radius n/4, nu = 0.0333, FP32, as one
    batch (two launches per step over all domains: pseudopotential, collision)."""
    import tempfile
    sweep = inputs.bubble_sweep(domains, seed=6)
    shapes = [(n, n, n) for n, _ in sweep]
    om = 1.0 / (3 * 0.0333 + 0.5)
    batch = L.lbm_batch_create(shapes, om, physics="sc", precision="fp32", G=[g for _, g in sweep])
    cells = sum(n ** 3 for n, _ in sweep)
    for k, (n, _) in enumerate(sweep):
        rho, u = inputs.static_bubble((n, n, n), n / 4.0)
        L.lbm_init_fields(L.lbm_batch_domain(batch, k), rho, u)
    cache = os.path.join(tempfile.gettempdir(), "lbm_tune_cache.json") if tune_cache == "tmp" else None
    tuned = L.lbm_autotune(batch, cache)
    L.lbm_batch_step(batch, 4)
    n_b = max(20, steps)
    t = timed(lambda n: L.lbm_batch_step(batch, n), n_b)
    L.lbm_sync(batch)
    info = L.lbm_batch_info(batch)
    L.lbm_destroy(batch)
    ach = 160 * cells * n_b / t / 1e9
    return {f"sc_batch_{domains}": {
        "MLUPS": cells * n_b / t / 1e6, "cells": cells, "steps": n_b, "bytes_per_lup": 160,
        "moved_bytes_per_lup": 236, "achieved_GBps": ach, "frac_of_hbm_peak": ach / peak, "launch": info,
        "autotune_MLUPS": tuned, "launches_per_step": 2,
        "note": "Shan-Chen interaction-strength sweep stepped as one batch: two passes per step "
                "(pseudopotential, then forced collision); 160 B/LUP algorithmic (populations read and written, psi "
                "written and read once); the two passes move 236 B"}}


def _sc(L, timed, steps, peak, sizes=(100, 256), launch="auto"):
    out = {}
    # Shan-Chen static bubble (Sec. III.G): periodic n^3, nu = 0.0333, G = -5,
    # sharp 1.95 / 0.15 droplet, FP32: the paper's 100^3 with R = 20, and 256^3
    # with R = 30 (the paper's largest radius; a sharp start much above it sends a
    # rarefaction wave into the droplet that empties its centre and diverges,
    # in the FP64 oracle as on the GPU).
    for n in sizes:
        R = 20.0 if n <= 100 else 30.0
        rho, u = inputs.static_bubble((n, n, n), R)
        c = L.lbm_create((n, n, n), 1 / (3 * 0.0333 + 0.5), physics="sc", precision="fp32", G=-5.0)
        L.lbm_init_fields(c, rho, u)
        tuned = L.lbm_autotune(c, None) if launch == "auto" else apply_launch(L, c, launch, None)
        shape = L.lbm_get_launch_shape(c)
        L.lbm_step(c, 3)
        n_c = max(20, steps // 2) * (8 if n == 100 else 1)
        t = timed(lambda k: L.lbm_step(c, k), n_c)
        L.lbm_reduce(c)
        L.lbm_destroy(c)
        ach = 160 * n ** 3 * n_c / t / 1e9
        out[f"sc_static_bubble_{n}"] = {
            "MLUPS": n ** 3 * n_c / t / 1e6, "steps": n_c, "radius": R, "bytes_per_lup": 160,
            "moved_bytes_per_lup": 152 if shape["variant"] == "fused" else 236, "achieved_GBps": ach,
            "frac_of_hbm_peak": ach / peak, "launch": shape, "autotune_MLUPS": tuned,
            "note": "fused: one kernel per step, psi of three planes in shared memory; direct: two passes "
                    "(pseudopotential, then collide); 160 B/LUP algorithmic (19 populations read and written, psi "
                    "written and read once)"}
    return out


def _rt(L, timed, steps, peak, launch="auto"):
    # Rayleigh-Taylor (Sec. III.H) on the colour-gradient step: 64 x 256 x 64, rho 3 over 1, Re 512, At 0.5,
    # walls at bottom and top, F = (rho - 2) g, FP32.  Timed from t = 0 (the interface is still flat-ish).
    W = 64
    g = 0.04 ** 2 / W
    nu = W * 0.04 / 512.0
    rho, u, phase = inputs.rayleigh_taylor(W)
    shape = (W, 4 * W, W)
    c = L.lbm_create(shape, 1 / (3 * nu + 0.5), periodic=(True, False, True), g=(0.0, -g, 0.0), rho_ref=2.0,
                     physics="cgm", precision="fp32", alpha_r=7 / 9, alpha_b=1 / 3, A=0.0, beta=0.7)
    L.lbm_init_fields(c, rho, u, phase=phase)
    tuned = L.lbm_autotune(c, None) if launch == "auto" else apply_launch(L, c, launch, None)
    shape_l = L.lbm_get_launch_shape(c)
    L.lbm_step(c, 3)
    n_c = max(20, steps // 2) * 4
    t = timed(lambda k: L.lbm_step(c, k), n_c)
    L.lbm_reduce(c)
    L.lbm_destroy(c)
    cells = W * 4 * W * W
    ach = CGM_BYTES * cells * n_c / t / 1e9
    return {"cgm_rayleigh_taylor_64x256x64": {
        "MLUPS": cells * n_c / t / 1e6, "steps": n_c, "bytes_per_lup": CGM_BYTES, "moved_bytes_per_lup": 284,
        "launch": shape_l, "autotune_MLUPS": tuned, "achieved_GBps": ach, "frac_of_hbm_peak": ach / peak,
        "note": "colour-gradient two-pass step with walls; " + CGM_NOTE}}


def _appd(L, timed, steps, n=256):
    # App. D's timing comparison on its workload, the 3D Taylor-Green vortex (Sec. III.E, u0 = 0.05, tau = 0.53):
    # raw- against central-moment collision, D3Q19, FP32 (HBM-bound) and FP64 (FP64-ALU-bound), n^3.
    rho, u = inputs.taylor_green_3d(n, u0=0.05)
    out = {}
    for prec in ("fp32", "fp64"):
        row = {}
        for lat in ("d3q19", "d3q27"):
            for coll in ("rm", "cm"):
                c = L.lbm_create((n, n, n), 1 / 0.53, precision=prec, collision=coll, lattice=lat)
                L.lbm_init_fields(c, rho, u)
                L.lbm_set_launch_shape(c, 0, 256, 0, 1)
                L.lbm_step(c, 3)
                k = max(20, steps // (4 if prec == "fp32" else 20))
                t = timed(lambda m: L.lbm_step(c, m), k)
                L.lbm_destroy(c)
                row[f"Q{lat[-2:]}-{coll.upper()}"] = {"MLUPS": n ** 3 * k / t / 1e6, "steps": k}
        base = row["Q19-RM"]["MLUPS"]
        row["time_relative_to_Q19-RM"] = {key: base / v["MLUPS"] for key, v in row.items()}
        out[prec] = row
    out["note"] = ("direct kernels, one node per thread; the paper's CPU times relative to Q19-RM at D = 128: "
                   "Q19-CM 1.06, Q27-RM 1.53, Q27-CM 1.82 (Table of App. D)")
    return {f"appD_timing_taylor_green_{n}": out}


def _channel(L, timed, steps, peak, n=512):
    # Body-force channel with the paper's regularized on-node walls on y (x, z periodic), 512^3, FP32, the same
    # start as the headline workload.
    rho, u = inputs.noise_box((n, n, n), amp=1e-3, seed=1)
    c = L.lbm_create((n, n, n), 1 / TAU, periodic=(True, False, True), g=G, precision="fp32",
                     wall_model="regularized")
    L.lbm_init_fields(c, rho, u)
    del rho, u
    L.lbm_step(c, 3)
    n_c = max(20, steps // 4)
    t = timed(lambda k: L.lbm_step(c, k), n_c)
    L.lbm_reduce(c)
    L.lbm_destroy(c)
    ach = 152 * n ** 3 * n_c / t / 1e9
    return {f"fluid_regularized_channel_{n}": {
        "MLUPS": n ** 3 * n_c / t / 1e6, "steps": n_c, "bytes_per_lup": 152, "achieved_GBps": ach,
        "frac_of_hbm_peak": ach / peak,
        "note": "fluid_step_channel_kernel (rows 1..n-2 in the periodic node code, regularized rebuild of rows 0 and "
                "n-1)"}}


def apply_launch(L, ctx, spec, tune_cache):
    """'auto': autotune (timed dry runs, state unchanged); 'direct[:threads]',
    'pair[:threads]', 'zpair[:threads]', 'fused:threads:planes' or 'tma:stages:ctas': a
    fixed launch shape (profiling).  Returns the tuned
    MLUPS or None."""
    if spec == "auto":
        return L.lbm_autotune(ctx, tune_cache)
    parts = spec.split(":")
    if parts[0] in ("direct", "pair", "zpair"):
        L.lbm_set_launch_shape(ctx, {"direct": 0, "pair": 2, "zpair": 4}[parts[0]],
                               int(parts[1]) if len(parts) > 1 else 256, 0, 1)
    elif parts[0] == "tma":
        L.lbm_set_launch_shape(ctx, 1, 256, int(parts[1]), int(parts[2]))
    elif parts[0] == "fused":
        L.lbm_set_launch_shape(ctx, 3, int(parts[1]), int(parts[2]), 1)
    else:
        raise ValueError(spec)
    return None


WARM_WEIGHTS = os.path.join(ROOT, "paper_2010_01628_gb300", "weights", "cavity128_warmstart.npz")


def warm_start_record():
    """The full warm-start study (512 training states, 32 held-out Reynolds
    numbers) from its committed record (python -m
    paper_2010_01628_gb300.surrogate; minutes of GPU time, so it is not re-run
    inside the benchmark).  Context beside the measured arm below."""
    try:
        with open(os.path.join(ROOT, "profiles", "warmstart_cavity128.json")) as fh:
            d = json.load(fh)
        d = {k: v for k, v in d.items() if k not in ("cases", "loss_history")}
        d["provenance"] = "recorded by the warm-start study run (profiles/warmstart_cavity128.json)"
        return d
    except Exception:
        return None


def warm_start_measured(L, torch, cases):
    """Time to the steady residual (1e-6), cold (from rest) and warm (from the
    committed network's prediction, inference inside the timed region), for the
    first `cases` held-out Reynolds numbers of the study, measured now; plus the
    solver's judgement of the network (prediction error against the cold run's
    converged fields, warm-vs-cold final fields)."""
    from paper_2010_01628_gb300 import surrogate as S

    w, meta = S.load_weights(WARM_WEIGHTS)
    n = int(meta["grid"])
    re_all = inputs.cavity_reynolds(meta["train_count"] + meta["heldout_count"], seed=meta["reynolds_seed"])
    held = [float(r) for r in re_all[meta["train_count"]:][:cases]]
    net = L.lbm_cnn_create((n, n, n), w)
    try:
        with ClockSampler(smi_device_id(torch)) as clk:
            rep = S.evaluate(net, n, held, tol=meta["tol"], check_every=meta["check_every"])
    finally:
        L.lbm_cnn_destroy(net)
    rep["clocks"] = clk.summary()
    rep.update({"grid": n, "heldout_cases": len(held), "tol": meta["tol"], "check_every": meta["check_every"],
                "weights": os.path.relpath(WARM_WEIGHTS, ROOT), "timer": "host wall clock, synchronised",
                "provenance": "measured in this benchmark run"})
    return rep


def time_steps(L, torch, ctx, steps, stream):
    start = torch.cuda.Event(enable_timing=True)
    stop = torch.cuda.Event(enable_timing=True)
    start.record(stream)
    L.lbm_step(ctx, steps)
    stop.record(stream)
    stop.synchronize()
    return start.elapsed_time(stop) / 1e3


def run_ours(args):
    import torch
    import torch.distributed as dist

    ranks = Ranks(device="cuda")
    world, rank, local = ranks.world, ranks.rank, ranks.local
    torch.cuda.set_device(local)
    if world > 1:
        dist.init_process_group("nccl", device_id=torch.device("cuda", local))
    from paper_2010_01628_gb300 import binding as L

    def barrier():
        ranks.barrier()
        torch.cuda.synchronize()

    max_over_ranks = ranks.max_over_ranks

    n, prec = args.n, args.precision
    stream = torch.cuda.current_stream()
    if args.only == "fma-probe":
        f64, f32 = L.lbm_probe_fma_rate()
        print(json.dumps({"only": "fma-probe", "fp64_fma_per_s": f64, "fp32_fma_per_s": f32}), flush=True)
        return 0
    if args.only == "warmstart":
        print(json.dumps({"only": "warmstart", "warm_start": warm_start_measured(L, torch, args.warm_cases)}),
              flush=True)
        return 0
    if args.only:
        peak, _ = measured_peaks()
        res = extra_workloads(L, torch, stream, args.steps, peak, only=args.only, domains=args.domains,
                              n_cgm=args.n if args.n != N else 256, tune_cache=args.tune_cache,
                              n_only=args.n if args.n != N else None, ranks=ranks, launch=args.launch)
        if rank == 0:
            print(json.dumps({"only": args.only, "workloads": res}), flush=True)
        return 0
    rho, u = inputs.noise_box((n, n, n), amp=1e-3, seed=1)
    import tempfile
    tune_cache = os.path.join(tempfile.gettempdir(), "lbm_tune_cache.json") if args.tune_cache == "tmp" else None
    ctx = L.lbm_create((n, n, n), 1 / TAU, g=G, precision=prec)
    L.lbm_init_fields(ctx, rho, u)
    tuned = apply_launch(L, ctx, args.launch, tune_cache)
    shape = L.lbm_get_launch_shape(ctx)
    L.lbm_step(ctx, args.warmup)
    barrier()
    with ClockSampler(smi_device_id(torch)) as clk:
        barrier()
        t_dev = time_steps(L, torch, ctx, args.steps, stream)
        barrier()
    t_dev = max_over_ranks(t_dev)
    cells = n ** 3
    value = world * cells * args.steps / t_dev / 1e6
    launch_s = t_dev / args.steps
    peak, peak_kind = measured_peaks()
    achieved = algorithmic_bytes(n, prec) / launch_s / 1e9
    traffic = committed_traffic(f"fluid_step_{shape['variant']}_{prec}_{n}")
    L.lbm_reduce(ctx)  # divergence check of the timed run (raises on NaN)
    L.lbm_destroy(ctx)

    # Other storage precisions of the same workload (short runs, same method).
    variants = {}
    if not args.no_variants:
        for vp in ("fp64", "fp16", "bf16"):
            if vp == prec:
                continue
            vsteps = max(10, args.steps // 10)
            c2 = L.lbm_create((n, n, n), 1 / TAU, g=G, precision=vp)
            L.lbm_init_fields(c2, rho, u)
            apply_launch(L, c2, "auto", tune_cache)
            vshape = L.lbm_get_launch_shape(c2)
            L.lbm_step(c2, 3)
            barrier()
            tv = max_over_ranks(time_steps(L, torch, c2, vsteps, stream))
            L.lbm_destroy(c2)
            torch.cuda.empty_cache()
            ach = algorithmic_bytes(n, vp) / (tv / vsteps) / 1e9
            variants[vp] = {"MLUPS": world * cells * vsteps / tv / 1e6, "steps": vsteps,
                            "achieved_GBps": ach, "frac_of_hbm_peak": ach / peak, "launch": vshape}

    # End to end through the C ABI with host buffers: upload the initial
    # fields from pinned host memory, K steps, read the fields back.
    e2e = None
    if not args.no_e2e:
        rho_h = torch.from_numpy(rho).pin_memory()
        u_h = torch.from_numpy(u).pin_memory()
        rho_o = torch.empty_like(rho_h).pin_memory()
        u_o = torch.empty_like(u_h).pin_memory()
        c3 = L.lbm_create((n, n, n), 1 / TAU, g=G, precision=prec)
        apply_launch(L, c3, args.launch, tune_cache)
        # one untimed pass through the same calls (first-use costs of the copy path)
        L.lbm_init_fields(c3, rho_h, u_h)
        L.lbm_step(c3, 1)
        L.lbm_fields(c3, (n, n, n), rho=rho_o, u=u_o)
        torch.cuda.synchronize()
        barrier()
        t0 = time.perf_counter()
        L.lbm_init_fields(c3, rho_h, u_h)
        L.lbm_step(c3, args.steps)
        L.lbm_fields(c3, (n, n, n), rho=rho_o, u=u_o)
        torch.cuda.synchronize()
        te = max_over_ranks(time.perf_counter() - t0)
        L.lbm_destroy(c3)
        io_bytes = (rho.nbytes + u.nbytes)
        e2e = {"value": world * cells * args.steps / te / 1e6, "unit": "MLUPS",
               "h2d_bytes_per_step": io_bytes / args.steps, "d2h_bytes_per_step": io_bytes / args.steps,
               "note": "lbm_init_fields(pinned host rho,u) + K x lbm_step + lbm_fields(pinned host rho,u)"}

    extra = None
    if not args.no_variants:
        extra = extra_workloads(L, torch, stream, args.steps, peak, ranks=ranks)
        torch.cuda.empty_cache()

    warm = None
    if args.warm_cases > 0 and rank == 0:
        warm = warm_start_measured(L, torch, args.warm_cases)
        torch.cuda.empty_cache()

    cpu = None
    if rank == 0 and world == 1 and not args.no_cpu:
        cpu = cpu_baseline_sample()

    if rank == 0:
        line = {"metric": METRIC, "value": value, "unit": "MLUPS", "n_gpus": world, "steps": args.steps,
                "warmup": args.warmup, "ms_per_step": launch_s * 1e3, "higher_is_better": True, "scaling": "weak",
                "vs_baseline": None, "dtype": DTYPE_NAME[prec], "data": "synthetic",
                "config": workload_config(n, prec) | {"parallelism": f"replicas x{world}", "launch": shape,
                                                      "autotune_MLUPS": tuned},
                "roofline": {"bound": "hbm", "achieved": achieved, "peak": peak, "unit": "GB/s",
                             "frac": achieved / peak, "traffic": traffic, "peak_kind": peak_kind,
                             "kernel": {"tma": "fluid_step_tma_kernel", "pair": "fluid_step_pair_kernel",
                                        "zpair": "fluid_step_zpair_kernel"}.get(
                                 shape["variant"], "fluid_step_kernel") + f"<{prec}>",
                             "algorithmic_bytes_per_launch": algorithmic_bytes(n, prec)},
                "cpu_baseline": cpu, "e2e": e2e, "gpu_launches": args.steps, "clocks": clk.summary(),
                "variants": variants, "workloads": extra, "warm_start": warm,
                "warm_start_study": warm_start_record()}
        print(json.dumps(line), flush=True)
    if world > 1:
        dist.destroy_process_group()
    return 0


def main():
    ap = argparse.ArgumentParser()
    ap.add_argument("--gpus", type=int, default=1)
    ap.add_argument("--steps", type=int, default=1000)
    ap.add_argument("--warmup", type=int, default=20)
    ap.add_argument("--impl", default="ours", choices=["ours", "reference"])
    ap.add_argument("--precision", default="fp32", choices=list(BYTES_PER_VALUE))
    ap.add_argument("--n", type=int, default=N)
    ap.add_argument("--no-variants", action="store_true")
    ap.add_argument("--no-e2e", action="store_true")
    ap.add_argument("--no-cpu", action="store_true")
    ap.add_argument("--warm-cases", type=int, default=8,
                    help="held-out cavities timed warm vs cold (0: skip the measured warm-start arm)")
    ap.add_argument("--only", choices=["tg32", "mhd_batch", "cgm", "cgm_batch", "sc", "sc_batch", "rt", "channel",
                                       "appd", "fma-probe", "warmstart", "cnn"],
                    default=None,
                    help="run one secondary workload alone (profiling)")
    ap.add_argument("--domains", type=int, default=64, help="domains of the MHD batch workload")
    ap.add_argument("--launch", default="auto",
                    help="launch shape: auto | direct[:threads] | pair[:threads] | "
                         "zpair[:threads] | tma:stages:ctas | fused:threads:planes")
    ap.add_argument("--tune-cache", default="tmp", choices=["tmp", "none"],
                    help="autotuner cache of the batch workload: a file in the temp dir, or none")
    args = ap.parse_args()
    if args.warmup < 3:
        args.warmup = 3
    if args.impl == "reference":
        return run_reference(args)
    return run_ours(args)


if __name__ == "__main__":
    sys.exit(main())
