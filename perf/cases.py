"""Timed workloads of the library, as a user's program runs them through the public binding.

A pass of a flow case is what such a program repeats: set the fields (``lbm_init_fields``, device tensors), advance n
steps (``lbm_step``, ``lbm_batch_step`` or ``lbm_run_to_steady``) and read the fields back (``lbm_fields``), kept as a
snapshot in the solver's own storage precision.  The context, its launch shape and the buffers are made once, in
``prepare``.  A pass of the network case is one forward and backward pass of the warm-start network.

``exact`` states the same workloads in plain torch binary64: populations stored unshifted, moments by matrix products,
the two colours as two distributions.
"""
import functools
import math
import os

import numpy as np
import torch

from paper_2010_01628_gb300 import binding as L

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))
WEIGHTS = os.path.join(ROOT, "paper_2010_01628_gb300", "weights", "cavity128_warmstart.npz")
DEV = "cuda"
F64 = torch.float64
SWEEP_SIZES = (32, 48, 64, 96)
DTYPES = {"fp64": torch.float64, "fp32": torch.float32, "fp16": torch.float16, "bf16": torch.bfloat16}


def listed():
    return [
        # accuracy and convergence studies: the 32^3 Taylor-Green vortex in double precision, 200 steps
        {"name": "taylor_green_32_fp64", "kind": "vortex", "nx": 32, "ny": 32, "nz": 32, "steps": 200, "precision": "fp64"},
        # 2D validation runs (one node in z): the double shear layer, small enough that launches count
        {"name": "shear_layer_256_fp32", "kind": "shear", "nx": 256, "ny": 256, "nz": 1, "steps": 100, "precision": "fp32"},
        # the warm-started lid-driven cavity: network inference, then 300 walled steps with residual checks
        {"name": "cavity_128_warm", "kind": "cavity", "nx": 128, "ny": 128, "nz": 128, "steps": 300, "precision": "fp32"},
        # a channel with the on-node regularized walls, ragged in all three axes
        {"name": "channel_regularized", "kind": "channel", "nx": 250, "ny": 129, "nz": 190, "steps": 50, "precision": "fp32"},
        # the headline flow: 512^3 periodic box with a body force, autotuned
        {"name": "box_512_fp32", "kind": "box", "nx": 512, "ny": 512, "nz": 512, "steps": 20, "precision": "fp32",
         "autotune": True},
        # the same flow stored in 16 bits, autotuned
        {"name": "box_256_fp16", "kind": "box", "nx": 256, "ny": 256, "nz": 256, "steps": 100, "precision": "fp16",
         "autotune": True},
        # a Hartmann-number sweep: 64 uneven magnetohydrodynamic channels in one batch
        {"name": "hartmann_sweep_64", "kind": "sweep_mhd", "domains": 64, "steps": 50, "precision": "fp32"},
        # colour-gradient droplets, density ratio 10
        {"name": "droplets_256", "kind": "droplets", "nx": 256, "ny": 256, "nz": 256, "steps": 40, "precision": "fp32"},
        # Rayleigh-Taylor instability: colour gradient between two walls
        {"name": "rayleigh_taylor_64", "kind": "rt", "nx": 64, "ny": 256, "nz": 64, "steps": 100, "precision": "fp32"},
        # the Shan-Chen static bubble of the Laplace test
        {"name": "bubble_100", "kind": "bubble", "nx": 100, "ny": 100, "nz": 100, "steps": 200, "precision": "fp32"},
        # an interaction-strength sweep: 64 uneven Shan-Chen boxes in one batch
        {"name": "bubble_sweep_64", "kind": "sweep_sc", "domains": 64, "steps": 50, "precision": "fp32"},
        # training the warm-start network: forward and backward at its full grid
        {"name": "network_gradient_128", "kind": "network", "nx": 128, "ny": 128, "nz": 128},
    ]


def draw(rng):
    def size(lo, hi):
        return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))

    def steps(nodes, rate, most, lo=8):
        # at most about 60 ms of stepping at `rate` updates per second, never less than `lo` steps
        return max(lo, min(size(lo, most), int(0.06 * rate / nodes)))

    kind = rng.choice(["vortex", "shear", "cavity", "channel", "box", "box", "box", "sweep_mhd", "droplets", "rt", "bubble",
                       "sweep_sc", "network"])
    c = {"kind": kind, "precision": "fp32"}
    if kind.startswith("sweep"):
        c["domains"] = size(4, 64)
        c["steps"] = size(10, 50)
        return c
    if kind == "vortex":
        n = size(16, 160)
        c.update(nx=n, ny=n, nz=n, precision="fp64", steps=steps(n ** 3, 2e9, 200))
    elif kind == "shear":
        n = size(128, 1024)
        c.update(nx=n, ny=n, nz=1, precision=rng.choice(["fp32", "fp64"]), steps=size(20, 100))
    elif kind == "cavity":
        n = size(48, 160)
        c.update(nx=n, ny=n, nz=n, steps=size(100, 300))
    elif kind == "channel":
        c.update(nx=size(48, 300), ny=size(33, 300), nz=size(48, 300))
        c["steps"] = steps(c["nx"] * c["ny"] * c["nz"], 4e10, 100)
    elif kind == "box":
        c["precision"] = rng.choice(["fp32", "fp32", "fp16", "bf16"])
        c.update(nx=size(48, 480), ny=size(48, 480), nz=size(48, 480), autotune=rng.choice([True, False]))
        c["steps"] = steps(c["nx"] * c["ny"] * c["nz"], 4e10, 100)
    elif kind == "droplets":
        n = size(96, 256)
        c.update(nx=n, ny=n, nz=n, steps=steps(n ** 3, 1.5e10, 100))
    elif kind == "rt":
        n = size(32, 96)
        c.update(nx=n, ny=4 * n, nz=n, steps=size(20, 100))
    elif kind == "bubble":
        n = size(72, 256)
        c.update(nx=n, ny=n, nz=n, steps=steps(n ** 3, 2e10, 200))
    else:
        c.update(nx=size(32, 128), ny=size(32, 128), nz=size(32, 128))
        del c["precision"]
    return c


# ---- inputs -----------------------------------------------------------------------------------------------------
def _gen(seed):
    g = torch.Generator(device=DEV)
    g.manual_seed(int(seed))
    return g


def _axes(nx, ny, nz):
    a = [torch.arange(n, dtype=F64, device=DEV) for n in (nx, ny, nz)]
    return a[0].view(1, 1, -1), a[1].view(1, -1, 1), a[2].view(-1, 1, 1)


def _noise(g, amp, nx, ny, nz):
    return (torch.rand((3, nz, ny, nx), generator=g, dtype=F64, device=DEV) * 2 - 1) * amp


def _spheres(n, rng, r_min, r_max, fraction=0.10, gap=4.0):
    """Non-overlapping spheres (centre, radius) in a periodic cube, added until they fill `fraction` of it."""
    c, r, vol = np.zeros((0, 3)), np.zeros(0), 0.0
    for _ in range(20000):
        if vol >= fraction * n ** 3:
            break
        rr, cc = rng.uniform(r_min, r_max), rng.uniform(0, n, size=3)
        d = np.abs(c - cc)
        d = np.minimum(d, n - d)
        if np.any((d * d).sum(axis=1) < (r + rr + gap) ** 2):
            continue
        c, r = np.vstack([c, cc]), np.append(r, rr)
        vol += 4.0 / 3.0 * math.pi * rr ** 3
    return c, r


def _droplet_fields(n, rng, r_min, r_max, ratio, width=4.0):
    """rho and the order parameter of tanh-profiled droplets of density `ratio` in a fluid of density 1."""
    phase = torch.full((n, n, n), -1.0, dtype=F64, device=DEV)
    for c, r in zip(*_spheres(n, rng, r_min, r_max)):
        reach = min(int(math.ceil(r + 6 * width)), n // 2 - 1)
        i = [torch.arange(int(c[a]) - reach, int(c[a]) + reach + 1, device=DEV) for a in range(3)]
        d = [(t.to(F64) - float(c[a])) ** 2 for a, t in enumerate(i)]
        dist = (d[2].view(-1, 1, 1) + d[1].view(1, -1, 1) + d[0].view(1, 1, -1)).sqrt_()
        at = ((i[2] % n).view(-1, 1, 1), (i[1] % n).view(1, -1, 1), (i[0] % n).view(1, 1, -1))
        phase[at] = torch.maximum(phase[at], torch.tanh(2 * (float(r) - dist) / width))
    return ratio * (1 + phase) / 2 + (1 - phase) / 2, phase


def _bubble_fields(n, radius, shift, width=0.0):
    x, y, z = _axes(n, n, n)
    c = (n - 1) / 2.0
    d2 = (x - c - shift[0]) ** 2 + (y - c - shift[1]) ** 2 + (z - c - shift[2]) ** 2
    if width:
        return 0.15 + 0.9 * (1 + torch.tanh((radius - d2.sqrt()) / width))
    return torch.where(d2 <= radius * radius, 1.95, 0.15).to(F64)


def _problem(case, seed):
    """What one case solves: `par`, the arguments of lbm_create, and the initial fields."""
    kind, rng, g = case["kind"], np.random.default_rng(seed), _gen(seed)
    nx, ny, nz = case["nx"], case["ny"], case["nz"]
    par, fields = {"precision": case["precision"]}, {}
    rho = torch.ones((nz, ny, nx), dtype=F64, device=DEV)
    x, y, z = _axes(nx, ny, nz)
    if kind == "vortex":  # Taylor-Green, its origin moved by the seed
        k, s = 2 * math.pi / nx, rng.uniform(0, 2 * math.pi, 3)
        X, Y, Z = k * x + s[0], k * y + s[1], k * z + s[2]
        u = 0.05 * torch.stack([X.cos() * Y.sin() * Z.sin(), -0.5 * X.sin() * Y.cos() * Z.sin(), -0.5 * X.sin() * Y.sin() * Z.cos()])
        omega = 1 / 0.53
    elif kind == "shear":  # double shear layer, Re = 3e4, moved along x by the seed
        u0 = 0.57 / math.sqrt(3.0)
        Y, X = y / ny, x / nx + rng.uniform()
        ux = torch.where(Y <= 0.5, torch.tanh(80 * (Y - 0.25)), torch.tanh(80 * (0.75 - Y))) * u0
        uy = u0 * 0.05 * torch.sin(2 * math.pi * (X + 0.25))
        u = torch.stack([ux.expand(nz, ny, nx), uy.expand(nz, ny, nx), torch.zeros_like(rho)])
        omega = 1 / (3 * u0 * ny / 3e4 + 0.5)
    elif kind == "cavity":  # lid along +x at 0.1
        re = rng.uniform(100.0, 1000.0)
        par.update(periodic=(False, False, False), lid_u=(0.1, 0.0, 0.0))
        omega, u = 1 / (3 * 0.1 * nx / re + 0.5), None
        fields["reynolds"] = re
    elif kind == "channel":
        par.update(periodic=(True, False, True), wall_model="regularized", g=(1e-6, 0.0, 0.0))
        omega, u = 1 / 0.6, _noise(g, 1e-3, nx, ny, nz)
    elif kind == "box":
        par.update(g=(1e-6, 0.0, 0.0))
        omega, u = 1 / 0.6, _noise(g, 1e-3, nx, ny, nz)
    elif kind == "droplets":
        omega, ratio = 1 / 0.8, 10.0
        par.update(physics="cgm", alpha_b=1 / 3, alpha_r=1 - (2 / 3) / ratio, A=9e-4 * omega / 4, beta=0.7)
        rho, fields["phase"] = _droplet_fields(nx, rng, 8.0, 24.0, ratio)
        u = torch.zeros((3, nz, ny, nx), dtype=F64, device=DEV)
    elif kind == "rt":  # heavy fluid over light fluid, the interface moved by the seed
        W, s = nx, rng.uniform(0, 2 * math.pi, 2)
        grav = 0.04 ** 2 / W
        omega = 1 / (3 * W * 0.04 / 512 + 0.5)
        par.update(physics="cgm", alpha_b=1 / 3, alpha_r=7 / 9, A=0.0, beta=0.7, periodic=(True, False, True), g=(0.0, -grav, 0.0), rho_ref=2.0)
        heavy = y > 0.5 * ny + 0.05 * W * (torch.cos(2 * math.pi * x / W + s[0]) + torch.cos(2 * math.pi * z / W + s[1]))
        rho = torch.where(heavy, 3.0, 1.0).to(F64)
        fields["phase"] = torch.where(heavy, 1.0, -1.0).to(F64)
        u = torch.zeros((3, nz, ny, nx), dtype=F64, device=DEV)
    elif kind == "bubble":
        par.update(physics="sc", G=-5.0)
        rho = _bubble_fields(nx, rng.uniform(15.0, 30.0), rng.uniform(-2, 2, 3))
        omega, u = 1 / (3 * 0.0333 + 0.5), torch.zeros((3, nz, ny, nx), dtype=F64, device=DEV)
    else:
        raise ValueError(kind)
    fields.update(rho=rho.contiguous(), u=u)
    return omega, par, fields


def _sweep(case, seed):
    """Sizes, shared and per-domain parameters, and the initial fields of every domain of a sweep.  The sizes depend on the
    number of domains alone, so that a sweep's cost does not change with the seed."""
    nd = case["domains"]
    sizes = [SWEEP_SIZES[k] for k in np.random.default_rng(nd).integers(0, 4, nd)]
    rng = np.random.default_rng(seed)
    par = {"precision": case["precision"]}
    fields = []
    if case["kind"] == "sweep_mhd":  # Hartmann channels, Ha in [1, 20]
        nu = 0.1
        b0 = [2 * rng.uniform(1.0, 20.0) * nu / n for n in sizes]
        omega = 1 / (3 * nu + 0.5)
        par.update(physics="mhd", periodic=(True, False, True), tau_m=0.5 + nu / 0.25, b_wall=[(0.0, b, 0.0) for b in b0],
                   g=[(8 * nu * 0.01 / n ** 2, 0.0, 0.0) for n in sizes])
        g = _gen(seed)
        for n, b in zip(sizes, b0):
            B = torch.zeros((3, n, n, n), dtype=F64, device=DEV)
            B[1] = b
            fields.append({"rho": torch.ones((n, n, n), dtype=F64, device=DEV), "u": _noise(g, 1e-3, n, n, n), "B": B})
    else:  # static bubbles with a smooth start (stable below G = -5 too), interaction strength in [-5.2, -4.5]
        omega = 1 / (3 * 0.0333 + 0.5)
        par.update(physics="sc", G=[float(v) for v in rng.uniform(-5.2, -4.5, nd)])
        for n in sizes:
            fields.append({"rho": _bubble_fields(n, n / 4.0, rng.uniform(-1, 1, 3), 3.0), "u": torch.zeros((3, n, n, n), dtype=F64, device=DEV)})
    return sizes, omega, par, fields


def _network_inputs(case, seed):
    """Reynolds number, weights and a smooth steady-like target field for one training step."""
    nx, ny, nz = case["nx"], case["ny"], case["nz"]
    rng = np.random.default_rng(seed)
    w = np.load(WEIGHTS)["weights"].astype(np.float32)
    w = w * (1 + 0.05 * rng.standard_normal(w.size).astype(np.float32))
    x, y, z = _axes(nx, ny, nz)
    X, Y, Z = (x + 0.5) / nx, (y + 0.5) / ny, (z + 0.5) / nz
    a = rng.uniform(0.5, 1.5, 4)
    u = torch.stack([0.1 * a[0] * Y ** 4 * torch.sin(math.pi * X) * torch.sin(math.pi * Z),
                     -0.03 * a[1] * torch.sin(2 * math.pi * X) * torch.sin(math.pi * Y) * torch.sin(math.pi * Z),
                     0.01 * a[2] * torch.sin(math.pi * X) * torch.sin(math.pi * Y) * torch.sin(2 * math.pi * Z)]).contiguous()
    rho = (1 + 0.01 * a[3] * (X - 0.5) * Y * (1 + 0 * Z)).contiguous()
    return float(rng.uniform(100.0, 1000.0)), w, rho, u


# ---- the passes -------------------------------------------------------------------------------------------------
class _State:
    """Handles, inputs and output buffers of one prepared case."""

    def __init__(self, case):
        self.case, self.ctx, self.net = case, None, None

    def __del__(self):
        L.lbm_destroy(self.ctx)
        L.lbm_cnn_destroy(self.net)


def _outputs(n, keys):
    return {k: torch.empty((3 if k in "uB" else 1) * n, dtype=F64, device=DEV) for k in keys}


def prepare(case, seed):
    s = _State(case)
    kind = case["kind"]
    if kind == "network":
        s.shape = (case["nx"], case["ny"], case["nz"])
        s.re, w, s.rho, s.u = _network_inputs(case, seed)
        s.net = L.lbm_cnn_create(s.shape, w)
        L.lbm_cnn_set_input(s.net, s.re)
        return s
    if kind.startswith("sweep"):
        s.sizes, omega, par, s.fields = _sweep(case, seed)
        s.ctx = L.lbm_batch_create([(n, n, n) for n in s.sizes], omega, **par)
        s.views = [L.lbm_batch_domain(s.ctx, k) for k in range(len(s.sizes))]
        s.out = _outputs(sum(n ** 3 for n in s.sizes), ("rho", "u", "B") if kind == "sweep_mhd" else ("rho", "u"))
        s.parts, at = [], 0
        for n in s.sizes:
            s.parts.append({k: v[at * (3 if k in "uB" else 1):(at + n ** 3) * (3 if k in "uB" else 1)] for k, v in s.out.items()})
            at += n ** 3
        return s
    omega, par, s.fields = _problem(case, seed)
    s.shape = (case["nx"], case["ny"], case["nz"])
    s.ctx = L.lbm_create(s.shape, omega, **par)
    if kind == "cavity":
        s.net = L.lbm_cnn_create(s.shape, np.load(WEIGHTS)["weights"].astype(np.float32))
    if case.get("autotune"):
        L.lbm_init_fields(s.ctx, s.fields["rho"], s.fields["u"])
        L.lbm_autotune(s.ctx, None)
    s.out = _outputs(case["nx"] * case["ny"] * case["nz"], ("rho", "u", "phase") if "phase" in s.fields else ("rho", "u"))
    return s


def run(s):
    case = s.case
    kind = case["kind"]
    if kind == "network":
        loss, grad = L.lbm_cnn_gradient(s.net, s.rho, s.u)
        return {"loss": loss, "gradient": grad}
    dtype = DTYPES[case["precision"]]
    if kind.startswith("sweep"):
        for v, f in zip(s.views, s.fields):
            L.lbm_init_fields(v, f["rho"], f["u"], B=f.get("B"))
        L.lbm_batch_step(s.ctx, case["steps"])
        for n, v, p in zip(s.sizes, s.views, s.parts):
            L.lbm_fields(v, (n, n, n), rho=p["rho"], u=p["u"], B=p.get("B"), want=())
        return {k: v.to(dtype) for k, v in s.out.items()}
    out = {}
    if kind == "cavity":
        L.lbm_cnn_warm_start(s.net, s.ctx, s.fields["reynolds"])
        out["steps"], out["residual"] = L.lbm_run_to_steady(s.ctx, case["steps"], 100, 1e-12)
    else:
        L.lbm_init_fields(s.ctx, s.fields["rho"], s.fields["u"], phase=s.fields.get("phase"))
        L.lbm_step(s.ctx, case["steps"])
    L.lbm_fields(s.ctx, s.shape, rho=s.out["rho"], u=s.out["u"], phase=s.out.get("phase"), want=())
    out.update({k: v.to(dtype) for k, v in s.out.items()})
    return out


# floating-point operations of one node and step (multiply-adds counted as two), by hand from the printed equations
_FLOPS = {"vortex": 300, "shear": 300, "cavity": 300, "channel": 300, "box": 300, "droplets": 650, "rt": 650, "bubble": 400,
          "sweep_mhd": 550, "sweep_sc": 400}


def work(case):
    """The fields that go in and come out, once each, and the arithmetic of the updates: the state between two steps of a
    pass need not leave the chip, so it is not counted."""
    if case["kind"] == "network":
        n = case["nx"] * case["ny"] * case["nz"]
        macs = 27 * (16 * 32 + 32 * 32 + 32 * 32 + 32 * 4)
        return {"bytes": 4 * 8 * n, "flops": 2 * n * (3 * macs - 27 * 16 * 32)}  # no input gradient at the first layer
    if case["kind"].startswith("sweep"):
        nd = case["domains"]
        n = sum(SWEEP_SIZES[k] ** 3 for k in np.random.default_rng(nd).integers(0, 4, nd))
        values = 7 if case["kind"] == "sweep_mhd" else 4
    else:
        n = case["nx"] * case["ny"] * case["nz"]
        values = 5 if case["kind"] in ("droplets", "rt") else 4
    stored = {"fp64": 8, "fp32": 4, "fp16": 2, "bf16": 2}[case["precision"]]
    read = 0 if case["kind"] == "cavity" else 8 * values
    return {"bytes": n * (read + stored * values), "flops": n * case["steps"] * _FLOPS[case["kind"]]}


# ---- the same in 64 bits ----------------------------------------------------------------------------------------
_C = [(0, 0, 0), (-1, 0, 0), (0, -1, 0), (0, 0, -1), (-1, -1, 0), (-1, 1, 0), (-1, 0, -1), (-1, 0, 1), (0, -1, -1), (0, -1, 1)]
_C += [tuple(-v for v in c) for c in _C[1:]]
_OPP = [0] + list(range(10, 19)) + list(range(1, 10))
_W = [(1 / 3, 1 / 18, 1 / 36)[sum(v * v for v in c)] for c in _C]
_EXP = [(0, 0, 0), (1, 0, 0), (0, 1, 0), (0, 0, 1), (2, 0, 0), (0, 2, 0), (0, 0, 2), (1, 1, 0), (1, 0, 1), (0, 1, 1),
        (2, 1, 0), (1, 2, 0), (2, 0, 1), (1, 0, 2), (0, 2, 1), (0, 1, 2), (2, 2, 0), (2, 0, 2), (0, 2, 2)]
_PAIRS = [(0, 1, 7), (0, 2, 8), (1, 2, 9)]  # axes a, b and the row of the moment ab


@functools.lru_cache(maxsize=1)
def _matrices():
    m = np.array([[c[0] ** e[0] * c[1] ** e[1] * c[2] ** e[2] for c in _C] for e in _EXP], dtype=np.float64)
    return torch.tensor(m, device=DEV), torch.tensor(np.linalg.inv(m), device=DEV)


def _stream(f, periodic, lid=None):
    """Pull: out_i(x) = f_i(x - c_i); from behind a wall, the node's own opposite population, with the lid's term."""
    g = torch.empty_like(f)
    for i, c in enumerate(_C):
        g[i] = torch.roll(f[i], (c[2], c[1], c[0]), (-3, -2, -1))
        for a in range(3):
            if c[a] and not periodic[a]:
                at = 0 if c[a] > 0 else -1
                g[i].select(-1 - a, at).copy_(f[_OPP[i]].select(-1 - a, at))
        if lid is not None and c[1] < 0 and not periodic[1]:
            g[i][..., -1, :] += 6 * _W[i] * sum(c[a] * lid[a] for a in range(3))
    return g


def _gradient_sum(v, periodic):
    """sum_i w_i c_i v(x + c_i), with the node's own value behind a wall."""
    s = [torch.zeros_like(v) for _ in range(3)]
    for i, c in enumerate(_C[1:], 1):
        t = torch.roll(v, (-c[2], -c[1], -c[0]), (-3, -2, -1))
        for a in range(3):
            if c[a] and not periodic[a]:
                at = -1 if c[a] > 0 else 0
                t.select(-1 - a, at).copy_(v.select(-1 - a, at))
        for a in range(3):
            if c[a]:
                s[a] += c[a] * _W[i] * t
    return s


def _raw(f):
    m = _matrices()[0][:10] @ f.reshape(19, -1)
    return m.view(10, *f.shape[1:])


def _collide(m, F, omega, alpha=None, u=None):
    """Post-collision populations from the ten raw moments up to second order and the force; alpha: the colour gradient's."""
    rho = m[0]
    if u is None:
        u = [(m[1 + a] + 0.5 * F[a]) / rho for a in range(3)]
    h = [0.5 * F[a] for a in range(3)]
    keep = 1 - omega
    diag = [m[4 + a] - rho * u[a] ** 2 + 2 * u[a] * h[a] for a in range(3)]
    trace = rho if alpha is None else 1.5 * rho * (1 - alpha)
    mean = (diag[0] + diag[1] + diag[2]) / 3
    k2 = [trace / 3 + keep * (d - mean) for d in diag]
    r = torch.empty((19,) + tuple(rho.shape), dtype=F64, device=rho.device)
    r[0] = rho
    for a in range(3):
        r[1 + a] = rho * u[a] + h[a]
        r[4 + a] = k2[a] + 2 * u[a] * h[a] + rho * u[a] ** 2
    for (a, b, row), aab, abb, aabb in zip(_PAIRS, (10, 12, 14), (11, 13, 15), (16, 17, 18)):
        kab = keep * (m[row] - rho * u[a] * u[b] + u[a] * h[b] + u[b] * h[a])
        kaab, kabb, kaabb = h[b] / 3, h[a] / 3, rho / 9
        if alpha is not None:
            e = rho * (3 * alpha - 1) / 6
            kaab, kabb = kaab + e * u[b], kabb + e * u[a]
            s2 = u[a] ** 2 + u[b] ** 2
            kaabb = rho * (1 + s2 - alpha * (1 + 3 * s2)) / 6
        r[row] = kab + u[a] * h[b] + u[b] * h[a] + rho * u[a] * u[b]
        r[aab] = kaab + 2 * u[a] * kab + u[b] * k2[a] + u[a] ** 2 * h[b] + 2 * u[a] * u[b] * h[a] + rho * u[a] ** 2 * u[b]
        r[abb] = kabb + 2 * u[b] * kab + u[a] * k2[b] + u[b] ** 2 * h[a] + 2 * u[a] * u[b] * h[b] + rho * u[b] ** 2 * u[a]
        r[aabb] = (kaabb + 2 * u[b] * kaab + 2 * u[a] * kabb + u[b] ** 2 * k2[a] + u[a] ** 2 * k2[b] + 4 * u[a] * u[b] * kab
                   + 2 * u[a] * u[b] ** 2 * h[a] + 2 * u[b] * u[a] ** 2 * h[b] + rho * u[a] ** 2 * u[b] ** 2)
    return (_matrices()[1] @ r.view(19, -1)).view_as(r)


def _equilibrium(rho, u, alpha=None):
    zero = torch.zeros_like(rho)
    m = torch.stack([rho] + [rho * v for v in u] + [rho * v * v for v in u] + [rho * u[a] * u[b] for a, b, _ in _PAIRS])
    return _collide(m, [zero] * 3, 1.0, alpha, u)


def _regularize(f, y, sign, uw, g):
    """Rebuilds the populations of the wall row y (f: pulled) from the known ones; sign: the inward normal's."""
    t = f[..., y, :]
    s0 = sum(t[i] for i in range(19) if _C[i][1] == 0)
    out = sum(t[i] for i in range(19) if _C[i][1] == -sign)
    rho = (s0 + 2 * out) / (1 - sign * uw[1] + 0.5 * sign * g[1])
    one = torch.ones_like(rho)
    eq = _equilibrium(rho, [(uw[a] - 0.5 * g[a]) * one for a in range(3)])
    n = torch.stack([(t[_OPP[i]] - eq[_OPP[i]]) if _C[i][1] == sign else t[i] - eq[i] for i in range(19)])
    P = [[sum(c[a] * c[b] * n[i] for i, c in enumerate(_C) if c[a] * c[b]) for b in range(3)] for a in range(3)]
    for i, c in enumerate(_C):
        q = sum((c[a] * c[b] - (a == b) / 3) * P[a][b] for a in range(3) for b in range(3))
        t[i] = eq[i] + 4.5 * _W[i] * q


def _in_slabs(f, fn, cells=1 << 24):
    """f = fn(f slab) in place, in slabs along z."""
    k = max(1, cells * f.shape[2] // f[0].numel())
    for z in range(0, f.shape[2], k):
        f[:, :, z:z + k] = fn(f[:, :, z:z + k].contiguous(), z, k)


def _fluid_exact(omega, par, fields, steps, residual_at=0):
    """Single phase and Shan-Chen; fields [batch, nz, ny, nx] and [batch, 3, nz, ny, nx]; g, G and omega may be per domain."""
    per, lid = par.get("periodic", (True,) * 3), par.get("lid_u")
    g, G = par.get("g", (0.0, 0.0, 0.0)), par.get("G")
    reg = par.get("wall_model") == "regularized"
    f = torch.empty((19,) + tuple(fields["rho"].shape), dtype=F64, device=DEV)
    _in_slabs(f, lambda s, z, k: _equilibrium(fields["rho"][:, z:z + k], [fields["u"][:, a, z:z + k] for a in range(3)]))
    fields = None

    def pulled():
        p = _stream(f, per, lid)
        if reg:
            _regularize(p, 0, 1, (0.0, 0.0, 0.0), g)
            _regularize(p, -1, -1, lid or (0.0, 0.0, 0.0), g)
        force = None
        if G is not None:
            psi = 1 - torch.exp(-p.sum(dim=0))
            force = [-G * psi * s for s in _gradient_sum(psi, per)]
        return p, force

    def forced(m, force, z, k):
        return [m[0] * g[a] + (0 if force is None else force[a][:, z:z + k]) for a in range(3)]

    def read():
        p, force = pulled()
        rho, u = torch.empty_like(p[0]), torch.empty((3,) + tuple(p[0].shape), dtype=F64, device=DEV)

        def take(s, z, k):
            m = _raw(s)
            F = forced(m, force, z, k)
            rho[:, z:z + k] = m[0]
            for a in range(3):
                u[a][:, z:z + k] = (m[1 + a] + 0.5 * F[a]) / m[0]
            return s
        _in_slabs(p, take)
        return rho, u.transpose(0, 1)

    last, res = None, -1.0
    for n in range(steps):
        if residual_at and n % residual_at == 0:
            last, at = read()[1], n
        p, force = pulled()

        def one(s, z, k):
            m = _raw(s)
            return _collide(m, forced(m, force, z, k), omega)
        _in_slabs(p, one)
        f = p
    rho, u = read()
    if residual_at:
        res = float((u - last).norm() / u.norm()) / (steps - at)
    return rho, u, res


def _mhd_exact(omega, par, fields, steps):
    """Fluid populations and the D3Q7 magnetic ones; rho [batch, ...], u and B [batch, 3, ...]; g and b_wall [3] of [batch, 1, 1, 1]."""
    per, g, bw, tau = par["periodic"], par["g"], par["b_wall"], par["tau_m"]
    cm = [(0, 0, 0), (1, 0, 0), (-1, 0, 0), (0, 1, 0), (0, -1, 0), (0, 0, 1), (0, 0, -1)]
    wm, opp = [1 / 4] + [1 / 8] * 6, [0, 2, 1, 4, 3, 6, 5]

    def eq(u, b):
        return [[wm[i] * (b[k] + 4 * sum(c[a] * (u[a] * b[k] - b[a] * u[k]) for a in range(3) if c[a])) for k in range(3)] for i, c in enumerate(cm)]

    u0, b0 = [fields["u"][:, a] for a in range(3)], [fields["B"][:, a] for a in range(3)]
    f, h = _equilibrium(fields["rho"], u0), eq(u0, b0)

    def pulled():
        p, q = _stream(f, per), []
        for i, c in enumerate(cm):
            q.append([])
            for k in range(3):
                t = torch.roll(h[i][k], (c[2], c[1], c[0]), (-3, -2, -1))
                for a in range(3):
                    if c[a] and not per[a]:
                        at = 0 if c[a] > 0 else -1
                        t.select(-1 - a, at).copy_((-h[opp[i]][k] + 2 * wm[i] * bw[k]).select(-1 - a, at))
                q[i].append(t)
        m = _raw(p)
        b = [sum(q[i][k] for i in range(7)) for k in range(3)]
        v = [m[1 + a] / m[0] for a in range(3)]
        N = [[q[2 * a + 1][k] - q[2 * a + 2][k] - (v[a] * b[k] - b[a] * v[k]) for k in range(3)] for a in range(3)]
        j = [-4 / tau * (N[(k + 1) % 3][(k + 2) % 3] - N[(k + 2) % 3][(k + 1) % 3]) for k in range(3)]
        F = [m[0] * g[k] + j[(k + 1) % 3] * b[(k + 2) % 3] - j[(k + 2) % 3] * b[(k + 1) % 3] for k in range(3)]
        u = [(m[1 + a] + 0.5 * F[a]) / m[0] for a in range(3)]
        return m, q, b, F, u

    for _ in range(steps):
        m, q, b, F, u = pulled()
        f, e = _collide(m, F, omega), eq(u, b)
        h = [[q[i][k] + (e[i][k] - q[i][k]) / tau for k in range(3)] for i in range(7)]
    m, q, b, F, u = pulled()
    return m[0], torch.stack(u, 1), torch.stack(b, 1)


def _cgm_exact(omega, par, fields, steps):
    """Two colour distributions: the total f and the red one r; fields [1, nz, ny, nx]."""
    per, g, ref = par.get("periodic", (True,) * 3), par.get("g", (0.0, 0.0, 0.0)), par.get("rho_ref", 0.0)
    ar, ab, A, beta = par["alpha_r"], par["alpha_b"], par["A"], par["beta"]
    rho, red = fields["rho"], fields["rho"] * (1 + fields["phase"]) / 2
    f = _equilibrium(rho, [fields["u"][:, a] for a in range(3)], (red * ar + (rho - red) * ab) / rho)
    r = f * (red / rho)

    def pulled():
        p, q = _stream(f, per), _stream(r, per)
        m, red = _raw(p), q.sum(dim=0)
        alpha = (red * ar + (m[0] - red) * ab) / m[0]
        F = [(m[0] - ref) * g[a] for a in range(3)]
        return m, red, alpha, F, (2 * red - m[0]) / m[0]

    for _ in range(steps):
        m, red, alpha, F, phi = pulled()
        f = _collide(m, F, omega, alpha)
        gr = [3 * s for s in _gradient_sum(phi, per)]
        n2 = gr[0] ** 2 + gr[1] ** 2 + gr[2] ** 2
        nrm = n2.sqrt()
        safe2, safe = torch.where(n2 > 1e-24, n2, 1.0), torch.where(nrm > 1e-12, nrm, 1.0)
        amp = torch.where(n2 > 1e-24, A * nrm, 0.0)
        mix = torch.where(nrm > 1e-12, beta * red * (m[0] - red) / m[0] * (1 - alpha) / safe, 0.0)
        r = torch.empty_like(f)
        for i, c in enumerate(_C[1:], 1):
            cg = sum(c[a] * gr[a] for a in range(3) if c[a])
            axis = i in (1, 2, 3, 10, 11, 12)
            f[i] += amp * (_W[i] * cg * cg / safe2 - (1 / 18 if axis else 1 / 36))
            r[i] = red / m[0] * f[i] + mix * cg * (1 / 12 if axis else 1 / (24 * math.sqrt(2)))
        f[0] = m[0] - f[1:].sum(dim=0)
        r[0] = red - r[1:].sum(dim=0)
    m, red, alpha, F, phi = pulled()
    return m[0], torch.stack([(m[1 + a] + 0.5 * F[a]) / m[0] for a in range(3)], 1), phi


def _network_layers(params):
    ch, out, at = (16, 32, 32, 32, 4), [], 0
    for a, b in zip(ch, ch[1:]):
        out.append((params[at:at + 27 * a * b].view(b, a, 27), params[at + 27 * a * b:at + 27 * a * b + b]))
        at += 27 * a * b + b
    return out


def _network(params, shape, re):
    """Outputs [4, nz, ny, nx] of the warm-start network."""
    nx, ny, nz = shape
    x, y, z = _axes(nx, ny, nz)
    v = [2 * (x + 0.5) / nx - 1, 2 * (y + 0.5) / ny - 1, 2 * (z + 0.5) / nz - 1]
    r, one = (re - 550.0) / 450.0, torch.ones((nz, ny, nx), dtype=F64, device=DEV)
    ch = [r * one] + [one * t for t in v] + [one * (y == ny - 1)]
    for fn in (lambda t: torch.cos(0.5 * math.pi * t), lambda t: torch.sin(math.pi * t), lambda t: torch.cos(math.pi * t)):
        ch += [one * fn(t) for t in v]
    a = torch.stack(ch + [r * r * one, r * 0.5 * (v[1] + 1) * one])
    layers = _network_layers(params)
    for l, (w, b) in enumerate(layers):
        p = torch.nn.functional.pad(a, (1, 1, 1, 1, 1, 1))
        t = b.view(-1, 1).expand(w.shape[0], nx * ny * nz)
        for k in range(27):
            dx, dy, dz = k % 3, (k // 3) % 3, k // 9
            t = t + w[:, :, k] @ p[:, dz:dz + nz, dy:dy + ny, dx:dx + nx].reshape(p.shape[0], -1)
        a = t.view(-1, nz, ny, nx)
        if l < len(layers) - 1:
            a = torch.relu(a)
    return a


def exact(case, seed):
    kind = case["kind"]
    if kind == "network":
        re, w, rho, u = _network_inputs(case, seed)
        p = torch.tensor(w, dtype=F64, device=DEV, requires_grad=True)
        out = _network(p, (case["nx"], case["ny"], case["nz"]), re)
        t = torch.cat([(rho.unsqueeze(0) - 1) * 30, u * 10])
        loss = ((out - t) ** 2).mean()
        loss.backward()
        return {"loss": float(loss.detach()), "gradient": p.grad}
    if kind.startswith("sweep"):
        sizes, omega, par, fields = _sweep(case, seed)
        keys = ("rho", "u", "B") if kind == "sweep_mhd" else ("rho", "u")
        got = [None] * len(sizes)
        for n in sorted(set(sizes)):  # the domains of one size together
            at = [k for k, m in enumerate(sizes) if m == n]
            stacked = {key: torch.stack([fields[k][key] for k in at]) for key in keys}
            mine = dict(par)
            for key in ("g", "b_wall"):
                if key in par:
                    mine[key] = [torch.tensor([par[key][k][a] for k in at], dtype=F64, device=DEV).view(-1, 1, 1, 1) for a in range(3)]
            if "G" in par:
                mine["G"] = torch.tensor([par["G"][k] for k in at], dtype=F64, device=DEV).view(-1, 1, 1, 1)
            v = _mhd_exact(omega, mine, stacked, case["steps"]) if kind == "sweep_mhd" else _fluid_exact(omega, mine, stacked, case["steps"])
            for j, k in enumerate(at):
                got[k] = [t[j].reshape(-1) for t in v[:len(keys)]]
        return {key: torch.cat([d[i] for d in got]) for i, key in enumerate(keys)}
    omega, par, fields = _problem(case, seed)
    shape = (case["nx"], case["ny"], case["nz"])
    if kind == "cavity":
        w = torch.tensor(np.load(WEIGHTS)["weights"], dtype=F64, device=DEV)
        y = _network(w, shape, fields["reynolds"])
        fields = {"rho": 1 + y[0] / 30, "u": y[1:] / 10}
        del y
    fields = {k: v.unsqueeze(0) for k, v in fields.items()}
    if kind in ("droplets", "rt"):
        rho, u, phi = _cgm_exact(omega, par, fields, case["steps"])
        return {"rho": rho.reshape(-1), "u": u.reshape(-1), "phase": phi.reshape(-1)}
    rho, u, res = _fluid_exact(omega, par, fields, case["steps"], 100 if kind == "cavity" else 0)
    out = {"rho": rho.reshape(-1), "u": u.reshape(-1)}
    if kind == "cavity":
        out.update(steps=case["steps"], residual=res)
    return out
