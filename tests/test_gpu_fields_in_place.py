"""Device field arrays are read and written in place: the same state and the same values as through host arrays."""
import numpy as np
import pytest

from paper_2010_01628_gb300 import inputs

pytestmark = pytest.mark.gpu
KINDS = {
    "fluid": (dict(precision="fp32"), ("rho", "u")),
    "channel_fp64": (dict(precision="fp64", periodic=(True, False, True), wall_model="regularized"), ("rho", "u")),
    "bf16": (dict(precision="bf16"), ("rho", "u")),
    "mhd": (dict(physics="mhd", tau_m=0.9, periodic=(True, False, True), b_wall=(0, 0.01, 0)), ("rho", "u", "B")),
    "cgm": (dict(physics="cgm", alpha_r=7 / 9, A=1e-3), ("rho", "u", "phase")),
    "sc": (dict(physics="sc", G=-5.0), ("rho", "u", "phase")),
    "q27": (dict(lattice="d3q27"), ("rho", "u")),
}


def _fields(shape, keys):
    rho, u = inputs.random_fields(shape, 3)
    f = {"rho": rho, "u": u, "phase": np.random.default_rng(1).uniform(-1, 1, rho.shape),
         "B": 0.01 * np.random.default_rng(2).standard_normal(u.shape)}
    return {k: f[k] for k in keys}


@pytest.mark.parametrize("kind", sorted(KINDS))
@pytest.mark.parametrize("shape", [(37, 5, 3), (64, 8, 8), (1, 4, 2)])
def test_device_arrays_equal_host_arrays(kind, shape):
    import torch

    from paper_2010_01628_gb300 import binding as L
    kw, keys = KINDS[kind]
    f = _fields(shape, keys)
    given = {k: v for k, v in f.items() if not (k == "phase" and kind == "sc")}
    out, states = [], []
    for device in (False, True):
        ctx = L.lbm_create(shape, 1.6, **kw)
        try:
            # one value into a larger buffer: in place needs no more than 8-byte alignment
            arg = {k: (torch.cat([torch.zeros(1, dtype=torch.float64), torch.from_numpy(v).reshape(-1)]).cuda()[1:]
                       .reshape(v.shape) if device else v) for k, v in given.items()}
            L.lbm_init_fields(ctx, arg["rho"], arg.get("u"), phase=arg.get("phase"), B=arg.get("B"))
            states.append(L.lbm_get_populations(ctx))
            L.lbm_step(ctx, 2)
            dst = {k: (torch.full(v.shape, 7.0, dtype=torch.float64, device="cuda") if device else np.empty(v.shape))
                   for k, v in f.items()}
            got = L.lbm_fields(ctx, shape, want=(), **dst)
            out.append({k: v.cpu().numpy() if device else v for k, v in got.items()})
        finally:
            L.lbm_destroy(ctx)
    assert np.array_equal(states[0], states[1])
    for k in keys:
        assert np.array_equal(out[0][k], out[1][k]), k


def test_absent_velocity_and_unwanted_outputs():
    import torch

    from paper_2010_01628_gb300 import binding as L
    shape = (20, 6, 5)
    f = _fields(shape, ("rho",))
    rho = torch.from_numpy(f["rho"]).cuda()
    got = []
    for r, u in ((rho, None), (f["rho"], np.zeros((3, 5, 6, 20)))):
        ctx = L.lbm_create(shape, 1.6, precision="fp64")
        try:
            L.lbm_init_fields(ctx, r, u)
            o = torch.empty((5, 6, 20), dtype=torch.float64, device="cuda")
            L.lbm_fields(ctx, shape, rho=o, want=())
            got.append((L.lbm_get_populations(ctx), o.cpu().numpy()))
        finally:
            L.lbm_destroy(ctx)
    assert np.array_equal(got[0][0], got[1][0]) and np.array_equal(got[0][1], got[1][1])
