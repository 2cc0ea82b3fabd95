"""Multi-step calls replay captured graphs of 16 steps: the state must be bitwise that of single-step calls."""
import numpy as np
import pytest

from paper_2010_01628_gb300 import inputs

pytestmark = pytest.mark.gpu
SHAPE = (37, 21, 14)
KINDS = {
    "fluid_fp64": dict(precision="fp64"),
    "channel": dict(periodic=(True, False, True), wall_model="regularized", g=(1e-5, 0, 0)),
    "cavity_fp16": dict(precision="fp16", periodic=(False,) * 3, lid_u=(0.05, 0, 0)),
    "mhd": dict(physics="mhd", tau_m=0.9, periodic=(True, False, True), b_wall=(0, 0.01, 0)),
    "cgm": dict(physics="cgm", alpha_r=7 / 9, A=1e-3),
    "sc": dict(physics="sc", G=-5.0),
    "q27": dict(lattice="d3q27"),
}


def _make(L, kw, **more):
    rho, u = inputs.random_fields(SHAPE, 3)
    ctx = L.lbm_create(SHAPE, 1.6, **kw, **more)
    extra = {}
    if kw.get("physics") == "cgm":
        extra["phase"] = np.random.default_rng(1).uniform(-1, 1, rho.shape)
    if kw.get("physics") == "mhd":
        extra["B"] = 0.01 * np.random.default_rng(2).standard_normal(u.shape)
    L.lbm_init_fields(ctx, rho, u, **extra)
    return ctx


def _state(L, ctx):
    try:
        L.lbm_sync(ctx)
        return L.lbm_get_populations(ctx)
    finally:
        L.lbm_destroy(ctx)


@pytest.mark.parametrize("kind", sorted(KINDS))
def test_graph_replay_equals_single_steps(kind):
    from paper_2010_01628_gb300 import binding as L
    calls = (15, 16, 1, 17, 49)  # below, at and above one graph, from both buffers, with remainders
    a = _make(L, KINDS[kind])
    for n in calls:
        L.lbm_step(a, n)
    b = _make(L, KINDS[kind])
    for _ in range(sum(calls)):
        L.lbm_step(b, 1)
    assert np.array_equal(_state(L, a), _state(L, b))


def test_graphs_follow_the_launch_shape():
    from paper_2010_01628_gb300 import binding as L
    a, b = _make(L, {"precision": "fp32"}), _make(L, {"precision": "fp32"})
    for threads in (64, 32, 128):
        L.lbm_set_launch_shape(a, 0, threads)
        L.lbm_step(a, 33)
        L.lbm_step(b, 33)
    assert L.lbm_get_launch_shape(a)["threads"] == 128
    assert np.array_equal(_state(L, a), _state(L, b))


def test_steps_inside_a_callers_capture():
    import torch

    from paper_2010_01628_gb300 import binding as L
    s = torch.cuda.Stream()
    with torch.cuda.stream(s):
        a = _make(L, {"precision": "fp32"}, stream=s.cuda_stream)
        g = torch.cuda.CUDAGraph()
        with torch.cuda.graph(g, stream=s):
            L.lbm_step(a, 34)
        g.replay()  # the capture recorded the steps and ran none
        g.replay()
        s.synchronize()
    b = _make(L, {"precision": "fp32"})
    L.lbm_step(b, 68)
    assert np.array_equal(_state(L, a), _state(L, b))
