"""Replayed steps against single ones, bitwise, where graphs of 4 steps follow those of 16: every remainder from both
buffers, each launch variant, and batches of every module; a profile of the call shows that graphs did run."""
import numpy as np
import pytest

from paper_2010_01628_gb300 import inputs

pytestmark = pytest.mark.gpu
SHAPE = (64, 10, 9)
# odd counts leave the other buffer current: remainders 4 .. 15 of 16 from each, twice, so that every graph is made
CALLS = [32 + r for r in range(4, 16)] * 2 + [33] + [32 + r for r in range(4, 16)] * 2
VARIANTS = {
    "direct": (dict(precision="fp32"), (0, 64)),
    "staged": (dict(precision="fp32", periodic=(True, False, True), lid_u=(0.05, 0, 0)), (1, 64, 4, 2)),
    "pair": (dict(precision="fp16"), (2, 32)),
    "zpair": (dict(precision="bf16", periodic=(False,) * 3), (4, 64)),
    "fused": (dict(physics="sc", G=-5.0), (3, 256, 4)),
    "channel": (dict(periodic=(True, False, True), wall_model="regularized", g=(1e-5, 0, 0)), (0, 64)),
}
BATCHES = {
    "fluid": dict(lid_u=(0.03, 0, 0)),
    "mhd": dict(physics="mhd", tau_m=0.9, b_wall=(0, 0.01, 0)),
    "cgm": dict(physics="cgm", alpha_r=7 / 9, A=1e-3),
    "sc": dict(physics="sc", G=-4.5),
}


@pytest.fixture(scope="module", autouse=True)
def _profiler():
    """A process's first profile may miss the events of its start."""
    import torch
    torch.ones(8, device="cuda").sum().item()
    _replays(lambda: torch.ones(8, device="cuda").sum().item())


def _replays(run):
    """Number of cudaGraphLaunch calls that `run` makes."""
    import torch
    with torch.profiler.profile(activities=[torch.profiler.ProfilerActivity.CPU,
                                            torch.profiler.ProfilerActivity.CUDA]) as p:
        run()
        torch.cuda.synchronize()
    return sum("GraphLaunch" in e.name for e in p.events())


def _start(L, ctx, shape, kw, seed):
    rho, u = inputs.random_fields(shape, seed, u_amp=0.02)
    more = {}
    if kw.get("physics") == "cgm":
        more["phase"] = np.random.default_rng(1).uniform(-1, 1, rho.shape)
    if kw.get("physics") == "mhd":
        more["B"] = 0.01 * np.random.default_rng(2).standard_normal(u.shape)
    L.lbm_init_fields(ctx, rho, u, **more)


def _states(L, ctx, domains):
    """The populations, of a batch without the padding between its domains."""
    return [L.lbm_get_populations(L.lbm_batch_domain(ctx, d) if domains else ctx) for d in range(domains or 1)]


def _compare(L, make, step, domains=0):
    a, b = make(), make()
    try:
        for k, n in enumerate(CALLS):
            step(a, n)
            for _ in range(n):
                step(b, 1)
            if k % 6 == 0 or k + 1 == len(CALLS):
                for x, y in zip(_states(L, a, domains), _states(L, b, domains)):
                    assert np.array_equal(x, y), (k, n)
        assert _replays(lambda: step(a, 44)) == 5  # 2 x 16 + 3 x 4
        assert _replays(lambda: step(a, 15)) == 3
        assert _replays(lambda: step(a, 3)) == 0
    finally:
        L.lbm_destroy(a)
        L.lbm_destroy(b)


@pytest.mark.parametrize("kind", sorted(VARIANTS))
def test_each_launch_variant(kind):
    from paper_2010_01628_gb300 import binding as L
    kw, shape = VARIANTS[kind]

    def make():
        ctx = L.lbm_create(SHAPE, 1.6, **kw)
        L.lbm_set_launch_shape(ctx, *shape)
        _start(L, ctx, SHAPE, kw, 3)
        return ctx

    _compare(L, make, L.lbm_step)


@pytest.mark.parametrize("kind", sorted(BATCHES))
@pytest.mark.parametrize("precision", ["fp32", "fp64"])
@pytest.mark.parametrize("periodic", [(True,) * 3, (True, False, True)])
def test_batches(kind, precision, periodic):
    from paper_2010_01628_gb300 import binding as L
    kw = dict(BATCHES[kind], precision=precision, periodic=periodic)
    shapes = [(9, 7, 5), (16, 4, 8), (5, 12, 3)]

    def make():
        b = L.lbm_batch_create(shapes, 1.6, **kw)
        for d, s in enumerate(shapes):
            _start(L, L.lbm_batch_domain(b, d), s, kw, 20 + d)
        return b

    _compare(L, make, L.lbm_batch_step, len(shapes))
