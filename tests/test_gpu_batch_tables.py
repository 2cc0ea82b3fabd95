"""Batches of more than 128 domains: small ones with their tables in device memory (one launch a pass), large FP32 ones
with a launch per 128 domains, against the same domains in batches whose tables are kernel parameters.  The compilations
of the node code round apart: the parity bounds of the precisions."""
import json

import numpy as np
import pytest

from paper_2010_01628_gb300 import inputs

pytestmark = pytest.mark.gpu
TOL = {"fp64": 1e-12, "fp32": 1e-5}
KINDS = {
    "fluid": dict(lid_u=(0.03, 0, 0), g=(1e-5, 0, 0)),
    "mhd": dict(physics="mhd", b_wall=(0, 0.01, 0)),
    "cgm": dict(physics="cgm", alpha_r=7 / 9, A=1e-3),
    "sc": dict(physics="sc", G=-4.5),
}


def _fields(kw, shape, seed):
    rho, u = inputs.random_fields(shape, seed, u_amp=0.02)
    rng = np.random.default_rng(seed)
    more = {}
    if kw.get("physics") == "cgm":
        more["phase"] = rng.uniform(-0.9, 0.9, rho.shape)
    if kw.get("physics") == "mhd":
        more["B"] = 0.01 * rng.standard_normal(u.shape)
    return rho, u, more


def _run(L, kw, precision, shapes, per, tau, first, tune):
    own = {"tau_m": [0.7 + 0.001 * (first + k) for k in range(len(shapes))]} if kw.get("physics") == "mhd" else {}
    b = L.lbm_batch_create(shapes, [1 / t for t in tau], periodic=per, precision=precision, **kw, **own)
    try:
        for k, s in enumerate(shapes):
            rho, u, more = _fields(kw, s, 100 + first + k)
            L.lbm_init_fields(L.lbm_batch_domain(b, k), rho, u, **more)
        if tune:
            before = L.lbm_get_populations(b)
            L.lbm_autotune(b)
            assert np.array_equal(before, L.lbm_get_populations(b))
        for n in (1, 33, 2):
            L.lbm_batch_step(b, n)
        L.lbm_sync(b)
        info = L.lbm_batch_info(b)
        return [L.lbm_fields(L.lbm_batch_domain(b, k), s) for k, s in enumerate(shapes)], info
    finally:
        L.lbm_destroy(b)


def _compare(L, kind, precision, shapes, walls, tune):
    rng = np.random.default_rng(8)
    nd = len(shapes)
    tau = list(rng.uniform(0.8, 1.2, nd))
    per = [tuple(bool(v) for v in rng.integers(0, 2, 3)) if walls else (True,) * 3 for _ in shapes]
    whole, info = _run(L, KINDS[kind] if walls or kind != "fluid" else {}, precision, shapes, per, tau, 0, tune)
    t = info["threads"]
    assert info["tiles"] == info["grid"] == sum(-(-int(np.prod(s)) // t) for s in shapes)
    half = nd // 2
    for a, b in ((0, half), (half, nd)):
        part, _ = _run(L, KINDS[kind] if walls or kind != "fluid" else {}, precision, shapes[a:b], per[a:b], tau[a:b],
                       a, False)
        for k, (x, y) in enumerate(zip(whole[a:b], part)):
            for f in ("rho", "u"):
                assert np.linalg.norm(x[f] - y[f]) <= TOL[precision] * np.linalg.norm(y["rho"]), (a + k, f)


@pytest.mark.parametrize("kind", sorted(KINDS))
@pytest.mark.parametrize("precision", ["fp64", "fp32"])
@pytest.mark.parametrize("walls", [True, False])
def test_many_small_domains(kind, precision, walls):
    from paper_2010_01628_gb300 import binding as L
    rng = np.random.default_rng(5)
    shapes = [(1, 1, 1), (1, 5, 3), (33, 1, 2), (2, 3, 129), (31, 9, 1), (256, 1, 1), (16, 16, 1), (257, 1, 1)]
    shapes += [tuple(int(v) for v in rng.integers(1, 9, 3)) for _ in range(190)]
    _compare(L, kind, precision, shapes, walls, tune=walls)


@pytest.mark.parametrize("kind", ["fluid", "cgm"])
def test_many_large_domains(kind):
    from paper_2010_01628_gb300 import binding as L
    shapes = [(21, 20, 20), (22, 19, 21)] * 64 + [(20, 21, 21)]  # over 2^19 nodes for each of the two launches
    _compare(L, kind, "fp32", shapes, True, tune=False)


def test_a_callers_graph_outlives_a_change_of_cta_size(tmp_path):
    import torch

    from paper_2010_01628_gb300 import binding as L
    shapes = [(9, 5, 7)] * 130
    s = torch.cuda.Stream()
    states = []
    for change in (False, True):
        b = L.lbm_batch_create(shapes, 1.6, precision="fp64", stream=s.cuda_stream)
        try:
            for d in range(len(shapes)):
                rho, u = inputs.random_fields(shapes[d], d, u_amp=0.02)
                L.lbm_init_fields(L.lbm_batch_domain(b, d), rho, u)
            g = torch.cuda.CUDAGraph()
            with torch.cuda.graph(g, stream=s):
                L.lbm_batch_step(b, 4)
            if change:
                cache = tmp_path / "t.json"
                L.lbm_autotune(b, str(cache))
                (key, entry), = json.loads(cache.read_text()).items()
                other = 128 if L.lbm_batch_info(b)["threads"] == 256 else 256
                cache.write_text(json.dumps({key: dict(entry, threads=other)}))
                L.lbm_autotune(b, str(cache))
                assert L.lbm_batch_info(b)["threads"] == other
            with torch.cuda.stream(s):
                g.replay()
            L.lbm_batch_step(b, 2)
            L.lbm_sync(b)
            states.append([L.lbm_get_populations(L.lbm_batch_domain(b, d)) for d in range(len(shapes))])
            del g
        finally:
            L.lbm_destroy(b)
    for x, y in zip(*states):
        assert np.array_equal(x, y)
