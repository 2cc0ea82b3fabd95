"""Batches of more domains than one launch's table holds (128), with degenerate and ragged boxes, against each domain
run alone (FP64; both sides run the same node code, compiled apart: 1e-12 is the parity bound of that precision)."""
import numpy as np
import pytest

from paper_2010_01628_gb300 import inputs

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("physics", ["fluid", "sc"])
def test_more_domains_than_one_table(physics):
    from paper_2010_01628_gb300 import binding as L
    rng = np.random.default_rng(8)
    shapes = [(1, 1, 1), (1, 5, 3), (33, 1, 2), (2, 3, 129), (31, 9, 1)]
    shapes += [tuple(int(v) for v in rng.integers(1, 9, 3)) for _ in range(126)]
    tau = rng.uniform(0.8, 1.2, len(shapes))
    per = [tuple(bool(v) for v in rng.integers(0, 2, 3)) for _ in shapes]
    kw = dict(physics=physics, precision="fp64", G=-4.5 if physics == "sc" else 0.0)
    fields = [inputs.random_fields(s, 100 + k, u_amp=0.02) for k, s in enumerate(shapes)]
    b = L.lbm_batch_create(shapes, list(1 / tau), periodic=per, **kw)
    try:
        for k, f in enumerate(fields):
            L.lbm_init_fields(L.lbm_batch_domain(b, k), *f)
        for n in (3, 17, 2):
            L.lbm_batch_step(b, n)
        got = [L.lbm_fields(L.lbm_batch_domain(b, k), s) for k, s in enumerate(shapes)]
    finally:
        L.lbm_destroy(b)
    for k, s in enumerate(shapes):
        ctx = L.lbm_create(s, 1 / tau[k], periodic=per[k], **kw)
        try:
            L.lbm_init_fields(ctx, *fields[k])
            L.lbm_step(ctx, 22)
            ref = L.lbm_fields(ctx, s)
        finally:
            L.lbm_destroy(ctx)
        for f in ("rho", "u"):
            assert np.linalg.norm(got[k][f] - ref[f]) <= 1e-12 * np.linalg.norm(ref["rho"]), (k, s, f)
