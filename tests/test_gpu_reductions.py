"""lbm_reduce's sums against FP64 sums of the exported fields, at node counts that leave a partial block, a partial
warp, fewer nodes than one block, and several strides of the whole grid."""
import numpy as np
import pytest

from paper_2010_01628_gb300 import inputs

pytestmark = pytest.mark.gpu
EPS = {"fp64": 2.0 ** -52, "fp32": 2.0 ** -23}
KINDS = {
    "periodic": dict(),
    "walls": dict(periodic=(False,) * 3, lid_u=(0.05, 0, 0)),
    "channel": dict(periodic=(True, False, True), wall_model="regularized", g=(1e-5, 0, 0)),
    "mhd": dict(physics="mhd", tau_m=0.9),
    "cgm": dict(physics="cgm", alpha_r=7 / 9, A=1e-3, periodic=(True, False, True)),
    "sc": dict(physics="sc", G=-5.0),
    "q27": dict(lattice="d3q27"),
}


@pytest.mark.parametrize("kind", sorted(KINDS))
@pytest.mark.parametrize("shape", [(3, 5, 7), (33, 4, 3), (256, 4, 5), (97, 83, 81)])
@pytest.mark.parametrize("precision", ["fp64", "fp32"])
def test_sums_and_residual(kind, shape, precision):
    from paper_2010_01628_gb300 import binding as L
    kw, eps = KINDS[kind], EPS[precision]
    rho, u = inputs.random_fields(shape, 7)
    ctx = L.lbm_create(shape, 1.6, precision=precision, **kw)
    extra = {}
    if kw.get("physics") == "cgm":
        extra["phase"] = np.random.default_rng(1).uniform(-1, 1, rho.shape)
    if kw.get("physics") == "mhd":
        extra["B"] = 0.01 * np.random.default_rng(2).standard_normal(u.shape)
    try:
        L.lbm_init_fields(ctx, rho, u, **extra)
        prev = None
        for _ in range(3):
            L.lbm_step(ctx, 1)
            f = L.lbm_fields(ctx, shape)
            mass, mom, res = L.lbm_reduce(ctx)
            r, v = f["rho"], f["u"]
            # a node's rho and u are sums of up to 27 values of size <= rho: 32 eps rho; the FP64 sums add n 2^-53
            unit = (32 * eps + r.size * 2.0 ** -53) * r.sum()
            assert abs(mass - r.sum()) <= unit
            assert np.abs(np.array(mom) - (r * v).sum(axis=(1, 2, 3))).max() <= 2 * unit
            if prev is None:
                assert res == -1.0
            else:
                norm = np.linalg.norm(v)
                # |d(du)| <= 64 eps per component, so the quotient moves by 64 eps sqrt(3 n) / |u| and by its own rounding
                bound = 64 * eps * np.sqrt(v.size) / norm * 2 + 1e-12
                want = np.linalg.norm(v - prev) / norm
                assert abs(res - want) <= bound * max(1.0, want)
            prev = v
    finally:
        L.lbm_destroy(ctx)
