"""Step kernels that number a plane's nodes through (rows that do not fill whole CTAs) against those that take one row
per CTA: both run the same node code, so 16 steps agree to the rounding of its two compilations."""
import numpy as np
import pytest

from paper_2010_01628_gb300 import inputs

pytestmark = pytest.mark.gpu
# (precision, state bound): eps of the arithmetic (the 16-bit formats: of the storage) times 16 steps, relative to the state
BOUND = {"fp64": 16 * 2.0 ** -52, "fp32": 16 * 2.0 ** -23, "fp16": 16 * 2.0 ** -10, "bf16": 16 * 2.0 ** -7}
NP = {"fp64": np.float64, "fp32": np.float32, "fp16": np.float16}
KINDS = {
    "periodic": dict(),
    "walls": dict(periodic=(False,) * 3, lid_u=(0.05, 0, 0)),
    "channel": dict(periodic=(True, False, True), wall_model="regularized", g=(1e-5, 0, 0)),
    "raw": dict(collision="rm"),
    "mhd": dict(physics="mhd", tau_m=0.9, periodic=(True, False, True), b_wall=(0, 0.01, 0)),
    "cgm": dict(physics="cgm", alpha_r=7 / 9, A=1e-3),
    "cgm_walls": dict(physics="cgm", alpha_r=7 / 9, A=1e-3, periodic=(True, False, True)),
    "sc": dict(physics="sc", G=-5.0),
    "q27": dict(lattice="d3q27", periodic=(True, True, False)),
}


def _values(L, ctx, precision):
    raw = L.lbm_get_populations(ctx)
    if precision == "bf16":
        return (raw.view(np.uint16).astype(np.uint32) << 16).view(np.float32).astype(np.float64)
    return raw.view(NP[precision]).astype(np.float64)


def _run(shape, kw, precision, variant, threads):
    from paper_2010_01628_gb300 import binding as L
    rho, u = inputs.random_fields(shape, 5)
    ctx = L.lbm_create(shape, 1.6, precision=precision, **kw)
    extra = {}
    if kw.get("physics") == "cgm":
        extra["phase"] = np.random.default_rng(1).uniform(-1, 1, rho.shape)
    if kw.get("physics") == "mhd":
        extra["B"] = 0.01 * np.random.default_rng(2).standard_normal(u.shape)
    try:
        L.lbm_set_launch_shape(ctx, variant, threads)
        L.lbm_init_fields(ctx, rho, u, **extra)
        L.lbm_step(ctx, 16)
        return _values(L, ctx, precision)
    finally:
        L.lbm_destroy(ctx)


# nx = 96 fills CTAs of 32 threads (row form) and not those of 64 or 128 (numbered through); 160 likewise
@pytest.mark.parametrize("kind", sorted(KINDS))
@pytest.mark.parametrize("shape,threads", [((96, 7, 5), 128), ((160, 4, 3), 64), ((96, 3, 4), 256)])
def test_flat_equals_rows(kind, shape, threads):
    for precision in ("fp64", "fp32"):
        a, b = (_run(shape, KINDS[kind], precision, 0, t) for t in (32, threads))
        assert np.linalg.norm(a - b) <= BOUND[precision] * np.linalg.norm(a), precision


@pytest.mark.parametrize("precision", ["fp16", "bf16"])
@pytest.mark.parametrize("variant", [0, 4])
@pytest.mark.parametrize("kind", ["periodic", "walls"])
def test_flat_equals_rows_16bit(kind, variant, precision):
    for shape in ((96, 7, 5), (96, 5, 4)):  # odd and even z: the z-pairs' last thread
        a, b = (_run(shape, KINDS[kind], precision, variant, t) for t in (32, 128))
        assert np.linalg.norm(a - b) <= BOUND[precision] * np.linalg.norm(a)
