"""One step with a plane's nodes numbered through against one with a CTA per row segment, node by node: the two
compilations of the node code round differently, by no more than the arithmetic's last bits or one unit of the storage."""
import numpy as np
import pytest

pytestmark = pytest.mark.gpu
Y, W = dict(periodic=(True, False, True)), dict(periodic=(False,) * 3)
CGM = dict(physics="cgm", alpha_r=7 / 9, A=1e-3)
KINDS = {
    "periodic": {}, "walls": dict(W, lid_u=(0.05, 0, 0)), "channel": dict(Y, g=(1e-5, 0, 0)),
    "channel_regularized": dict(Y, wall_model="regularized"), "raw_walls": dict(W, collision="rm"),
    "mhd": dict(physics="mhd", tau_m=0.9), "mhd_walls": dict(Y, physics="mhd", tau_m=0.9, b_wall=(0, 0.01, 0)),
    "cgm": CGM, "cgm_y": dict(CGM, **Y), "cgm_walls": dict(CGM, **W),
    "sc": dict(physics="sc", G=-5.0), "sc_walls": dict(Y, physics="sc", G=-5.0),
    "q27": dict(lattice="d3q27"), "q27_walls": dict(W, lattice="d3q27"),
}


def _step(shape, kw, precision, variant, threads):
    from paper_2010_01628_gb300 import binding as L
    rng = np.random.default_rng(7)
    ctx = L.lbm_create(shape, 1.6, precision=precision, **kw)
    try:
        L.lbm_set_launch_shape(ctx, variant, threads)
        n = shape[0] * shape[1] * shape[2]
        rho = 1.0 + 0.1 * rng.uniform(-1, 1, shape[::-1])
        u = 0.05 * rng.uniform(-1, 1, (3,) + shape[::-1])
        more = {}
        if kw.get("physics") == "cgm":
            more["phase"] = rng.uniform(-0.9, 0.9, rho.shape)
        if kw.get("physics") == "mhd":
            more["B"] = 0.05 * rng.uniform(-1, 1, u.shape)
        L.lbm_init_fields(ctx, rho, u, **more)
        L.lbm_step(ctx, 1)
        raw = L.lbm_get_populations(ctx)
    finally:
        L.lbm_destroy(ctx)
    if precision == "bf16":
        return (raw.view(np.uint16).astype(np.uint32) << 16).view(np.float32).astype(np.float64).reshape(-1, n)
    return raw.view({"fp64": np.float64, "fp32": np.float32, "fp16": np.float16}[precision]).astype(np.float64).reshape(-1, n)


# (nx, threads of the row form, threads of the numbered form): rows that fill CTAs of 32 threads and not the larger ones
SHAPES = [((96, 7, 5), 32, 128), ((160, 4, 3), 32, 64), ((32, 9, 3), 32, 256), ((96, 3, 4), 32, 256)]


@pytest.mark.parametrize("kind", sorted(KINDS))
@pytest.mark.parametrize("precision", ["fp64", "fp32"])
def test_numbered_planes_equal_rows(kind, precision):
    eps = 2.0 ** (-52 if precision == "fp64" else -23)
    for shape, rows, flat in SHAPES:
        a, b = (_step(shape, KINDS[kind], precision, 0, t) for t in (rows, flat))
        # about 300 operations on values of the state's size, a rounding each, adding like a random walk and doubled
        assert np.abs(a - b).max() <= 40 * eps * np.abs(a).max(), (shape, flat)


@pytest.mark.parametrize("kind", ["periodic", "walls", "channel", "channel_regularized"])
@pytest.mark.parametrize("precision", ["fp16", "bf16"])
@pytest.mark.parametrize("variant", [0, 4])
def test_numbered_planes_equal_rows_16bit(kind, precision, variant):
    if variant == 4 and kind == "channel_regularized":
        pytest.skip("the z-pair step has half-way walls only")
    unit = 2.0 ** (-10 if precision == "fp16" else -7)
    for shape, rows, flat in SHAPES:
        a, b = (_step(shape, KINDS[kind], precision, variant, min(t, 128)) for t in (rows, flat))
        # one unit of the stored value; the smallest values move by the collision's own rounding in FP32
        assert (np.abs(a - b) <= unit * np.abs(a) + 40 * 2.0 ** -23 * np.abs(a).max()).all(), (shape, flat)
