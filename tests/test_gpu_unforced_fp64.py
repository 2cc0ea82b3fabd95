"""The double-precision step without a body force (its own collision) against the general collision, which the batched
step runs: same values to the parity bound of that precision, and the same handling of zeros, subnormals, huge values,
infinities and NaN, where its power-of-two scalings cannot be exponent arithmetic."""
import numpy as np
import pytest

from paper_2010_01628_gb300 import inputs

pytestmark = pytest.mark.gpu
CASES = [dict(), dict(periodic=(False,) * 3, lid_u=(0.05, 0.0, 0.0)), dict(periodic=(True, False, True))]


def _pair(L, shape, omega, kw):
    a = L.lbm_create(shape, omega, precision="fp64", **kw)
    b = L.lbm_batch_create([shape], omega, precision="fp64", **kw)
    return a, b, L.lbm_batch_domain(b, 0)


@pytest.mark.parametrize("kw", CASES)
@pytest.mark.parametrize("shape", [(33, 9, 7), (32, 8, 8), (1, 3, 2), (20, 1, 1)])
@pytest.mark.parametrize("omega", [0.6, 1.0, 1.9])
def test_unforced_equals_general(kw, shape, omega):
    from paper_2010_01628_gb300 import binding as L
    rho, u = inputs.random_fields(shape, 4)
    a, b, v = _pair(L, shape, omega, kw)
    try:
        for c in (a, v):
            L.lbm_init_fields(c, rho, u)
        L.lbm_step(a, 9)
        L.lbm_batch_step(b, 9)
        x, y = (L.lbm_get_populations(c).view(np.float64) for c in (a, v))
    finally:
        L.lbm_destroy(a)
        L.lbm_destroy(b)
    assert np.linalg.norm(x - y) <= 1e-12 * np.linalg.norm(y)


@pytest.mark.parametrize("special", ["zero", "subnormal", "tiny", "huge", "inf", "nan"])
def test_special_values(special):
    from paper_2010_01628_gb300 import binding as L
    shape, n = (16, 4, 3), 192
    rng = np.random.default_rng(3)
    f = 1e-3 * rng.standard_normal((19, n))
    some = rng.random((19, n)) < 0.3
    if special == "zero":
        f[:] = 0.0
    elif special in ("inf", "nan"):
        f[7, 100] = np.inf if special == "inf" else np.nan
    else:
        f[:] = {"subnormal": 4e-320, "tiny": 3e-308, "huge": 1e300}[special] * rng.uniform(-1, 1, (19, n))
        if special != "huge":
            f[some] = 0.0
    a, b, v = _pair(L, shape, 1.7, {})
    try:
        for c in (a, v):
            L.lbm_set_populations(c, f)
        L.lbm_step(a, 1)
        L.lbm_batch_step(b, 1)
        x, y = (L.lbm_get_populations(c).view(np.float64) for c in (a, v))
    finally:
        L.lbm_destroy(a)
        L.lbm_destroy(b)
    if special == "huge":  # rho u u overflows in either: nothing finite is expected, nothing hangs or faults
        assert x.shape == y.shape
        return
    assert np.array_equal(np.isfinite(x), np.isfinite(y))
    ok = np.isfinite(y)
    scale = np.abs(f[np.isfinite(f)]).max()
    # 1e-12 of the state, and for subnormal states a few units of the smallest subnormal
    assert np.abs(x[ok] - y[ok]).max() <= 1e-12 * scale + 40 * 5e-324
