"""The double-precision step without a body force beside walls on x or z (channels, with walls on y alone, have a kernel
of their own), and at magnitudes near the largest double, against the general collision, which the batched step runs."""
import numpy as np
import pytest

from paper_2010_01628_gb300 import inputs

pytestmark = pytest.mark.gpu


def _both(L, shape, omega, steps, kw, start):
    a = L.lbm_create(shape, omega, precision="fp64", **kw)
    b = L.lbm_batch_create([shape], omega, precision="fp64", **kw)
    v = L.lbm_batch_domain(b, 0)
    try:
        for c in (a, v):
            start(c)
        L.lbm_step(a, steps)
        L.lbm_batch_step(b, steps)
        return [L.lbm_get_populations(c).view(np.float64) for c in (a, v)]
    finally:
        L.lbm_destroy(a)
        L.lbm_destroy(b)


@pytest.mark.parametrize("kw", [dict(periodic=(False, True, True)), dict(periodic=(True, True, False)),
                                dict(periodic=(True, False, False), lid_u=(0.05, 0.0, 0.0))])
@pytest.mark.parametrize("shape", [(33, 9, 7), (32, 8, 8), (20, 1, 1)])
def test_unforced_equals_general_beside_walls(kw, shape):
    from paper_2010_01628_gb300 import binding as L
    rho, u = inputs.random_fields(shape, 4)
    x, y = _both(L, shape, 1.9, 9, kw, lambda c: L.lbm_init_fields(c, rho, u))
    assert np.linalg.norm(x - y) <= 1e-12 * np.linalg.norm(y)


@pytest.mark.parametrize("size", [1e150, 1e300, 2e305])
def test_large_values(size):
    """Positive populations keep |u| below 1, so one collision stays finite up to the scalings by 2 and 4."""
    from paper_2010_01628_gb300 import binding as L
    shape, n = (16, 4, 3), 192
    f = size * np.random.default_rng(3).uniform(0.0, 1.0, (19, n))
    x, y = _both(L, shape, 1.7, 1, {}, lambda c: L.lbm_set_populations(c, f))
    assert np.isfinite(y).all() and np.isfinite(x).all()
    assert np.abs(x - y).max() <= 1e-12 * size
