"""Channel steps, interior and wall rows in one launch, against the FP64 oracle where the wall rows' CTAs are partial,
hold both walls or part of one, and where one interior row is left."""
import pytest

from helpers import gpu_run, oracle_run, rel_l2
from paper_2010_01628_gb300 import inputs

pytestmark = pytest.mark.gpu
TOL = {"fp64": 1e-12, "fp32": 1e-5, "fp16": 1e-3, "bf16": 4e-3}  # the parity bounds of the other channel tests


@pytest.mark.parametrize("walls", ["bounce_back", "regularized"])
@pytest.mark.parametrize("shape", [(5, 3, 4), (128, 4, 2), (129, 3, 2), (300, 5, 3)])
@pytest.mark.parametrize("precision", sorted(TOL))
def test_channel_rows(walls, shape, precision):
    rho, u = inputs.random_fields(shape, seed=71, u_amp=0.03)
    kw = dict(periodic=(True, False, True), wall_model=walls, lid_u=(0.04, 0.0, -0.01), g=(2e-5, 0.0, 5e-6))
    o = oracle_run(shape, 1.5, 20, rho, u, **kw)
    r = gpu_run(shape, 1.5, 20, rho, u, precision=precision, **kw)
    assert max(rel_l2(r[k], o[k]) for k in ("rho", "u")) <= TOL[precision]
