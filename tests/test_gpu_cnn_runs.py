"""The network kernels at the edges of their tiles and y-runs (one voxel, one row, exactly one tile per row, one voxel
more, runs cut by the CTAs' tile ranges), against the FP64 network; bounds as in tests/test_gpu_cnn.py (BF16 operands:
2^-9 per rounding, three hidden layers)."""
import numpy as np
import pytest

from oracle import cnn_oracle as C

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("shape", [(1, 1, 1), (1, 7, 3), (2, 1, 5), (127, 3, 2), (128, 3, 2), (129, 2, 2), (16, 41, 9), (40, 1, 31)])
def test_gradient_and_forward_at_the_edges(shape):
    from paper_2010_01628_gb300 import binding as L
    nx, ny, nz = shape
    n = nx * ny * nz
    p = (0.12 * np.random.default_rng(9).standard_normal(C.param_count())).astype(np.float32)
    rng = np.random.default_rng(10)
    rho = 1.0 + 0.01 * rng.standard_normal((nz, ny, nx))
    u = 0.05 * rng.standard_normal((3, nz, ny, nx))
    net = L.lbm_cnn_create(shape, p)
    try:
        L.lbm_cnn_set_input(net, 300.0)
        y = L.lbm_cnn_forward(net, n)
        loss, g = L.lbm_cnn_gradient(net, rho, u)
        loss2, g2 = L.lbm_cnn_gradient(net, rho, u)
    finally:
        L.lbm_cnn_destroy(net)
    X = C.features(shape, 300.0)
    ref = C.forward(p.astype(np.float64), X)[-1].reshape(-1, 4)
    assert np.linalg.norm(y - ref) <= 3e-2 * np.linalg.norm(ref)
    lref, gref = C.loss_and_grad(p.astype(np.float64), X, rho, u)
    assert abs(loss - lref) <= 2e-2 * lref
    assert np.linalg.norm(g - gref) <= 5e-2 * np.linalg.norm(gref)
    assert loss == loss2 and np.array_equal(g, g2)  # fixed order of all sums
