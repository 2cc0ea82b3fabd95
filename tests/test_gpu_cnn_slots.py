"""The network's convolutions zero only the row slots that a CTA stages: grids of few tiles per CTA, run after a large one
has left its rows in shared memory, give bitwise what they give at first and match the FP64 network (BF16 operands, four
layers: 3e-2, as in tests/test_gpu_cnn.py)."""
import numpy as np
import pytest

from oracle import cnn_oracle as C

pytestmark = pytest.mark.gpu


# tiles are rows here: below and above one per CTA (152 or 304), runs of one tile, of a few, and cut by the CTAs' ranges
@pytest.mark.parametrize("shape", [(8, 8, 8), (3, 1, 1), (5, 1, 330), (4, 2, 310), (6, 5, 123), (7, 400, 1), (2, 9, 170)])
def test_small_grids_after_a_large_one(shape):
    from paper_2010_01628_gb300 import binding as L
    nx, ny, nz = shape
    n = nx * ny * nz
    p = (0.12 * np.random.default_rng(9).standard_normal(C.param_count())).astype(np.float32)
    net, big = L.lbm_cnn_create(shape, p), L.lbm_cnn_create((128, 32, 32), p)
    try:
        L.lbm_cnn_set_input(net, 300.0)
        L.lbm_cnn_set_input_raw(big, np.full((32 * 32 * 128, C.CH[0]), 50.0, dtype=np.float32))
        first = L.lbm_cnn_forward(net, n)
        for _ in range(3):
            L.lbm_cnn_forward(big, 128 * 32 * 32)
            assert np.array_equal(first, L.lbm_cnn_forward(net, n))
    finally:
        L.lbm_cnn_destroy(net)
        L.lbm_cnn_destroy(big)
    ref = C.forward(p.astype(np.float64), C.features(shape, 300.0))[-1].reshape(-1, 4)
    assert np.linalg.norm(first - ref) <= 3e-2 * np.linalg.norm(ref)
