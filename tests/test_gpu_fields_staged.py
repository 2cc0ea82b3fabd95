"""Field arrays that kernels do not use in place (managed memory, arrays off 8-byte alignment, host arrays beside device
arrays) are copied through the staging slabs: the same state and values as through aligned device arrays."""
import ctypes

import numpy as np
import pytest

from paper_2010_01628_gb300 import inputs

pytestmark = pytest.mark.gpu
SHAPE = (37, 5, 6)
N = 37 * 5 * 6


class _Managed:
    """float64 buffers in managed memory, seen by the host as numpy arrays."""

    def __init__(self):
        import torch
        torch.cuda.init()  # loads the runtime library
        self.rt = ctypes.CDLL("libcudart.so." + torch.version.cuda.split(".")[0])
        self.ptrs = []

    def array(self, shape):
        p, n = ctypes.c_void_p(), int(np.prod(shape))
        assert self.rt.cudaMallocManaged(ctypes.byref(p), ctypes.c_size_t(8 * n), 1) == 0
        self.ptrs.append(p)
        return np.frombuffer((ctypes.c_double * n).from_address(p.value), dtype=np.float64).reshape(shape)

    def free(self):
        for p in self.ptrs:
            self.rt.cudaFree(p)


def _off4(shape):
    """Device memory for float64 values that starts 4 bytes off their alignment."""
    import torch
    return torch.zeros(8 * int(np.prod(shape)) + 8, dtype=torch.uint8, device="cuda")[4:-4]


@pytest.mark.parametrize("form", ["managed", "misaligned", "mixed"])
def test_staged_arrays_equal_arrays_in_place(form):
    import torch

    from paper_2010_01628_gb300 import binding as L
    rho, u = inputs.random_fields(SHAPE, 3)
    got = []
    managed = _Managed() if form == "managed" else None
    try:
        for staged in (False, True):
            ins = [torch.from_numpy(rho).cuda(), torch.from_numpy(u).cuda()]
            outs = [torch.zeros_like(t) for t in ins]
            if staged and form == "managed":
                m = [managed.array(t.shape) for t in (*ins, *outs)]
                for a, v in zip(m, (rho, u)):
                    a[...] = v
                ins, outs = m[:2], m[2:]
            elif staged and form == "misaligned":
                raw = [t.reshape(-1).view(torch.uint8) for t in ins]
                ins, outs = [_off4(rho.shape), _off4(u.shape)], [_off4(rho.shape), _off4(u.shape)]
                for t, v in zip(ins, raw):
                    t.copy_(v)
                assert all(t.data_ptr() % 8 == 4 for t in (*ins, *outs))
            elif staged:
                ins[0], outs[1] = rho, np.zeros(u.shape)  # one host and one device array each way
            at = [t.ctypes.data if isinstance(t, np.ndarray) else t.data_ptr() for t in (*ins, *outs)]
            torch.cuda.synchronize()
            ctx = L.lbm_create(SHAPE, 1.6, precision="fp64")
            try:
                L._check(L._lib.lbm_init_fields(ctx, at[0], at[1], None, None), ctx)
                state = L.lbm_get_populations(ctx)
                L.lbm_step(ctx, 2)
                L._check(L._lib.lbm_fields(ctx, at[2], at[3], None, None), ctx)
            finally:
                L.lbm_destroy(ctx)
            vals = [np.array(t) if isinstance(t, np.ndarray) else t.cpu().numpy() for t in outs]
            got.append((state, *[v.reshape(-1).view(np.uint8) for v in vals]))
    finally:
        if managed:
            managed.free()
    for a, b in zip(*got):
        assert np.array_equal(a, b)
