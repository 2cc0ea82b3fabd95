"""Long calls of one thread (the first of a context makes its graphs) beside a thread that synchronises the device, which
CUDA refuses while any stream of the context is captured: neither sees an error, and the states are those of single steps."""
import threading
import time

import numpy as np
import pytest

from paper_2010_01628_gb300 import inputs

pytestmark = pytest.mark.gpu
KINDS = {"fluid": {}, "sc": dict(physics="sc", G=-4.5), "batch": dict(physics="sc", G=-4.5)}


@pytest.mark.parametrize("kind", sorted(KINDS))
def test_graphs_are_made_beside_device_synchronisations(kind):
    import torch

    from paper_2010_01628_gb300 import binding as L
    shape, kw = (16, 9, 8), KINDS[kind]
    rho, u = inputs.random_fields(shape, 3, u_amp=0.02)

    def run(steps):
        if kind == "batch":
            ctx = L.lbm_batch_create([shape] * 3, 1.6, **kw)
            view = L.lbm_batch_domain(ctx, 1)
        else:
            ctx = view = L.lbm_create(shape, 1.6, **kw)
        try:
            L.lbm_init_fields(view, rho, u)
            for n in steps:
                L.lbm_step(ctx, n)
            L.lbm_sync(ctx)
            return L.lbm_get_populations(view)
        finally:
            L.lbm_destroy(ctx)

    ref = run([1] * 76)
    stop, errors, count = threading.Event(), [], [0]

    def synchronise():
        try:
            while not stop.is_set():
                torch.cuda.synchronize()
                count[0] += 1
        except Exception as e:  # shown by the test's thread
            errors.append(e)

    t = threading.Thread(target=synchronise)
    t.start()
    try:
        end, runs = time.monotonic() + 1.5, 0
        while time.monotonic() < end and not errors:
            assert np.array_equal(ref, run([44, 32]))
            runs += 1
    finally:
        stop.set()
        t.join()
    assert not errors, (errors, runs, count)
    assert runs > 10 and count[0] > 100
