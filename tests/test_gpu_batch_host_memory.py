"""Batch steps allocate no host memory: with operator new failing, as it may in a long-running program, the step still
runs (an exception would leave through the C entry point and end the process)."""
import os
import shutil
import subprocess
import sys

import pytest

pytestmark = pytest.mark.gpu
ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))
NEW = r"""
#include <cstdlib>
#include <new>
static thread_local bool armed = false;
extern "C" void refuse_new(int on) { armed = on != 0; }
void* operator new(std::size_t n) {
    void* p = armed && n >= 8192 ? nullptr : std::malloc(n ? n : 1);  // a table of 128 domains is 8 KB and more
    if (!p) throw std::bad_alloc();
    return p;
}
void* operator new[](std::size_t n) { return operator new(n); }
void operator delete(void* p) noexcept { std::free(p); }
void operator delete[](void* p) noexcept { std::free(p); }
void operator delete(void* p, std::size_t) noexcept { std::free(p); }
void operator delete[](void* p, std::size_t) noexcept { std::free(p); }
"""
RUN = r"""
import ctypes, sys
import numpy as np
from paper_2010_01628_gb300 import binding as L
refuse = ctypes.CDLL(sys.argv[1]).refuse_new
states = []
for on in (0, 1):
    b = L.lbm_batch_create([(9, 5, 4)] * 130, 1.6, physics=sys.argv[2], precision="fp64", G=-4.5)
    refuse(on)
    L.lbm_batch_step(b, 5)
    refuse(0)
    L.lbm_sync(b)
    states.append(L.lbm_get_populations(b))
    L.lbm_destroy(b)
assert np.array_equal(*states)
print("ran")
"""


@pytest.mark.parametrize("physics", ["fluid", "mhd", "cgm", "sc"])
def test_steps_without_host_memory(physics, tmp_path):
    src, so = tmp_path / "new.cpp", tmp_path / "libnew.so"
    src.write_text(NEW)
    subprocess.run([shutil.which("g++") or "c++", "-shared", "-fPIC", str(src), "-o", str(so)], check=True)
    env = dict(os.environ, LD_PRELOAD=str(so), PYTHONPATH=ROOT)
    p = subprocess.run([sys.executable, "-c", RUN, str(so), physics], env=env, cwd=ROOT, capture_output=True, text=True,
                       timeout=300)
    assert p.returncode == 0 and "ran" in p.stdout, p.stderr[-2000:]
