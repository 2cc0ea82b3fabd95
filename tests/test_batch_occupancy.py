"""Every pass of the batched step leaves room for two CTAs of 256 threads per SM (128 registers a thread): with one, an SM
idles from a CTA's last loads to its successor's first."""
import os
import re
import subprocess


def test_two_ctas_of_each_pass_fit(tmp_path):
    from paper_2010_01628_gb300 import build
    src = os.path.join(build.CSRC, "lbm_batch.cu")
    r = subprocess.run([build.nvcc(), *build.ARCH, "-O3", "-std=c++17", "-Xptxas", "-v", "-c", src, "-o",
                        str(tmp_path / "b.o")], capture_output=True, text=True)
    assert r.returncode == 0, r.stderr
    used = {}
    for m in re.finditer(r"Compiling entry function '(\S*batch_pass_kernel\S*)'.*?Used (\d+) registers", r.stderr, re.S):
        used[m.group(1)] = int(m.group(2))
    assert len(used) == 48  # 4 modules, 2 of them in two passes, 2 precisions, walls or none, both tables
    assert max(used.values()) <= 128, max(used.items(), key=lambda kv: kv[1])
