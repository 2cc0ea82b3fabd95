"""Which rows are numbered through: the rule of lbm_internal.h on the CPU, at widths on both sides of each kernel's line
(measured times of the two forms beside the rule)."""
import subprocess

import pytest

MAIN = r"""
#include "lbm_internal.h"
#include <cstdio>
#include <cstdlib>
int main(int argc, char** argv) {
    for (int i = 1; i + 2 < argc; i += 3) {
        lbm::Box b{atoi(argv[i]), 8, 4, 7u, 0};
        b.n = (size_t)b.nx * 32;
        const int bx = atoi(argv[i + 1]);
        const bool flat = lbm::step_flat(b, bx, atoi(argv[i + 2]));
        const dim3 g = lbm::step_grid(b, bx, b.ny, flat);
        // every node of the plane has a thread, and no CTA is without one
        const long t = (long)g.x * bx;
        if (flat ? (g.y != 1 || t < (long)b.nx * b.ny || t - bx >= (long)b.nx * b.ny)
                 : (g.y != (unsigned)b.ny || t < b.nx || t - bx >= b.nx)) return 1;
        printf("%d", (int)flat);
    }
    printf("\n");
    return 0;
}
"""


@pytest.fixture(scope="module")
def flat(tmp_path_factory):
    from paper_2010_01628_gb300 import build
    d = tmp_path_factory.mktemp("flat")
    (d / "m.cu").write_text(MAIN)
    r = subprocess.run([build.nvcc(), *build.ARCH, "-std=c++17", "-I", build.CSRC, str(d / "m.cu"), "-o", str(d / "m")],
                       capture_output=True, text=True)
    assert r.returncode == 0, r.stderr

    def rule(worth, *rows):
        args = [str(v) for nx, bx in rows for v in (nx, bx, worth)]
        p = subprocess.run([str(d / "m"), *args], capture_output=True, text=True, timeout=60)
        assert p.returncode == 0, (args, p.stdout)
        return p.stdout.strip()

    return rule


def test_full_rows_are_kept(flat):
    for worth in (0, 7, 15, 20):
        assert flat(worth, (32, 32), (64, 32), (64, 64), (128, 128), (256, 128), (256, 256), (1024, 256)) == "0" * 7


def test_kernels_that_gain_at_every_width(flat):
    assert flat(0, (1, 32), (31, 32), (33, 32), (100, 64), (127, 64), (160, 128), (250, 128), (252, 128), (500, 256)) == "1" * 9


def test_colour_gradient_y_walls_and_channels(flat):  # 20 %
    assert flat(20, (1, 32), (33, 32), (40, 32), (48, 32), (72, 64), (80, 64), (96, 64), (100, 64)) == "1" * 8
    assert flat(20, (120, 64), (127, 64), (136, 128), (160, 128), (190, 128), (200, 128), (250, 128), (252, 128), (300, 256),
                (400, 256), (500, 256), (2000, 256)) == "0" * 12


def test_shan_chen_periodic(flat):  # 7 %
    assert flat(7, (40, 32), (72, 64), (100, 64), (112, 64), (144, 128), (200, 128)) == "1" * 6
    assert flat(7, (120, 64), (127, 64), (160, 128), (190, 128), (240, 128), (250, 128), (384, 256)) == "0" * 7


def test_walls_of_colour_gradient_and_d3q27(flat):  # 15 %
    assert flat(15, (33, 32), (72, 64), (100, 64), (108, 64), (136, 128)) == "1" * 5
    assert flat(15, (112, 64), (120, 64), (160, 128), (240, 128), (252, 128), (400, 256)) == "0" * 6
