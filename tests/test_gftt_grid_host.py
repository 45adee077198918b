"""The selection's cell grid for every minimum distance the detector accepts: a
grid of at least one cell whose cells are at least as wide as the distance (or
as the level), within the kernel's cell count."""

import os
import subprocess

import pytest

CSRC = os.path.join(os.path.dirname(os.path.dirname(os.path.abspath(__file__))), "paper_2607_01757_gb300", "csrc")

SRC = r"""
#include <cstdio>
#include <cstdlib>
#include "vt_gftt_grid.h"
int main(int, char **a) {
    int c, x, y;
    vt::gftt_grid(atoi(a[1]), atoi(a[2]), atoi(a[3]), 16384, c, x, y);
    printf("%d %d %d\n", c, x, y);
}
"""


@pytest.fixture(scope="module")
def grid(tmp_path_factory):
    d = tmp_path_factory.mktemp("grid")
    src, exe = d / "grid.cpp", str(d / "grid")
    src.write_text(SRC)
    subprocess.run(["g++", "-std=c++17", "-I", CSRC, str(src), "-o", exe],
                   check=True)

    def f(w, h, md):
        out = subprocess.run([exe, str(w), str(h), str(md)], check=True, capture_output=True, text=True).stdout
        return tuple(int(v) for v in out.split())

    return f


@pytest.mark.parametrize("min_dist", [1, 10, 46340, 46341, 65534, 65535, 65536, 2**31 - 753, 2**31 - 752, 2**31 - 1])
@pytest.mark.parametrize("size", [(1, 1), (752, 480), (65535, 2), (65535, 32767)])
def test_grid(grid, size, min_dist):
    w, h = size
    cell, cx, cy = grid(w, h, min_dist)
    assert cx >= 1 and cy >= 1 and cx * cy <= 16384
    assert (cx - 1) * cell < w <= cx * cell and (cy - 1) * cell < h <= cy * cell
    assert cell >= min(min_dist, max(w, h))
