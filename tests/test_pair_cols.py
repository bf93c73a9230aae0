"""The columns that a lane of the two-node stream-collide kernel loads
(lbm_cols.h, compiled for the host): inside the row for every lane of every
block, also the lanes -- and whole warps -- past the row's end, and the
periodic neighbours of its pair for the lanes on the row."""
import os
import shutil
import subprocess

import numpy as np
import pytest

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))
CSRC = os.path.join(ROOT, "paper_1407_4524_gb300", "csrc")

PROGRAM = r"""
#include <cstdio>
#include <cstdlib>
#include "lbm_cols.h"
int main(int argc, char **argv) {
    const int nx = atoi(argv[1]), lanes = atoi(argv[2]);
    for (int t = 0; t < lanes; ++t) {
        const lbm::PairCols c = lbm::pair_cols(2 * t, nx);
        std::printf("%d %d %d\n", c.own, c.left, c.right);
    }
}
"""


@pytest.fixture(scope="module")
def program(tmp_path_factory):
    cxx = shutil.which("g++") or shutil.which("c++")
    if cxx is None:
        pytest.skip("no C++ compiler")
    d = tmp_path_factory.mktemp("cols")
    src, exe = d / "cols.cpp", d / "cols"
    src.write_text(PROGRAM)
    subprocess.run([cxx, "-O1", "-I", CSRC, str(src), "-o", str(exe)], check=True)
    return str(exe)


@pytest.mark.parametrize("nx", [4, 6, 62, 64, 66, 126, 128, 130, 192, 254, 256, 258, 386, 514, 1022])
def test_columns_stay_inside_the_row(program, nx):
    lanes = (nx // 2 + 127) // 128 * 128  # whole blocks of 128 threads
    out = subprocess.run([program, str(nx), str(lanes)], capture_output=True, text=True, check=True).stdout
    own, left, right = np.array([line.split() for line in out.splitlines()], dtype=int).T
    for c in (own, left, right):
        assert c.min() >= 0 and c.max() <= nx - 2 and not (c % 2).any()
    x0 = 2 * np.arange(nx // 2)
    assert np.array_equal(own[:nx // 2], x0)
    assert np.array_equal(left[:nx // 2], (x0 - 2) % nx)
    assert np.array_equal(right[:nx // 2], (x0 + 2) % nx)
