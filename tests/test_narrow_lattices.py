"""Lattices of a few columns: the launches of several steps are left to those
that gain from them."""
import ctypes
import os
import subprocess
import time

import numpy as np
import pytest

from paper_1204_4098_gb300 import lbm

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))
SOURCE = r"""
#include "lbm_geometry.h"
extern "C" int applies(int nx, int ny) {
  return lbm::two_step_applies(LBM_VARIANT_AUTO, LBM_FP32, nx, ny, 0, 4.0);
}
"""


def test_one_and_three_columns_take_one_step_per_launch(tmp_path):
    src, so = tmp_path / "h.cpp", tmp_path / "h.so"
    src.write_text(SOURCE)
    subprocess.run(["g++", "-std=c++17", "-shared", "-fPIC", "-I", os.path.join(ROOT, "include"),
                    "-I", os.path.join(ROOT, "paper_1204_4098_gb300", "csrc"), str(src), "-o",
                    str(so)], check=True)
    H = ctypes.CDLL(str(so))
    for ny in (31001, 200000):
        assert [nx for nx in range(1, 12) if H.applies(nx, ny)] == \
            [nx for nx in range(1, 12) if nx not in (1, 3) and nx * ny >= 176 * 176]


def seconds(call):
    call()
    out = []
    for _ in range(5):
        t = time.perf_counter()
        call()
        out.append(time.perf_counter() - t)
    return min(out)


@pytest.mark.gpu
@pytest.mark.parametrize("nx,ny", [(1, 31001), (1, 200000), (2, 15500), (3, 20000), (5, 20000),
                                   (1, 5000), (3, 3000)])
def test_the_automatic_kernel_is_no_slower(nx, ny):
    rho = np.full((ny, nx), 0.12) * np.random.default_rng(1).uniform(0.999, 1.001, (ny, nx))
    t = []
    # (the one-step kernel that the automatic choice has for the width)
    for variant in (lbm.VARIANT_AUTO, lbm.VARIANT_REGISTER if nx % 2 else lbm.VARIANT_PAIR):
        with lbm.Lattice(nx, ny, 0.9) as lat:
            lat.set_variant(variant)
            lat.init_density(rho)
            t.append(seconds(lambda: lat.step(400, lbm.IMPROVED, 0.8, 0.1)))
    assert t[0] < 1.1 * t[1]
