"""Band heights of the batch's two-step items (lbm_batch_host.h) beyond the
lattice's own height, compiled with the host C++ compiler: an item is then the
whole height, up to the largest height that can be asked for."""
import ctypes
import os
import subprocess

import pytest

from paper_1204_4098_gb300 import lbm

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))
SOURCE = r"""
#include "lbm_batch_host.h"
extern "C" int items(int layout, int nx, int ny, int rows, int* out, int cap) {
  std::vector<lbm::TwoItem> v;
  lbm::two_items({lbm::TwoLattice{0, nx, ny, layout}}, rows, v);
  for (int k = 0; k < int(v.size()) && k < cap; ++k) {
    out[3 * k] = v[k].strip; out[3 * k + 1] = v[k].y0; out[3 * k + 2] = v[k].y1;
  }
  return int(v.size());
}
"""
HEIGHTS = [300, 301, 2 ** 30 - 1, 2 ** 30, 2 ** 30 + 5, 2 ** 31 - 301, 2 ** 31 - 300, 2 ** 31 - 1]


@pytest.fixture(scope="module")
def H(tmp_path_factory):
    d = tmp_path_factory.mktemp("items")
    src, so = d / "h.cpp", d / "h.so"
    src.write_text(SOURCE)
    subprocess.run(["g++", "-std=c++17", "-O1", "-shared", "-fPIC", "-I",
                    os.path.join(ROOT, "include"), "-I",
                    os.path.join(ROOT, "paper_1204_4098_gb300", "csrc"), str(src), "-o", str(so)],
                   check=True)
    return ctypes.CDLL(str(so))


@pytest.mark.parametrize("rows", HEIGHTS)
@pytest.mark.parametrize("layout,nx,strips", [(0, 200, 4), (1, 201, 4), (2, 64, 1), (2, 32, 1)])
def test_an_item_is_at_most_the_height(H, layout, nx, strips, rows):
    out = (ctypes.c_int * 24)()
    n = H.items(layout, nx, 300, rows, out, 8)
    got = [tuple(out[3 * k:3 * k + 3]) for k in range(min(n, 8))]
    assert sorted(got) == [(s, 0, 300) for s in range(strips)]


@pytest.mark.gpu
@pytest.mark.parametrize("rows", [2 ** 30, 2 ** 31 - 1])
def test_largest_heights_run(rows):
    inst = [dict(nx=nx, ny=30, T_over_Tc=0.9, tau=0.8, sigma=0.0, scheme=lbm.SC)
            for nx in (32, 64, 66, 67)]
    b = lbm.Batch(inst, window=20, conv=lbm.CONV_NONE, max_steps=10 ** 6, rows_per_item=rows)
    g, l, _ = lbm.maxwell(lbm.temperature(0.9))
    b.init_slabs([g] * 4, [l] * 4, [5.0] * 4)
    assert b.run(2) == 4
    assert all(r["steps"] == 40 for r in b.results())
