"""Host rules of the two-step launches (lbm_geometry.h, lbm_batch_host.h),
compiled with the host C++ compiler: every row of every strip exactly once."""
import ctypes
import os
import subprocess

import numpy as np
import pytest

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))
SOURCE = r"""
#include "lbm_batch_host.h"
#include "lbm_geometry.h"
extern "C" {
void geometry(int nx, int ny, int* out) {
  const lbm::StripGeometry g = lbm::two_step_geometry(nx, ny, 152);
  out[0] = g.n_strips; out[1] = g.band_rows; out[2] = g.n_bands; out[3] = g.grid;
}
void tiles(int nx, int ny, int* out) {
  const lbm::TileGeometry g = lbm::tile_geometry(0, 0, nx, ny, 0, 4.0, 152);
  out[0] = g.n_cols; out[1] = g.rows; out[2] = g.grid; out[3] = g.threads;
}
int applies(int variant, int precision, int nx, int ny, int rows, double b) {
  return lbm::two_step_applies(variant, precision, nx, ny, rows, b);
}
static std::vector<lbm::TwoLattice> lattices(int n, const int* sizes) {
  std::vector<lbm::TwoLattice> v;
  for (int i = 0; i < n; ++i) v.push_back(lbm::TwoLattice{i, sizes[2 * i], sizes[2 * i + 1]});
  return v;
}
int items(int n, const int* sizes, int rows, int* out, int cap) {
  std::vector<lbm::TwoItem> v;
  lbm::two_items(lattices(n, sizes), rows, v);
  for (int k = 0; k < int(v.size()) && k < cap; ++k) {
    out[4 * k] = v[k].inst; out[4 * k + 1] = v[k].strip;
    out[4 * k + 2] = v[k].y0; out[4 * k + 3] = v[k].y1;
  }
  return int(v.size());
}
int bands(int nx, int ny, int rows) { return lbm::two_item_bands(nx, ny, rows); }
int strips(int nx) { return lbm::two_item_strips(nx); }
int grid(int n) { return lbm::two_item_grid(n); }
int rows(int n, const int* sizes) { return lbm::two_item_rows(lattices(n, sizes), 152); }
}
"""


@pytest.fixture(scope="module")
def H(tmp_path_factory):
    d = tmp_path_factory.mktemp("two_step")
    src, so = d / "h.cpp", d / "h.so"
    src.write_text(SOURCE)
    subprocess.run(["g++", "-std=c++17", "-O1", "-shared", "-fPIC", "-I",
                    os.path.join(ROOT, "include"), "-I",
                    os.path.join(ROOT, "paper_1204_4098_gb300", "csrc"), str(src), "-o", str(so)],
                   check=True)
    return ctypes.CDLL(str(so))


def test_bands_cover_the_rows_in_one_wave(H):
    rng = np.random.default_rng(0)
    for nx, ny in [(1, 40000), (40000, 1), (8192, 8192), (200, 200)] + \
            [tuple(int(2 ** v) for v in rng.uniform(0, 13, 2)) for _ in range(200)]:
        out = (ctypes.c_int * 4)()
        H.geometry(nx, ny, out)
        n_strips, rows, bands, grid = out
        assert n_strips == (nx + 55) // 56 and grid == n_strips * bands
        assert bands * rows >= ny > (bands - 1) * rows
        assert grid <= max(152 * 12, n_strips)


def test_tiles_cover_the_lattice_in_one_wave(H):
    rng = np.random.default_rng(1)
    for nx, ny in [(1, 1), (2432, 1), (2433, 1), (1, 4864), (1, 4865)] + \
            [tuple(int(2 ** v) for v in rng.uniform(0, 12, 2)) for _ in range(300)]:
        out = (ctypes.c_int * 4)()
        H.tiles(nx, ny, out)
        cols, rows, grid, threads = out
        if rows == 0:  # too large for one wave of tiles of at most 32 rows
            assert (nx + 15) // 16 > 152 or -(-ny // (152 // ((nx + 15) // 16))) > 32
            continue
        assert cols == (nx + 15) // 16 and grid % cols == 0 and grid <= 152
        assert grid // cols * rows >= ny > (grid // cols - 1) * rows
        assert 2 * (threads // 32) >= rows + 16 and threads <= 768


def test_which_lattices_take_two_steps(H):
    H.applies.argtypes = [ctypes.c_int] * 5 + [ctypes.c_double]
    assert H.applies(0, 0, 200, 200, 0, 4.0)
    assert not H.applies(0, 0, 100, 100, 0, 4.0)       # too small
    assert not H.applies(0, 0, 1 << 16, 1 << 15, 0, 4.0)  # offsets beyond 32 bits
    assert not H.applies(0, 0, 200, 200, 8, 4.0)       # a requested band height
    assert not H.applies(0, 0, 200, 200, 0, 1e-13)     # subnormal reciprocals possible
    for variant in (1, 2, 3):
        assert not H.applies(variant, 0, 4096, 4096, 0, 4.0)
    assert not H.applies(0, 1, 4096, 4096, 0, 4.0)     # FP64
    for precision in (2, 3):  # 16-bit columns go in aligned pairs
        assert H.applies(0, precision, 4096, 4096, 0, 4.0)
        assert not H.applies(0, precision, 4095, 4096, 0, 4.0)


@pytest.mark.parametrize("rows", [4, 7, 33, 500])
def test_batch_items_cover_every_row_once_longest_first(H, rows):
    rng = np.random.default_rng(rows)
    sizes = [(2, 9), (32, 320), (33, 7), (64, 1), (65, 100), (512, 300), (1, 5)] + \
        [tuple(int(v) for v in rng.integers(1, 400, 2)) for _ in range(30)]
    flat = (ctypes.c_int * (2 * len(sizes)))(*[v for s in sizes for v in s])
    cap = sum(H.strips(nx) * H.bands(nx, ny, 4) for nx, ny in sizes)  # as allocated
    out = (ctypes.c_int * (4 * cap))()
    n = H.items(len(sizes), flat, rows, out, cap)
    assert n <= cap
    got = np.array(out[:4 * n]).reshape(n, 4)
    lengths = got[:, 3] - got[:, 2]
    assert np.all(lengths[:-1] >= lengths[1:]) and lengths[-1] >= 1
    for i, (nx, ny) in enumerate(sizes):
        for s in range(H.strips(nx)):
            mine = got[(got[:, 0] == i) & (got[:, 1] == s)]
            covered = np.concatenate([np.arange(a, b) for a, b in mine[:, 2:]])
            assert sorted(covered) == list(range(ny))
    assert 4 <= H.rows(len(sizes), flat) <= 256


def test_grids_round_up_in_few_steps(H):
    seen = set()
    for n in range(1, 20000):
        g = H.grid(n)
        assert n <= g <= max(n + 63, int(1.125 * n) + 1)
        seen.add(g)
    assert len(seen) < 100
