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
  out[0] = g.n_cols; out[1] = g.rows; out[2] = g.grid; out[3] = g.threads; out[4] = g.steps;
}
int applies(int variant, int precision, int nx, int ny, int rows, double b) {
  return lbm::two_step_applies(variant, precision, nx, ny, rows, b);
}
static std::vector<lbm::TwoLattice> lattices(int n, const int* sizes) {
  std::vector<lbm::TwoLattice> v;
  for (int i = 0; i < n; ++i) v.push_back(lbm::TwoLattice{i, sizes[2 * i], sizes[2 * i + 1]});
  lbm::two_layouts(v);
  return v;
}
// 6 ints per item: instance, strip, rows, chain, layout
int items(int n, const int* sizes, int rows, int wanted, int* out, int cap) {
  int m = 0, c = 0;
  for (const lbm::TwoChain& chain : lbm::two_chains(lattices(n, sizes), wanted)) {
    std::vector<lbm::TwoItem> v;
    lbm::two_items(chain.lat, rows, v);
    for (const lbm::TwoItem& t : v) {
      if (m < cap) {
        const int row[6] = {t.inst, t.strip, t.y0, t.y1, c, chain.layout};
        for (int k = 0; k < 6; ++k) out[6 * m + k] = row[k];
      }
      ++m;
    }
    ++c;
  }
  return m;
}
int bands(int nx, int ny, int rows) {
  return lbm::two_item_bands(lbm::TwoLattice{0, nx, ny, lbm::kTwoBatchAny}, rows);
}
int strips(int nx) {
  return lbm::two_item_strips(lbm::TwoLattice{0, nx, 1, lbm::kTwoBatchAny});
}
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
    def rows_of(steps, nx, ny):  # of the tiles when all start in one wave, else 0
        cols = -(-nx // (32 - 4 * steps))
        rows = -(-ny // (152 // cols)) if cols <= 152 else 48
        return rows if rows + 4 * steps <= 48 else 0

    for nx, ny in [(1, 1), (2432, 1), (2433, 1), (3648, 1), (3649, 1), (1, 4864), (1, 6080),
                   (1, 6081), (2 ** 31 - 1, 1), (1, 2 ** 31 - 1)] + \
            [tuple(int(2 ** v) for v in rng.uniform(0, 12, 2)) for _ in range(300)]:
        out = (ctypes.c_int * 5)()
        H.tiles(nx, ny, out)
        cols, rows, grid, threads, steps = out
        if rows == 0:
            assert not any(rows_of(t, nx, ny) for t in (2, 3, 4))
            continue
        assert 2 <= steps <= 4 and not any(rows_of(t, nx, ny) for t in range(steps + 1, 5))
        assert cols == -(-nx // (32 - 4 * steps)) and grid % cols == 0 and grid <= 152
        assert grid // cols * rows >= ny > (grid // cols - 1) * rows
        assert 2 * (threads // 32) >= rows + 4 * steps and threads <= 768


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


MIXED = [(2, 9), (32, 320), (33, 7), (64, 1), (65, 100), (512, 300), (1, 5)]
EVEN = [(2, 9), (32, 320), (64, 30), (66, 100), (512, 300)]
NARROW = [(32, 320)] * 9 + [(33, 30), (1, 5)]


@pytest.mark.parametrize("rows", [4, 7, 33, 500])
@pytest.mark.parametrize("first,odd", [(MIXED, True), (EVEN, False), (NARROW, True)])
def test_batch_items_cover_every_row_once_longest_first(H, rows, first, odd):
    rng = np.random.default_rng(rows)
    sizes = first + [tuple(int(v) for v in rng.integers(1, 30, 2) * (1 if odd else 2))
                     for _ in range(20)]
    flat = (ctypes.c_int * (2 * len(sizes)))(*[v for s in sizes for v in s])
    cap = sum(H.strips(nx) * H.bands(nx, ny, 4) for nx, ny in sizes)  # as allocated
    out = (ctypes.c_int * (6 * cap))()
    n = H.items(len(sizes), flat, rows, 3, out, cap)
    assert n <= cap
    got = np.array(out[:6 * n]).reshape(n, 6)
    chains = got[:, 4].max() + 1
    assert 1 <= chains <= 3 + 3
    for c in range(chains):  # one layout each, longest items first
        mine = got[got[:, 4] == c]
        lengths = mine[:, 3] - mine[:, 2]
        assert len(set(mine[:, 5])) == 1
        assert np.all(lengths[:-1] >= lengths[1:]) and lengths[-1] >= 1
    for i, (nx, ny) in enumerate(sizes):
        mine = got[got[:, 0] == i]
        assert len(set(mine[:, 4])) == 1  # an instance belongs to one chain
        layout = mine[0, 5]
        if layout == 0:
            assert nx % 2 == 0
        elif layout == 2:
            assert nx % 2 == 0 and nx <= 64
        for s in range(1 if layout == 2 else (nx + 55) // 56):
            rows_of = mine[mine[:, 1] == s]
            covered = np.concatenate([np.arange(a, b) for a, b in rows_of[:, 2:4]])
            assert sorted(covered) == list(range(ny))
        assert mine[:, 1].max() == (0 if layout == 2 else (nx + 55) // 56 - 1)
    assert 4 <= H.rows(len(sizes), flat) <= 256


def test_grids_round_up_in_few_steps(H):
    seen = set()
    for n in range(1, 20000):
        g = H.grid(n)
        assert n <= g <= max(n + 63, int(1.25 * n) + 1)
        seen.add(g)
    assert len(seen) < 100
