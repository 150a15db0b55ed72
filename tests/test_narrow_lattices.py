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


def seconds(calls):
    """The shortest of nine passes of each call, taken in turn."""
    out = [[] for _ in calls]
    for k in range(10):
        for call, times in zip(calls, out):
            t = time.perf_counter()
            call()
            if k:
                times.append(time.perf_counter() - t)
    return [min(t) for t in out]


@pytest.mark.gpu
@pytest.mark.parametrize("nx,ny", [(1, 31001), (1, 200000), (2, 15500), (3, 20000), (5, 20000),
                                   (1, 5000), (3, 3000)])
def test_the_automatic_kernel_is_no_slower(nx, ny):
    rho = np.full((ny, nx), 0.12) * np.random.default_rng(1).uniform(0.999, 1.001, (ny, nx))
    lats = []
    # (the one-step kernel that the automatic choice has for the width)
    for variant in (lbm.VARIANT_AUTO, lbm.VARIANT_REGISTER if nx % 2 else lbm.VARIANT_PAIR):
        lat = lbm.Lattice(nx, ny, 0.9)
        lat.set_variant(variant)
        lat.init_density(rho)
        lats.append(lat)
    auto, one = seconds([lambda lat=lat: lat.step(400, lbm.IMPROVED, 0.8, 0.1) for lat in lats])
    for lat in lats:
        lat.close()
    assert auto < 1.1 * one


@pytest.mark.gpu
@pytest.mark.parametrize("others", [0, 1, 24])
def test_batch_of_one_column_lattices_is_no_slower(others):
    widths = [1] * 96 + [32 + 3 * k for k in range(others)]
    inst = [dict(nx=nx, ny=320, T_over_Tc=0.9, tau=0.8, sigma=0.1, scheme=lbm.IMPROVED)
            for nx in widths]
    g, l, _ = lbm.maxwell(lbm.temperature(0.9))
    n, ms, density = len(inst), {}, {}
    for mode in (lbm.BATCH_AUTO, lbm.BATCH_WORKLIST):
        b = lbm.Batch(inst, window=200, conv=lbm.CONV_NONE, max_steps=10 ** 8, mode=mode,
                      rows_per_item=16)
        b.init_slabs([g] * n, [l] * n, [5.0] * n)
        times = []
        for _ in range(9):
            before = b.stats()["gpu_ms"]
            b.run(1)
            times.append(b.stats()["gpu_ms"] - before)
        ms[mode] = np.median(times)
        density[mode] = [b.density(k) for k in (0, n - 1)]
    for got, want in zip(density[lbm.BATCH_AUTO], density[lbm.BATCH_WORKLIST]):
        assert np.array_equal(got, want)
    assert ms[lbm.BATCH_AUTO] < 1.2 * ms[lbm.BATCH_WORKLIST]


@pytest.mark.gpu
def test_a_batch_goes_on_when_only_its_one_column_lattices_are_left():
    inst = [dict(nx=nx, ny=64, T_over_Tc=t, tau=tau, sigma=0.0, scheme=lbm.SC)
            for nx, t, tau in ((32, 0.45, 0.6), (1, 0.9, 1.0), (1, 0.85, 0.9))]
    b = lbm.Batch(inst, window=102, conv=lbm.CONV_NONE, max_steps=10 ** 8)
    mx = [lbm.maxwell(lbm.temperature(d["T_over_Tc"]))[:2] for d in inst]
    b.init_slabs([m[0] for m in mx], [m[1] for m in mx], [5.0] * 3)
    start = [b.density(k).astype(np.float64) for k in range(3)]
    for k in range(3):
        b.init_density(k, start[k])
    assert b.run(4) == 2 and b.result(0)["status"] == lbm.RUN_DIVERGED
    for k in (1, 2):
        with lbm.Lattice(1, 64, inst[k]["T_over_Tc"]) as lat:
            lat.set_variant(lbm.VARIANT_REGISTER)
            lat.init_density(start[k])
            lat.step(4 * 102, lbm.SC, inst[k]["tau"])
            for got, want in zip(b.moments(k), lat.observe()):
                assert np.array_equal(got, want)
