"""Two-step windows of the batch engine: what their device time covers, and
windows whose launches are no whole number of the captured chunks."""
import numpy as np
import pytest

from paper_1204_4098_gb300 import lbm

pytestmark = pytest.mark.gpu

T = 0.9
SMALL = [dict(nx=nx, ny=160, T_over_Tc=T, tau=0.8, sigma=0.1, scheme=lbm.IMPROVED)
         for nx in (32, 40, 48, 64, 72, 80)]


def batch(window, instances=SMALL, rows=16):
    b = lbm.Batch(instances, window=window, conv=lbm.CONV_NONE, max_steps=10 ** 8,
                  rows_per_item=rows)
    g, l, _ = lbm.maxwell(lbm.temperature(T))
    n = len(instances)
    b.init_slabs([g] * n, [l] * n, [5.0] * n)
    return b


def window_ms(b, n=1):
    ms = []
    for _ in range(n):
        before = b.stats()["gpu_ms"]
        b.run(1)
        ms.append(b.stats()["gpu_ms"] - before)
    return ms


def test_device_time_of_a_window_leaves_out_the_capture_of_its_graph():
    window_ms(batch(100), 3)  # kernels loaded, clocks up
    # the first window of a new batch captures its graph, the others have it
    first, later = [], []
    for _ in range(5):
        first_ms, *rest = window_ms(batch(100), 6)
        first.append(first_ms)
        later += rest
    assert min(first) < 1.5 * np.median(later)


def test_short_windows_cost_no_more_per_step_than_a_chunk():
    # 98 steps are 48 launches a chain and two steps one by one, 100 one chunk
    step = {}
    for window in (100, 98, 50):
        b = batch(window)
        window_ms(b, 3)
        step[window] = np.median(window_ms(b, 9)) / window
    # a window itself (tail, reduction, gaps) costs less than 50 steps of these
    assert step[98] < 1.5 * step[100]
    assert step[50] < 2.0 * step[100]


# (launches a chain: 0, 2, 8, 10; 48 and two steps; a chunk; a chunk and 2, 24, 48)
@pytest.mark.parametrize("window", [2, 4, 6, 16, 20, 98, 100, 102, 104, 150, 196])
def test_windows_of_any_length(window):
    inst = [dict(SMALL[k % 6], nx=nx, ny=ny) for k, (nx, ny) in
            enumerate([(32, 41), (64, 33), (114, 40), (66, 19), (57, 30), (1, 21), (3, 33)])]
    b = batch(window, inst, rows=8)
    start = []
    for k, d in enumerate(inst):
        start.append(b.density(k).astype(np.float64))
        b.init_density(k, start[k])
    assert b.run(2) == len(inst)
    for k, d in enumerate(inst):
        with lbm.Lattice(d["nx"], d["ny"], T) as lat:
            lat.set_variant(lbm.VARIANT_REGISTER)
            lat.init_density(start[k])
            lat.step(2 * window, d["scheme"], d["tau"], d["sigma"])
            for got, want in zip(b.moments(k), lat.observe()):
                assert np.array_equal(got, want), (k, d)


def test_a_batch_of_another_mode_holds_no_two_step_tables():
    torch = pytest.importorskip("torch")
    nx, ny = 2, 1 << 24  # (two-step items of 4 rows: 64 MB)
    held = {}
    for mode in (lbm.BATCH_AUTO, lbm.BATCH_WORKLIST):
        torch.cuda.synchronize()
        before = torch.cuda.mem_get_info()[0]
        b = lbm.Batch([dict(SMALL[0], nx=nx, ny=ny)], mode=mode)
        held[mode] = before - torch.cuda.mem_get_info()[0]
        b.close()
    assert held[lbm.BATCH_AUTO] - held[lbm.BATCH_WORKLIST] > 60 << 20
