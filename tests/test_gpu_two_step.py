"""The launches of several steps that the automatic kernel choice makes (two
steps on strips, up to four on tiles) against the one-step, one-column kernel
(VARIANT_REGISTER): the same populations, bit for bit."""
import numpy as np
import pytest

from paper_1204_4098_gb300 import inputs, lbm

pytestmark = pytest.mark.gpu

T = 0.9
SCHEMES = [lbm.SC, lbm.EDM, lbm.IMPROVED, lbm.NOFORCE, lbm.EDM_MOD, lbm.LADD, lbm.MRT]


def field(nx, ny, seed):
    g, l, _ = lbm.maxwell(lbm.temperature(T))
    rng = np.random.default_rng(seed)
    rho = inputs.spinodal(nx, ny, 0.5 * (g + l), amp=0.02, seed=seed)
    return rho, rng.uniform(-0.02, 0.02, (ny, nx)), rng.uniform(-0.02, 0.02, (ny, nx))


def populations(nx, ny, state, steps, scheme, variant, precision=lbm.FP32):
    with lbm.Lattice(nx, ny, T, precision=precision) as lat:
        lat.set_variant(variant)
        lat.set_mrt_rates(0.8, 1.1, 1.3)
        lat.init_density(*state)
        st = lat.step(steps, scheme, 0.8, 0.1, raise_on_error=False)
        return st, lat.populations()


def check(nx, ny, state, steps, scheme, precision=lbm.FP32):
    st_a, auto = populations(nx, ny, state, steps, scheme, lbm.VARIANT_AUTO, precision)
    st_r, ref = populations(nx, ny, state, steps, scheme, lbm.VARIANT_REGISTER, precision)
    assert st_a == st_r
    return auto, ref


# around the 56 columns of a strip and its 64 loaded ones, widths and heights
# below the halo (wrapped several times), odd and even, bands of one row to many
@pytest.mark.parametrize("nx,ny", [
    (1, 31001), (2, 15500), (3, 10400), (8, 4000), (9, 3500), (55, 600), (56, 600), (57, 601),
    (64, 512), (111, 300), (112, 300), (113, 301), (176, 176), (177, 179), (4099, 9), (4100, 8),
    (8000, 4), (10400, 3), (15501, 2), (31000, 1), (31001, 1), (640, 333)])
@pytest.mark.parametrize("steps", [2, 5])
def test_sizes(nx, ny, steps):
    auto, ref = check(nx, ny, field(nx, ny, nx + ny), steps, lbm.IMPROVED)
    assert np.array_equal(auto, ref)


# both kernels of each layout: launches of up to 8 warps per SM and of more
@pytest.mark.parametrize("nx,ny", [(900, 800), (901, 800), (2000, 1900), (2001, 1900)])
@pytest.mark.parametrize("scheme,precision", [(s, lbm.FP32) for s in SCHEMES] +
                         [(lbm.IMPROVED, lbm.BF16DEV), (lbm.MRT, lbm.FP16DEV)])
def test_few_and_many_warps(nx, ny, scheme, precision):
    auto, ref = check(nx, ny, field(nx, ny, 11), 3, scheme, precision)
    assert np.array_equal(auto, ref)


# 16-bit storage: the rounding between the two steps of a launch, every scheme
@pytest.mark.parametrize("precision", [lbm.BF16DEV, lbm.FP16DEV])
@pytest.mark.parametrize("nx,ny,scheme", [(200, 190, s) for s in SCHEMES] + [
    (2, 15500, lbm.IMPROVED), (56, 600, lbm.IMPROVED), (58, 601, lbm.SC), (112, 300, lbm.EDM),
    (640, 333, lbm.IMPROVED), (31000, 1, lbm.IMPROVED), (15500, 2, lbm.SC),
    (641, 333, lbm.IMPROVED)])  # (odd nx: one step per launch)
def test_16_bit_storage(precision, nx, ny, scheme):
    auto, ref = check(nx, ny, field(nx, ny, nx + ny), 21, scheme, precision)
    assert np.array_equal(auto, ref)


# tiles: one cell to the largest lattice they cover in a wave, widths around
# the 16, 20 and 24 columns of a tile (of 4, 3 and 2 steps), odd and even rows
# per tile, a ragged last tile
@pytest.mark.parametrize("nx,ny", [
    (1, 1), (2, 9), (1, 152), (15, 33), (16, 16), (17, 5), (32, 32), (40, 36), (33, 47), (64, 64),
    (100, 3), (3, 100), (2432, 1), (2417, 32), (120, 128), (270, 250), (48, 1600), (257, 101),
    (300, 300), (299, 331), (2441, 31), (3039, 36), (360, 360), (361, 341), (3647, 40), (1, 5000)])
@pytest.mark.parametrize("steps", [2, 3, 4, 9])
def test_tiles(nx, ny, steps):
    auto, ref = check(nx, ny, field(nx, ny, nx + ny), steps, lbm.IMPROVED)
    assert np.array_equal(auto, ref)


@pytest.mark.parametrize("scheme", SCHEMES)
@pytest.mark.parametrize("nx,ny", [(200, 190), (97, 60), (310, 290), (340, 370), (600, 300),
                                   (601, 301)])
def test_schemes_and_step_graphs(scheme, nx, ny):
    # 35 steps: two replays of a graph of 16 and what is left
    auto, ref = check(nx, ny, field(nx, ny, 5), 35, scheme)
    assert np.array_equal(auto, ref)


@pytest.mark.parametrize("nx,ny,precision", [(97, 60, lbm.FP32), (310, 290, lbm.FP32),
                                             (340, 370, lbm.FP32), (601, 301, lbm.FP32),
                                             (200, 190, lbm.BF16DEV), (60, 50, lbm.FP64)])
def test_long_runs_in_step_graphs(nx, ny, precision):
    # graphs of 64 and of 16 steps from either buffer, and what is left
    out = []
    for variant in (lbm.VARIANT_AUTO, lbm.VARIANT_REGISTER):
        with lbm.Lattice(nx, ny, T, precision=precision) as lat:
            lat.set_variant(variant)
            lat.init_density(*field(nx, ny, 7))
            for n in (1, 151, 128, 3, 127, 64):
                if variant == lbm.VARIANT_AUTO:
                    lat.step(n, lbm.IMPROVED, 0.8, 0.1)
                else:
                    for _ in range(n):
                        lat.step(1, lbm.IMPROVED, 0.8, 0.1)
            out.append(lat.populations())
    assert np.array_equal(*out)


@pytest.mark.parametrize("rows", [slice(None), slice(100, 140)])
@pytest.mark.parametrize("scheme", [lbm.IMPROVED, lbm.NOFORCE])
@pytest.mark.parametrize("nx,ny", [(190, 240), (590, 240)])
def test_densities_that_take_the_full_divisions(rows, scheme, nx, ny):
    # 1e-32 is inside the domain of psi but below the range in which the
    # reciprocals are taken without subnormal handling
    rho = np.full((ny, nx), 0.1)
    rho[rows] = 1e-32 * np.random.default_rng(1).uniform(1.0, 2.0, rho[rows].shape)
    auto, ref = check(nx, ny, (rho,), 2, scheme)
    assert np.array_equal(auto, ref, equal_nan=True)


@pytest.mark.parametrize("nx,ny", [(192, 192), (600, 400)])
def test_divergence_is_reported_in_any_step_of_a_launch(nx, ny):
    rho, ux, uy = field(nx, ny, 3)
    with lbm.Lattice(nx, ny, T) as lat:
        lat.init_density(rho, ux, uy)
        good = lat.populations()
    for bad_steps in (1, 2):  # a population lost at the start, or one that leaves later
        f = good.copy()
        f[1, 50, 60] = np.nan if bad_steps == 1 else 0.9
        for variant in (lbm.VARIANT_AUTO, lbm.VARIANT_REGISTER):
            with lbm.Lattice(nx, ny, T) as lat:
                lat.set_variant(variant)
                lat.set_populations(f)
                st = lat.step(2, lbm.SC, 0.8, raise_on_error=False)
                assert st == lbm.LBM_E_DIVERGED
                # the context stays usable
                lat.set_populations(good)
                assert lat.step(4, lbm.SC, 0.8, raise_on_error=False) == lbm.LBM_OK


# every row layout of the batch's two-step windows: whole rows in a half-warp
# (even nx <= 32) and in a warp (<= 64), strips of even and of padded odd
# widths, nx = 1; heights below and around a band
BATCH = [dict(nx=nx, ny=ny, T_over_Tc=T, tau=tau, sigma=0.1, scheme=scheme)
         for k, (nx, ny) in enumerate([(2, 9), (30, 41), (32, 128), (32, 5), (34, 37), (62, 20),
                                       (64, 33), (66, 19), (56, 7), (112, 40), (114, 3), (1, 21),
                                       (3, 33), (57, 30), (63, 1), (65, 18), (113, 25)])
         for scheme, tau in [(SCHEMES[k % 6], 0.8 + 0.02 * k)]]


@pytest.mark.parametrize("window,rows", [(20, 0), (20, 4), (10, 7), (14, 300)])
def test_batch_windows(window, rows):
    b = lbm.Batch(BATCH, window=window, tol=0.0, max_steps=10 ** 6, rows_per_item=rows,
                  conv=lbm.CONV_NONE)
    start = [field(d["nx"], d["ny"], k)[0] for k, d in enumerate(BATCH)]
    for k, r in enumerate(start):
        b.init_density(k, r)
    assert b.run(2) == len(BATCH)
    for k, d in enumerate(BATCH):
        with lbm.Lattice(d["nx"], d["ny"], T) as lat:
            lat.set_variant(lbm.VARIANT_REGISTER)
            lat.init_density(start[k])
            lat.step(2 * window, d["scheme"], d["tau"], d["sigma"])
            for got, want in zip(b.moments(k), lat.observe()):
                assert np.array_equal(got, want), d


def test_batch_instance_that_diverges_leaves_the_others_alone():
    inst = [dict(d) for d in BATCH[:4]]
    inst[1].update(T_over_Tc=0.45, tau=0.6, scheme=lbm.SC)
    b = lbm.Batch(inst, window=400, conv=lbm.CONV_NONE, max_steps=10 ** 6)
    alone = lbm.Batch(inst[2:3], window=400, conv=lbm.CONV_NONE, max_steps=10 ** 6)
    for k, d in enumerate(inst):
        g, l, _ = lbm.maxwell(lbm.temperature(d["T_over_Tc"]))
        rho = inputs.slab_step(d["nx"], d["ny"], g, l)
        b.init_density(k, rho)
        if k == 2:
            alone.init_density(0, rho)
    assert b.run(1) == 3 and alone.run(1) == 1
    assert b.result(1)["status"] == lbm.RUN_DIVERGED
    assert np.array_equal(b.density(2), alone.density(0))


# a caller's graph of an even number of steps leaves the state in the buffer it
# found it in, however many steps its launches take, so it can be replayed
@pytest.mark.parametrize("nx,ny,precision", [
    (66, 40, lbm.FP32), (310, 290, lbm.FP32), (340, 370, lbm.FP32), (600, 300, lbm.FP32),
    (601, 301, lbm.FP32), (600, 300, lbm.BF16DEV), (60, 50, lbm.FP64)])
@pytest.mark.parametrize("steps", [2, 4, 6, 10, 12, 18])
def test_replays_of_captured_steps(nx, ny, precision, steps):
    torch = pytest.importorskip("torch")
    stream = torch.cuda.Stream()
    with lbm.Lattice(nx, ny, T, precision=precision, stream=stream.cuda_stream) as lat:
        lat.init_density(*field(nx, ny, 3))
        torch.cuda.synchronize()
        graph = torch.cuda.CUDAGraph()
        with torch.cuda.graph(graph, stream=stream, capture_error_mode="thread_local"):
            lat.step_async(steps, lbm.IMPROVED, 0.8, 0.1)
        for _ in range(3):
            graph.replay()
        torch.cuda.synchronize()
        got = lat.populations()
    with lbm.Lattice(nx, ny, T, precision=precision) as lat:
        lat.init_density(*field(nx, ny, 3))
        lat.step(3 * steps, lbm.IMPROVED, 0.8, 0.1)
        assert np.array_equal(got, lat.populations())
