"""Initial states at rest: a density alone is the state of zero velocities, and
takes no longer than its arithmetic."""
import time

import numpy as np
import pytest

from paper_1204_4098_gb300 import lbm

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("precision", [lbm.FP32, lbm.FP64, lbm.BF16DEV, lbm.FP16DEV])
@pytest.mark.parametrize("nx,ny", [(1, 1), (31, 9), (64, 20), (65, 33)])
def test_no_velocity_is_zero_velocity(nx, ny, precision):
    rho = np.random.default_rng(nx).uniform(0.02, 0.3, (ny, nx))
    f = []
    for u in (None, np.zeros((ny, nx))):
        with lbm.Lattice(nx, ny, 0.85, precision=precision) as lat:
            lat.init_density(rho, u, u)
            f.append(lat.populations())
    assert np.array_equal(*f)


def test_batch_no_velocity_is_the_lattice():
    inst = [dict(nx=nx, ny=20, T_over_Tc=0.85, tau=1.0, sigma=0.0, scheme=lbm.SC)
            for nx in (1, 32, 33, 114, 115)]
    b = lbm.Batch(inst, window=2)
    for k, d in enumerate(inst):
        rho = np.random.default_rng(k).uniform(0.02, 0.3, (20, d["nx"]))
        b.init_density(k, rho)
        with lbm.Lattice(d["nx"], 20, 0.85) as lat:
            lat.init_density(rho)
            assert np.array_equal(b.moments(k)[0], lat.observe()[0])


@pytest.mark.parametrize("precision", [lbm.BF16DEV, lbm.FP16DEV])
def test_16_bit_state_at_rest_takes_its_arithmetic(precision):
    # About 54 operations of the FP64 pipe a cell (nine products, sums and
    # deviations with their conversions) at 0.58 T/s, 100 us, beside the copy of
    # the density and the call, 60 us; FP32 storage, 10 operations, takes 90 us in
    # all.  With f_eq of a moving cell it would be 150 operations, 260 us or more.
    n = 1024
    rho = lbm.host_array((n, n))
    rho[...] = 0.12
    t = {}
    for p in (lbm.FP32, precision):
        with lbm.Lattice(n, n, 0.85, precision=p) as lat:
            lat.init_density(rho)
            times = []
            for _ in range(9):
                t0 = time.perf_counter()
                lat.init_density(rho)
                times.append(time.perf_counter() - t0)
        t[p] = min(times)
    assert t[precision] < 2.3 * t[lbm.FP32]
