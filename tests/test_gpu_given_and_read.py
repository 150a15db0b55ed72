"""Initial states and read-back: the populations of a given state, the domain
check of its densities and the velocities read back, against the same formulas
in FP64 on the host."""
import numpy as np
import pytest

import oracle
from paper_1204_4098_gb300 import lbm

pytestmark = pytest.mark.gpu

E = np.array([(0, 0), (1, 0), (0, 1), (-1, 0), (0, -1), (1, 1), (-1, 1), (-1, -1), (1, -1)])
W = np.array([4 / 9] + [1 / 9] * 4 + [1 / 36] * 4)
SIZES = [(1, 1), (1, 9), (9, 1), (31, 8), (32, 7), (33, 17), (200, 65)]  # 32 x 8 per CTA


def _equilibrium(rho, u, v):
    eu = E[:, 0, None, None] * u + E[:, 1, None, None] * v
    return W[:, None, None] * rho * (1.0 + 3.0 * eu + 4.5 * eu * eu - 1.5 * (u * u + v * v))


@pytest.mark.parametrize("precision", [lbm.FP32, lbm.FP64])
@pytest.mark.parametrize("nx,ny", SIZES)
@pytest.mark.parametrize("given", ["rest", "ux", "uy", "both"])
def test_populations_of_a_given_state(nx, ny, given, precision):
    rng = np.random.default_rng(nx + 100 * ny)
    rho = rng.uniform(0.02, 0.3, (ny, nx))
    ux = rng.uniform(-0.1, 0.1, (ny, nx)) if given in ("ux", "both") else None
    uy = rng.uniform(-0.1, 0.1, (ny, nx)) if given in ("uy", "both") else None
    with lbm.Lattice(nx, ny, 0.85, precision=precision) as lat:
        lat.init_density(rho, ux, uy)
        f = lat.populations()
    zero = np.zeros_like(rho)
    want = _equilibrium(rho, zero if ux is None else ux, zero if uy is None else uy)
    # about ten roundings in FP64 of terms below 2 rho w, then one to the storage type
    eps = 2.0 ** -24 if precision == lbm.FP32 else 0.0
    assert np.all(np.abs(f - want) <= want * eps + 10 * 2.0 ** -53 * 2 * W[:, None, None] * rho)


def _radicand(rho):
    T = lbm.temperature(0.85)
    eta = rho  # a = R = 1, b = 4, G = -1
    p = rho * T * (1 + eta + eta**2 - eta**3) / (1 - eta) ** 3 - rho * rho
    return -2.0 * (p - rho / 3.0)


@pytest.mark.parametrize("precision", [lbm.FP32, lbm.FP64, lbm.BF16DEV])
@pytest.mark.parametrize("edge", ["radicand", "zero", "negative", "eta"])
def test_domain_of_given_densities(edge, precision):
    with lbm.Lattice(40, 11, 0.85, precision=precision) as lat:
        if edge == "radicand":  # the density at which the radicand changes sign
            lo, hi = 0.2, 0.99
            for _ in range(200):
                mid = 0.5 * (lo + hi)
                lo, hi = (mid, hi) if _radicand(mid) > 0 else (lo, mid)
            inside, outside = lo * (1 - 1e-9), lo * (1 + 1e-9)
        else:
            inside, outside = {"zero": (1e-40, 0.0), "negative": (1e-5, -1e-5),
                               "eta": (0.1, 1.0)}[edge]
        rho = np.full((11, 40), 0.12)
        rho[7, 33] = inside
        lat.init_density(rho)
        rho[7, 33] = outside
        with pytest.raises(lbm.LbmError):
            lat.init_density(rho)


@pytest.mark.parametrize("nx", [64, 63])  # two columns a lane, one
@pytest.mark.parametrize("scale", [1e-30, 1e-12, 1.0, 1e12, 1e30])
def test_velocities_are_the_rounded_quotients(nx, scale):
    rng = np.random.default_rng(nx)
    f = rng.uniform(0.01, 0.2, (9, 40, nx)) * scale * 10.0 ** rng.uniform(-4, 4, (40, nx))
    f[:, 3] = 0.0
    with lbm.Lattice(nx, 40, 0.85) as lat:
        lat.init_density(np.full((40, nx), 0.12))
        lat.step(1, lbm.NOFORCE, 1.0)  # read-back without the force from here on
        lat.set_populations(f)
        f = lat.populations().astype(np.float32)
        out = [np.zeros((40, nx)) for _ in range(3)]
        d = lbm.ctypes.POINTER(lbm.ctypes.c_double)
        lbm.lib().lbm_get_moments(lat.ctx, *[o.ctypes.data_as(d) for o in out])
    rho = f[0]
    for a in range(1, 9):
        rho = rho + f[a]
    jx = (f[1] - f[3]) + (f[5] - f[6]) + (f[8] - f[7])
    jy = (f[2] - f[4]) + (f[5] + f[6]) - (f[7] + f[8])
    with np.errstate(all="ignore"):
        want = [rho.astype(np.float64)] + [j.astype(np.float64) / rho for j in (jx, jy)]
    for got, w in zip(out, want):
        assert np.array_equal(got, w, equal_nan=True)


@pytest.mark.parametrize("scale", [1e-32, 1e-30, 0.1])  # 2^-100 = 7.9e-31: below it, above it
@pytest.mark.parametrize("scheme", [lbm.SC, lbm.IMPROVED, lbm.MRT])
def test_fp64_steps_at_densities_of_any_scale(scheme, scale):
    nx, ny = 37, 21
    rho = scale * np.random.default_rng(3).uniform(0.95, 1.05, (ny, nx))
    with lbm.Lattice(nx, ny, 0.85, precision=lbm.FP64) as lat:
        lat.init_density(rho)
        lat.step(2, scheme, 0.9, 0.1)
        got = lat.observe()
    ref = oracle.Lattice(nx, ny, 0.85)
    ref.init_density(rho)
    rc, _ = ref.step(2, scheme, 0.9, 0.1)
    assert rc == 0
    # two steps of ~100 roundings each, errors grown tenfold at most by differences
    tol = 2 * 100 * 10 * 2.0 ** -53
    for g, w, unit in zip(got, ref.observe(), (scale, 1.0, 1.0)):
        assert np.max(np.abs(g - w)) <= tol * unit
