"""Densities near the lower end of the domain of psi at the columns where two
strips meet: a strip uses psi of columns that its neighbour owns, and has to
notice there what its neighbour notices, so the launches of two steps give the
one-step kernel's populations (VARIANT_REGISTER) bit for bit."""
import numpy as np
import pytest

from paper_1204_4098_gb300 import lbm

pytestmark = pytest.mark.gpu

T = 0.9
# A density at which the radicand of psi, about rho / 2, is below 2^-126 but
# 1 / rho is finite: the bare reciprocal root of it is infinite, its psi is not.
TINY = 2e-38
COLUMNS = [53, 54, 55, 56, 57, 58]  # strips own 56 columns


def run(nx, ny, variant, steps, scheme, tau, rho=None, f=None):
    with lbm.Lattice(nx, ny, T) as lat:
        lat.set_variant(variant)
        if f is None:
            lat.init_density(rho)
        else:
            lat.set_populations(f)
        st = lat.step(steps, scheme, tau, raise_on_error=False)
        return st, lat.populations()


def check(*args, **kw):
    st_a, auto = run(*args[:2], lbm.VARIANT_AUTO, *args[2:], **kw)
    st_r, ref = run(*args[:2], lbm.VARIANT_REGISTER, *args[2:], **kw)
    assert st_a == st_r == lbm.LBM_OK
    assert np.all(np.isfinite(ref))
    assert np.array_equal(auto, ref)


def tiny_column(nx, ny, c):
    rho = np.full((ny, nx), 0.1)
    rho[:, c] = TINY
    return rho


# (FP32 storage: next to other densities a 16-bit deviation cannot hold TINY)
@pytest.mark.parametrize("nx,ny", [(600, 400), (601, 401), (2000, 1900)])
@pytest.mark.parametrize("c", COLUMNS)
def test_first_step(nx, ny, c):
    check(nx, ny, 2, lbm.SC, 0.8, rho=tiny_column(nx, ny, c))


@pytest.mark.parametrize("nx,ny", [(600, 400), (601, 401), (2000, 1900)])
@pytest.mark.parametrize("c", COLUMNS)
def test_second_step(nx, ny, c):
    # The density is 1/8 everywhere, so the first step has no force, and with a
    # relaxation time this long it leaves the populations what they are but for
    # omega f_eq.  Column c moves away, the others rest: the second step finds
    # the 5/9 omega / 8 = TINY that relaxation put in its way.
    f = np.zeros((9, ny, nx))
    f[0] = 0.125
    f[0, :, c] = 0.0
    f[1, :, c] = f[3, :, c] = 0.0625
    check(nx, ny, 2, lbm.EDM, 5.0 / 72.0 / TINY, f=f)


@pytest.mark.parametrize("widths", [(600, 114), (600, 601)])  # columns in pairs, one by one
@pytest.mark.parametrize("c", COLUMNS)
def test_batch(widths, c):
    ny = 60
    inst = [dict(nx=nx, ny=ny, T_over_Tc=T, tau=0.8, sigma=0.0, scheme=lbm.SC) for nx in widths]
    b = lbm.Batch(inst, window=4, conv=lbm.CONV_NONE, max_steps=10 ** 6)
    for k, nx in enumerate(widths):
        b.init_density(k, tiny_column(nx, ny, c))
    assert b.run(1) == len(inst)
    for k, nx in enumerate(widths):
        with lbm.Lattice(nx, ny, T) as lat:
            lat.set_variant(lbm.VARIANT_REGISTER)
            lat.init_density(tiny_column(nx, ny, c))
            lat.step(4, lbm.SC, 0.8)
            for got, want in zip(b.moments(k), lat.observe()):
                assert np.all(np.isfinite(want))
                assert np.array_equal(got, want)
