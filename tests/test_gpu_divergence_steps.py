"""Divergence in each step of a launch of several: populations that meet in one
cell in a chosen step, and nowhere before, take its density out of the domain of
psi.  The one-step kernel (VARIANT_REGISTER) says in which step that is."""
import numpy as np
import pytest

from paper_1204_4098_gb300 import lbm

pytestmark = pytest.mark.gpu

T, TAU = 0.9, 1e6  # relaxation does nothing in a few steps: populations travel
E = [(0, 0), (1, 0), (0, 1), (-1, 0), (0, -1), (1, 1), (-1, 1), (-1, -1), (1, -1)]


def meeting(nx, ny, x, y, step):
    """Density 0.1 at rest; eight cells step - 1 away send 0.08 to (x, y) each.
    All of it there, 0.74, is above the domain (0.45 or so); two of them in one
    cell, 0.26, are not."""
    f = np.zeros((9, ny, nx))
    f[0] = 0.1
    for a in range(1, 9):
        ex, ey = E[a]
        f[a, (y - (step - 1) * ey) % ny, (x - (step - 1) * ex) % nx] = 0.08
    return f


def status(nx, ny, f, steps, variant, precision):
    with lbm.Lattice(nx, ny, T, precision=precision) as lat:
        lat.set_variant(variant)
        lat.set_populations(f)
        return lat.step(steps, lbm.EDM, TAU, raise_on_error=False)


# launches of four, three and two steps on tiles, of two on strips
@pytest.mark.parametrize("nx,ny,most,precision", [
    (192, 192, 4, lbm.FP32), (300, 300, 3, lbm.FP32), (361, 341, 2, lbm.FP32),
    (600, 400, 2, lbm.FP32), (601, 401, 2, lbm.FP32), (2000, 1900, 2, lbm.FP32),
    (600, 400, 2, lbm.BF16DEV), (600, 400, 2, lbm.FP16DEV)])
@pytest.mark.parametrize("at", [(60, 50), (55, 0), (56, 17), (0, -1)])
def test_a_cell_that_leaves_the_domain_in_one_step(nx, ny, most, precision, at):
    x, y = at[0] % nx, at[1] % ny
    for step in range(1, most + 1):
        f = meeting(nx, ny, x, y, step)
        if step > 1:
            assert status(nx, ny, f, step - 1, lbm.VARIANT_REGISTER, precision) == lbm.LBM_OK
            assert status(nx, ny, f, step - 1, lbm.VARIANT_AUTO, precision) == lbm.LBM_OK
        for variant in (lbm.VARIANT_REGISTER, lbm.VARIANT_AUTO):
            # the launch's last step, and one before its last
            for steps in {step, most}:
                assert status(nx, ny, f, steps, variant, precision) == lbm.LBM_E_DIVERGED
