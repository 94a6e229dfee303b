"""D3Q19 steps of site pairs on a lattice with more tile rows along y than a
three-dimensional grid takes (65535): the tiles are then numbered along one
dimension.  Without noise a state that repeats along y stays the repeated state
of the short lattice, bit for bit."""
import numpy as np
import pytest

from paper_1012_3632_gb300 import Context, inputs

pytestmark = pytest.mark.gpu

EXCESS = dict(A=-0.01, B=0.1, rho_c=1.0, kappa=0.02)


@pytest.mark.parametrize("fe", [None, EXCESS], ids=["ideal", "excess"])
@pytest.mark.parametrize("X", [33, 64])
def test_repeated_state(X, fe):
    period, Y = 12, 131076
    rho = inputs.uniform_density((X, period, 1), seed=6).reshape(period, X)
    kw = dict(omega_shear=1.1, omega_bulk=0.9, omega_ghost=1.3, kT=0.0, precision="fp32", free_energy=fe)
    with Context(19, (X, period, 1), **kw) as c:
        c.init(rho=rho.ravel())
        c.step(3)
        want = c.get_populations().reshape(19, 1, period, X)
    with Context(19, (X, Y, 1), **kw) as c:
        c.init(rho=np.tile(rho, (Y // period, 1)).ravel())
        c.step(3)
        got = c.get_populations().reshape(19, Y // period, period, X)
    assert np.array_equal(got, np.broadcast_to(want, got.shape))
