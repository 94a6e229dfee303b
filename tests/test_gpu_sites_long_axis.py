"""The one-site steps (k_sites) over tiles and over threads in line, and on lattices
with more tile rows along y than a three-dimensional grid takes (65535).  Without
noise a state that repeats along y stays the repeated state of the short lattice,
bit for bit."""
import numpy as np
import pytest

from paper_1012_3632_gb300 import Context, inputs

pytestmark = pytest.mark.gpu


# tiles of 32 x 4 (D2Q9) and 32 x 2 x 2 sites; X = 33 and 5 leave their tiles partly
# empty, so that the threads go in line
@pytest.mark.parametrize("Q,X,Y,prec", [(9, 32, 270000, "fp32"), (9, 32, 270000, "bf16"), (9, 33, 1200, "bf16"),
                                        (9, 31, 1200, "fp32"), (19, 31, 131076, "bf16"), (19, 32, 131076, "fp64"),
                                        (19, 33, 600, "bf16"), (19, 5, 131076, "fp64")])
def test_repeated_state(Q, X, Y, prec):
    period = 12
    rho = inputs.uniform_density((X, period, 1), seed=6).reshape(period, X)
    kw = dict(omega_shear=1.1, omega_bulk=0.9, omega_ghost=1.3, kT=0.0, precision=prec)
    with Context(Q, (X, period, 1), **kw) as c:
        c.init(rho=rho.ravel())
        c.step(2)
        want = c.get_populations().reshape(Q, 1, period, X)
    with Context(Q, (X, Y, 1), **kw) as c:
        c.init(rho=np.tile(rho, (Y // period, 1)).ravel())
        c.step(2)
        got = c.get_populations().reshape(Q, Y // period, period, X)
    assert np.array_equal(got, np.broadcast_to(want, got.shape))
