"""The register transforms at every length that has them and that
test_gpu_spectra.py does not cover: structure factors on each axis against numpy,
and the coloured noise of the modified equilibrium against the oracle."""
import numpy as np
import pytest

import oracle
from paper_1012_3632_gb300 import MODES, Context, inputs, landau_free_energy

pytestmark = pytest.mark.gpu

LENGTHS = [18, 24, 27, 30, 36, 40, 45, 50, 54, 60, 72, 75, 80, 81, 90, 100, 108, 120, 125, 144, 150, 160, 162, 180, 216,
           240, 250, 270, 288, 300, 320, 324, 375, 405, 432, 450, 480, 486, 500, 540, 576, 600, 625, 640, 648, 675, 720,
           729, 750, 768, 800, 810, 864, 900, 960, 972, 1000]


@pytest.mark.parametrize("n", LENGTHS)
def test_structure_factor_on_each_axis(n):
    for dims in ((n, 3, 2), (5, n, 3), (9, 2, n)):
        X, Y, Z = dims
        with Context(19, dims, 1.1, kT=1e-4, seed=3) as c:
            c.init(thermal=True)
            c.step(1)
            f = c.moments(MODES)[7].reshape(Z, Y, X).copy()
            got = c.structure_factor(7)
            first = c.structure_factor(7, accumulate=True)
            mean = c.structure_factor(7, accumulate=True)
        want = (np.abs(np.fft.fftn(f)) ** 2 / f.size).ravel()
        want[0] = 0.0
        # 2^-24 for each of at most 30 passes with a twiddle product, a few roundings a
        # pass, against the field's 2-norm (the bound of test_gpu_spectra.py)
        eps = 2.0 ** -24
        scale = np.sqrt(want * (f ** 2).sum()) + 100 * eps * (f ** 2).sum()
        assert (np.abs(got - want) <= 2 * 100 * eps * scale).all()
        assert np.array_equal(first, got)
        assert np.abs(mean - got).max() <= 2.0 ** -52 * got.max()


@pytest.mark.parametrize("dims", [(18, 24), (27, 30), (36, 25), (40, 45), (50, 36)])
def test_coloured_noise(dims):
    dims = (*dims, 1)
    kw = dict(kT=1e-6, omega_shear=1.1, omega_bulk=0.9, omega_ghost=1.3, seed=8)
    fe = dict(landau_free_energy(1.0, 0.5, 0.1, 0.08), model=1)
    rho = inputs.uniform_density(dims, rho_c=1.0, amp=0.02, seed=2)
    with Context(9, dims, precision="fp32", free_energy=fe, **kw) as c:
        c.init(rho=rho)
        c.step(20)
        got = c.get_populations()
    p = oracle.Params(Q=9, dims=dims, nonideal=True, A=fe["A"], B=fe["B"], rho_c=fe["rho_c"], kappa=fe["kappa"],
                      total=True, model=1, **kw)
    want = oracle.run(p, oracle.init(p, rho=rho), 0, 20)
    assert np.abs(got - want).max() <= 2e-5  # the FP32 parity tolerance
