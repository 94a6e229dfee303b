"""Structure factors through the register transforms, the radix-by-radix ones
and the direct ones (csrc/flb_fft.cu): every length with a register plan on
every axis, ragged line groups, one- and two-dimensional lattices, against
numpy's FFT of the same field."""
import numpy as np
import pytest

from paper_1012_3632_gb300 import MODES, Context

pytestmark = pytest.mark.gpu

LENGTHS = [32, 48, 64, 96, 128, 135, 192, 200, 225, 243, 256, 360, 384, 400, 512, 1024]
D3 = ([(n, 3, 2) for n in LENGTHS] + [(5, n, 3) for n in LENGTHS] + [(9, 2, n) for n in LENGTHS] +
      [(32, 1, 1), (1, 1, 48), (1, 64, 1), (70, 33, 34), (37, 41, 29), (1031, 3, 2), (24, 90, 50), (67, 64, 128)])


@pytest.mark.parametrize("dims", D3)
@pytest.mark.parametrize("prec", ["fp32", "fp64"])
def test_structure_factor(dims, prec):
    X, Y, Z = dims
    with Context(19, dims, 1.1, kT=1e-4, seed=3, precision=prec) as c:
        c.init(thermal=True)
        c.step(2)
        f = c.moments(MODES)[7].reshape(Z, Y, X).copy()  # a stress mode: no constant to subtract
        once = c.structure_factor(7)
        first = c.structure_factor(7, accumulate=True)
        mean = c.structure_factor(7, accumulate=True)
    want = (np.abs(np.fft.fftn(f)) ** 2 / f.size).ravel()
    want[0] = 0.0
    # FP32 radix passes: 2^-24 each of at most 10 + 10 + 10 passes with a twiddle product,
    # a few roundings a pass, against the field's 2-norm
    eps = 2.0 ** -24 if prec == "fp32" else 2.0 ** -53
    scale = np.sqrt(want * (f ** 2).sum()) + 100 * eps * (f ** 2).sum()
    tol = 2 * 100 * eps * scale
    assert (np.abs(once - want) <= tol).all()
    assert np.array_equal(first, once)
    assert np.abs(mean - once).max() <= 2.0 ** -52 * once.max()
