"""The D3Q19 force-model step of FP32 and BF16 storage: density, mu and
collision passes (csrc/flb_force.cuh) at the sizes where their tiling, row
loads and sums can go wrong.

Row lengths X % 4 == 0, X even and X odd take quad, pair and single loads; a
tile is a row of 4 to 32 threads; mu handles two planes per thread (odd Z);
the sums of up to 16 steps are formed by one launch, in several blocks per
step from 2048 warp rows on.
"""
import numpy as np
import pytest

import oracle
from paper_1012_3632_gb300 import Context, inputs, landau_free_energy

pytestmark = pytest.mark.gpu

EXCESS = dict(A=-0.01, B=0.1, rho_c=1.0, kappa=0.02)
TOTAL = landau_free_energy(1.0, 0.5, 0.1, 0.08)
TOL = {"fp32": 2e-5, "bf16": 2e-3}  # the parity tolerances of the storage types

# (X, Y, Z): every gather width against ragged tiles, single planes and rows
DIMS = [(1, 1, 1), (2, 1, 2), (3, 2, 1), (4, 1, 3), (5, 9, 4), (12, 3, 7), (18, 5, 3), (31, 4, 2), (33, 3, 3),
        (66, 3, 2), (68, 5, 5), (130, 2, 3), (129, 3, 1), (132, 1, 1)]


@pytest.mark.parametrize("fe", [EXCESS, TOTAL], ids=["excess", "total"])
@pytest.mark.parametrize("dims", DIMS)
@pytest.mark.parametrize("prec", ["fp32", "bf16"])
def test_passes_against_the_oracle(dims, prec, fe):
    kw = dict(kT=1e-6, omega_shear=1.1, omega_bulk=0.9, omega_ghost=1.3, seed=21)
    rho = inputs.uniform_density(dims, seed=6)
    with Context(19, dims, precision=prec, free_energy=fe, **kw) as c:
        c.init(rho=rho)
        c.step(6)
        got = c.get_populations()
    p = oracle.Params(Q=19, dims=dims, nonideal=True, **fe, **kw)
    want = oracle.run(p, oracle.init(p, rho=rho), 0, 6)
    assert np.abs(got - want).max() <= TOL[prec]


@pytest.mark.parametrize("dims,n", [((8, 4, 3), 40), ((33, 10, 6), 21), ((128, 96, 96), 7), ((130, 90, 97), 5)])
def test_sums_over_several_launches(dims, n):
    """More steps than one sum launch takes, and more warp rows than one block
    of it: the sums equal the reduction of each state, the steps are those of
    flb_step, and a second run repeats them bit for bit."""
    V = int(np.prod(dims))
    kw = dict(kT=1e-5, omega_shear=1.1, seed=8, precision="fp32", free_energy=EXCESS)
    rho = inputs.uniform_density(dims, seed=7)
    with Context(19, dims, **kw) as a:
        a.init(rho=rho)
        want = []
        for _ in range(n):
            want.append(a.conservation())
            a.step(1)
        fa = a.get_sites(np.arange(0, V, max(1, V // 997)))
    got = []
    for _ in range(2):
        with Context(19, dims, **kw) as b:
            b.init(rho=rho)
            got.append(b.step_sums(n))
            fb = b.get_sites(np.arange(0, V, max(1, V // 997)))
        assert np.array_equal(fa, fb)
    want = np.array(want)
    assert np.abs(got[0][:, 0] - want[:, 0]).max() <= 1e-12 * V + 1e-5
    # FP32 sums of a warp's 128 sites of |g| <= 1e-2: below 128 * 0.3 * 2^-24 each, V / 128 of them
    assert np.abs(got[0][:, 1:] - want[:, 1:]).max() <= 1e-5 + V * 0.3 * 2.0 ** -24 / 50
    assert np.array_equal(got[0], got[1])
