"""The D2Q9 force-model step of FP32 and BF16 storage (k_step_gather2, site
pairs, tiles of 32 x 8 with a 2-site halo) at the edges of its tiles, with odd
rows and on lattices smaller than the halo."""
import numpy as np
import pytest

import oracle
from paper_1012_3632_gb300 import Context, inputs, landau_free_energy

pytestmark = pytest.mark.gpu

EXCESS = dict(A=-0.01, B=0.1, rho_c=1.0, kappa=0.02)
TOTAL = landau_free_energy(1.0, 0.5, 0.1, 0.08)
TOL = {"fp32": 2e-5, "bf16": 2e-3}  # the parity tolerances of the storage types

DIMS = [(1, 1), (2, 1), (3, 2), (5, 1), (30, 7), (31, 8), (32, 8), (33, 9), (34, 6), (63, 10), (64, 16), (66, 3),
        (127, 2), (130, 17)]


@pytest.mark.parametrize("fe", [EXCESS, TOTAL], ids=["excess", "total"])
@pytest.mark.parametrize("dims", DIMS)
@pytest.mark.parametrize("prec", ["fp32", "bf16"])
def test_pairs_against_the_oracle(dims, prec, fe):
    kw = dict(kT=1e-6, omega_shear=1.1, omega_bulk=0.9, omega_ghost=1.3, seed=21)
    rho = inputs.uniform_density((*dims, 1), seed=6)
    with Context(9, dims, precision=prec, free_energy=fe, **kw) as c:
        c.init(rho=rho)
        c.step(6)
        got = c.get_populations()
    p = oracle.Params(Q=9, dims=(*dims, 1), nonideal=True, **fe, **kw)
    want = oracle.run(p, oracle.init(p, rho=rho), 0, 6)
    assert np.abs(got - want).max() <= TOL[prec]
