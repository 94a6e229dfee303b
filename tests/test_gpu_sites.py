"""The step kernels of one site per lane (k_sites): FP64 D3Q19 ideal and force
model, D2Q9 ideal gas, at the sizes where their tiling and the change from 32
to 128 sites per block can go wrong, against the oracle."""
import numpy as np
import pytest

import oracle
from paper_1012_3632_gb300 import Context, inputs, landau_free_energy

pytestmark = pytest.mark.gpu

EXCESS = dict(A=-0.01, B=0.1, rho_c=1.0, kappa=0.02)
TOTAL = landau_free_energy(1.0, 0.5, 0.1, 0.08)
TOL = {"fp64": 1e-12, "fp32": 2e-5}  # the parity tolerances of the storage types

# rows of 4 to 32 lanes, single rows and planes, ragged last tiles; 24576 (D3Q19)
# and 65536 sites (D2Q9) are the last sizes stepped 32 sites per block
D3 = [(1, 1, 1), (5, 1, 1), (1, 9, 2), (3, 4, 33), (33, 5, 3), (32, 32, 24), (32, 32, 25), (29, 29, 29)]
D2 = [(1, 1, 1), (31, 2, 1), (33, 17, 1), (256, 256, 1), (256, 257, 1), (261, 275, 1)]


@pytest.mark.parametrize("prec,Q,dims,fe", [("fp64", 19, d, fe) for d in D3 for fe in (None, EXCESS, TOTAL)] +
                         [(p, 9, d, None) for d in D2 for p in ("fp64", "fp32")] +
                         [("fp32", 19, (27, 5, 4), None)])
@pytest.mark.parametrize("kT", [1e-5, 0.0])
def test_sites_against_the_oracle(prec, Q, dims, fe, kT):
    kw = dict(kT=kT, omega_shear=1.1, omega_bulk=0.9, omega_ghost=1.3, seed=31)
    rho = inputs.uniform_density(dims, seed=9)
    with Context(Q, dims, precision=prec, free_energy=fe, **kw) as c:
        c.init(rho=rho)
        c.step(3)
        got = c.get_populations()
    p = oracle.Params(Q=Q, dims=dims, nonideal=bool(fe), **(fe or {}), **kw)
    want = oracle.run(p, oracle.init(p, rho=rho), 0, 3)
    assert np.abs(got - want).max() <= TOL[prec]
