"""D3Q19 steps on both sides of the block counts up to which a step draws its
noise before it waits for the step before (csrc/flb_prec.cuh): 64 x 64 x Z has
16 Z blocks of 256 sites, the lines lie at 1216 (ideal gas) and 912 (force model)."""
import numpy as np
import pytest

import oracle
from paper_1012_3632_gb300 import Context, inputs

pytestmark = pytest.mark.gpu

EXCESS = dict(A=-0.01, B=0.1, rho_c=1.0, kappa=0.02)
TOL = {"fp32": 2e-5, "bf16": 2e-3}  # the parity tolerances of the storage types


@pytest.mark.parametrize("fe,dims", [(None, (64, 64, 76)), (None, (64, 64, 78)), (EXCESS, (64, 64, 57)),
                                     (EXCESS, (64, 64, 58)), (None, (63, 5, 3)), (EXCESS, (31, 4, 3))])
@pytest.mark.parametrize("prec", ["fp32", "bf16"])
@pytest.mark.parametrize("kT", [1e-5, 0.0])
def test_steps_against_the_oracle(fe, dims, prec, kT):
    kw = dict(kT=kT, omega_shear=1.1, omega_bulk=0.9, omega_ghost=1.3, seed=5)
    rho = inputs.uniform_density(dims, seed=6)
    with Context(19, dims, precision=prec, free_energy=fe, **kw) as c:
        c.init(rho=rho)
        c.step(3)
        got = c.get_populations()
    p = oracle.Params(Q=19, dims=dims, nonideal=fe is not None, **(fe or {}), **kw)
    want = oracle.run(p, oracle.init(p, rho=rho), 0, 3)
    assert np.abs(got - want).max() <= TOL[prec]
