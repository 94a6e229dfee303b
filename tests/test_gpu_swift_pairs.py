"""The modified-equilibrium step in site pairs (k_step_swift2): odd and even rows
at the edges of its tiles; FP32 storage against the oracle, BF16 storage against
the FP32 step of the same state."""
import numpy as np
import pytest

import oracle
from paper_1012_3632_gb300 import Context, inputs, landau_free_energy

pytestmark = pytest.mark.gpu
torch = pytest.importorskip("torch")

FE = landau_free_energy(1.0, 0.5, 0.1, 0.08)
DIMS = [(3, 2), (6, 3), (15, 8), (31, 5), (32, 9), (34, 4), (63, 6), (66, 3), (130, 5)]
KW = dict(kT=1e-6, omega_shear=1.1, omega_bulk=0.9, omega_ghost=1.3, seed=8)


@pytest.mark.parametrize("dims", DIMS)
def test_pairs_against_the_oracle(dims):
    rho = inputs.uniform_density((*dims, 1), rho_c=1.0, amp=0.02, seed=2)
    with Context(9, dims, precision="fp32", free_energy=dict(FE, model=1), **KW) as c:
        c.init(rho=rho)
        c.step(6)
        got = c.get_populations()
    p = oracle.Params(Q=9, dims=(*dims, 1), nonideal=True, A=FE["A"], B=FE["B"], rho_c=FE["rho_c"],
                      kappa=FE["kappa"], total=True, model=1, **KW)
    want = oracle.run(p, oracle.init(p, rho=rho), 0, 6)
    assert np.abs(got - want).max() <= 2e-5  # the parity tolerance of FP32 storage


@pytest.mark.parametrize("dims", DIMS)
def test_bf16_storage_is_the_rounded_fp32_step(dims):
    V = dims[0] * dims[1]
    gen = torch.Generator().manual_seed(V)
    w = torch.tensor([4 / 9] + [1 / 9] * 4 + [1 / 36] * 4)[:, None]
    g = (w * 0.05 * torch.randn((9, V), generator=gen)).bfloat16().cuda()
    out = {}
    for prec, dt in (("fp32", torch.float32), ("bf16", torch.bfloat16)):
        start, got = g.to(dt), torch.empty_like(g, dtype=dt)
        with Context(9, dims, precision=prec, free_energy=dict(FE, model=1), **KW) as c:
            c.set_state_device(start.data_ptr())
            c.step(1)
            c.get_state_device(got.data_ptr())
            c.synchronize()
        out[prec] = got
    assert torch.equal(out["fp32"].bfloat16(), out["bf16"])
