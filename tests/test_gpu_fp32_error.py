"""FP32 rounding of the kernels that work on two sites at once: no larger than that
of one site per thread.  The bounds are the errors against 64 bits that the one-site
kernels had on these states."""
import math

import numpy as np
import pytest

pytestmark = pytest.mark.gpu
torch = pytest.importorskip("torch")
from paper_1012_3632_gb300 import Context  # noqa: E402

LANDAU = dict(A=-0.025, B=0.4, rho_c=0.75, kappa=0.08, total=True)
EXCESS = dict(A=-0.01, B=0.1, rho_c=1.0, kappa=0.02)
W9 = torch.tensor([4 / 9] + [1 / 9] * 4 + [1 / 36] * 4, dtype=torch.float64)
W19 = torch.tensor([1 / 3] + [1 / 18] * 6 + [1 / 36] * 12, dtype=torch.float64)


def _stripe(X, Y, seed):
    """A liquid stripe between two tanh interfaces, deviations from rho0 = 1 in FP32."""
    gap, width = 0.5, math.sqrt(8 * 0.08 / 0.1) / 0.5
    y = torch.arange(Y, dtype=torch.float64) - 4 * np.random.default_rng(seed).random()
    p = torch.tanh(2 * (y - 0.25 * Y) / width) - torch.tanh(2 * (y - 0.75 * Y) / width)
    drho = (0.75 - gap / 2 + gap / 2 * p - 1.0)[:, None].expand(Y, X).reshape(-1)
    return (W9[:, None] * drho).float()


def _after(Q, dims, fe, prec, g, seed, n):
    dt = torch.float64 if prec == "fp64" else torch.float32
    g = g.to(dt).cuda()
    with Context(Q, dims, 1.0, 1.0, 1.0, kT=1e-7, free_energy=fe, seed=seed, precision=prec) as c:
        c.set_state_device(g.data_ptr())
        c.step(n)
        c.get_state_device(g.data_ptr())
        c.synchronize()
    return g.double().cpu()


@pytest.mark.parametrize("dims,n,bound", [((256, 96), 20, 1.06e-7), ((225, 135), 12, 1.005e-7)])
def test_modified_equilibrium_step(dims, n, bound):
    fe = dict(LANDAU, model=1)
    err = []
    for seed in range(1, 7):
        g = _stripe(*dims, seed)
        a, b = (_after(9, dims, fe, p, g, seed, n) for p in ("fp32", "fp64"))
        err.append(((a - b).norm() / b.norm()).item())
    # the mean over the seeds varies by half a percent
    assert np.mean(err) <= 1.01 * bound


@pytest.mark.parametrize("dims", [(24, 20, 16), (25, 19, 15)])
@pytest.mark.parametrize("fe,offset,bound", [(EXCESS, 0.0, 7.0e-8), (dict(LANDAU), -0.25, 6.8e-8), (None, 0.0, 6.56e-8)],
                         ids=["excess", "total", "ideal"])
def test_adjoint_step(dims, fe, offset, bound):
    V = int(np.prod(dims))
    z, y, x = torch.meshgrid(*[2 * math.pi * torch.arange(m, dtype=torch.float64) / m for m in reversed(dims)],
                             indexing="ij")
    err = []
    for seed in range(12):
        gen = torch.Generator().manual_seed(seed)
        drho = offset + 0.02 * torch.rand(V, generator=gen, dtype=torch.float64) - 0.01
        g = (W19[:, None] * (drho + 1e-4 * torch.randn((19, V), generator=gen, dtype=torch.float64))).float()
        ph = 2 * math.pi * torch.rand(2, generator=gen, dtype=torch.float64)
        smooth = (torch.sin(x + ph[0]) + torch.cos(y + ph[1]) * torch.sin(z)).reshape(-1)
        lam = (smooth + 0.2 * torch.randn((19, V), generator=gen, dtype=torch.float64)).float()
        out = []
        for prec, dt in (("fp32", torch.float32), ("fp64", torch.float64)):
            a, b = g.to(dt).cuda(), lam.to(dt).cuda()
            res, grad = torch.empty_like(b), torch.zeros(6, dtype=torch.float64, device="cuda")
            with Context(19, dims, 1.1, 0.9, 1.2, kT=1e-6, free_energy=fe, seed=seed, precision=prec) as c:
                c.adjoint_step(a.data_ptr(), 0, b.data_ptr(), res.data_ptr(), grad.data_ptr())
                c.synchronize()
            out.append(res.double().cpu())
        err.append(((out[0] - out[1]).norm() / out[1].norm()).item())
    assert np.mean(err) <= 1.01 * bound
