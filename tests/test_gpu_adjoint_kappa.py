"""The kappa gradient of one adjoint step in FP32 against FP64 on the same inputs,
for a fluid whose density is far from rho0: its rounding is that of the
differences between neighbours, not that of the offset."""
import pytest

pytestmark = pytest.mark.gpu
torch = pytest.importorskip("torch")
from paper_1012_3632_gb300 import Context  # noqa: E402

TOTAL = dict(A=-0.025, B=0.4, rho_c=0.75, kappa=0.08, total=True)
EXCESS = dict(A=-0.01, B=0.1, rho_c=1.0, kappa=0.02)
C9 = [(1, 0, 0), (0, 1, 0), (0, 0, 1), (1, 1, 0), (1, -1, 0), (1, 0, 1), (1, 0, -1), (0, 1, 1), (0, 1, -1)]
W9 = [1 / 18] * 3 + [1 / 36] * 6


def _kappa_gradient(dims, g, lam, fe, prec):
    dt = torch.float64 if prec == "fp64" else torch.float32
    g, lam = g.to(dt).cuda(), lam.to(dt).cuda()
    out, grad = torch.empty_like(lam), torch.zeros(6, dtype=torch.float64, device="cuda")
    with Context(19, dims, 1.1, 0.9, 1.2, kT=0.0, free_energy=fe, seed=6, precision=prec) as c:
        c.adjoint_step(g.data_ptr(), 0, lam.data_ptr(), out.data_ptr(), grad.data_ptr())
        torch.cuda.synchronize()
    return grad[3].item()


@pytest.mark.parametrize("fe", [EXCESS, TOTAL], ids=["excess", "total"])
@pytest.mark.parametrize("dims", [(20, 12, 10), (9, 7, 5), (2, 3, 1)])
@pytest.mark.parametrize("offset", [-0.5, 0.0, 0.25])
def test_rounding_is_that_of_the_differences(dims, offset, fe):
    X, Y, Z = dims
    V = X * Y * Z
    gen = torch.Generator().manual_seed(V)
    # all of the deviation in the rest population, in units of 2^-20: the density is
    # the same number in both precisions
    drho = offset + 2.0 ** -20 * torch.randint(0, 64, (V,), generator=gen).double()
    g = torch.zeros((19, V), dtype=torch.float64)
    g[0] = drho
    lam = torch.randn((19, V), generator=gen, dtype=torch.float64).float().double()
    got, want = (_kappa_gradient(dims, g, lam, fe, p) for p in ("fp32", "fp64"))
    # T = 3 sum_r sum_i w_i |rho_i - rho|.  |mubar| <= M = 3 sum_i w_i |c_i| rho |Fbar|
    # with |Fbar| <= 1.1 max|lam| at rest (3 times the first moments of w lam) and
    # sum_i w_i |c_i| = 1.  mubar carries at most 64 roundings of values up to M (sums of
    # 19 terms, the force, 18 neighbours), each of which meets lap rho (6 sum w |..| = 2 T
    # in all), the products and their sums 16 of values up to 2 M T.
    r = drho.reshape(Z, Y, X)
    T = 6 * sum(w * (torch.roll(r, (-c[2], -c[1], -c[0]), (0, 1, 2)) - r).abs().sum().item() for c, w in zip(C9, W9))
    M = 3 * 1.1 * lam.abs().max().item() * (1 + drho.max().item())
    assert abs(got - want) <= 2.0 ** -24 * M * T * (2 * 64 + 2 * 16)
