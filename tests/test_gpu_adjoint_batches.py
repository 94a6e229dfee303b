"""Adjoint segments at the edges of their batches of 8 steps and of the two-site
tiling of the FP32 collision (odd and even rows, unaligned arrays)."""
import pytest

pytestmark = pytest.mark.gpu
torch = pytest.importorskip("torch")
from paper_1012_3632_gb300 import Context  # noqa: E402

EXCESS = dict(A=-0.01, B=0.1, rho_c=1.0, kappa=0.02)
TOTAL = dict(A=-0.025, B=0.4, rho_c=0.75, kappa=0.08, total=True)
OMEGA = (1.1, 0.9, 1.2)


def _fields(dims, n):
    gen = torch.Generator().manual_seed(sum(dims) + n)
    V = dims[0] * dims[1] * dims[2]
    w = torch.tensor([1 / 3] + [1 / 18] * 6 + [1 / 36] * 12, dtype=torch.float64)[:, None]
    # FP32 values in both precisions
    g = (w * 0.05 * torch.randn((19, V), generator=gen, dtype=torch.float64)).float()
    return g, (1 + 0.1 * torch.randn((19, V), generator=gen, dtype=torch.float64)).float()


def _at(t, offset):
    """A copy of t on the device, `offset` elements behind a 256-byte boundary."""
    buf = torch.empty(t.numel() + offset, dtype=t.dtype, device="cuda")
    out = buf[offset:].view(t.shape)
    out.copy_(t)
    return out


def _segment(dims, n, fe, prec, offset=0):
    dt = torch.float64 if prec == "fp64" else torch.float32
    g, lam = (_at(t.to(dt), offset) for t in _fields(dims, n))
    states = _at(torch.zeros((n,) + tuple(g.shape), dtype=dt), offset)
    grad = torch.zeros(6, dtype=torch.float64, device="cuda")
    with Context(19, dims, *OMEGA, kT=1e-5, free_energy=fe, seed=6, precision=prec) as c:
        c.adjoint_segment(g.data_ptr(), 3, n, states.data_ptr(), lam.data_ptr(), grad.data_ptr())
        torch.cuda.synchronize()
    return lam.cpu(), grad.cpu(), states.cpu()


def _single_steps(dims, n, fe, prec):
    dt = torch.float64 if prec == "fp64" else torch.float32
    g, lam = (t.to(dt).cuda() for t in _fields(dims, n))
    grad = torch.zeros(6, dtype=torch.float64, device="cuda")
    with Context(19, dims, *OMEGA, kT=1e-5, free_energy=fe, seed=6, precision=prec) as c:
        c.set_state_device(g.data_ptr())
        c.step_count = 3
        st = [g.clone()]
        for _ in range(n - 1):
            c.step(1)
            st.append(torch.empty_like(g))
            c.get_state_device(st[-1].data_ptr())
        for k in reversed(range(n)):
            nxt = torch.empty_like(lam)
            c.adjoint_step(st[k].data_ptr(), 3 + k, lam.data_ptr(), nxt.data_ptr(), grad.data_ptr())
            lam = nxt
        torch.cuda.synchronize()
    return lam.cpu(), grad.cpu(), torch.stack(st).cpu()


@pytest.mark.parametrize("fe", [None, EXCESS, TOTAL], ids=["ideal", "excess", "total"])
@pytest.mark.parametrize("dims,n", [((7, 5, 3), 8), ((6, 5, 4), 9), ((8, 3, 5), 17), ((33, 4, 2), 1), ((2, 2, 2), 2)])
def test_segment_against_single_steps_and_fp64(dims, n, fe):
    lam, grad, states = _segment(dims, n, fe, "fp32")
    # the same arithmetic step by step, and from arrays that begin at an odd element
    for other in (_single_steps(dims, n, fe, "fp32"), _segment(dims, n, fe, "fp32", offset=1)):
        assert torch.equal(states, other[2]) and torch.equal(lam, other[0])
        assert torch.equal(grad, other[1])
    l64, g64, _ = _segment(dims, n, fe, "fp64")
    # A step back multiplies by matrices of 19 terms twice (moments, transpose): 40
    # roundings of values up to the largest one, doubled for the gradient terms.
    tol = 80 * n * 2.0 ** -24
    assert (lam.double() - l64).abs().max() <= tol * l64.abs().max()
    # A site left out or counted twice moves a sum by about 1 / V; the rounding of
    # its terms is bounded by tol relative to their magnitudes, which a cancelling
    # sum over V random terms undercuts by sqrt(V) or so: 1 % of the largest gradient.
    used = 6 if fe else 3
    assert torch.all(grad[used:] == 0)
    for part in (slice(0, 3), slice(3, 6))[: used // 3]:
        assert torch.allclose(grad[part], g64[part], rtol=1e-2, atol=1e-2 * g64[part].abs().max().item())


@pytest.mark.parametrize("n", [8, 9])
def test_fp64_batches(n):
    for a, b in zip(_segment((5, 4, 3), n, EXCESS, "fp64"), _single_steps((5, 4, 3), n, EXCESS, "fp64")):
        assert torch.equal(a, b)
