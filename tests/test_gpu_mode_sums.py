"""Mode variances (k_mode_sums): rows that 32 does not divide, one warp per
block and eight, one block and many, several lattices in one launch, against
the variance of the mode field itself."""
import numpy as np
import pytest
import torch

from paper_1012_3632_gb300 import MODE_VAR, MODES, Batch, Context

pytestmark = pytest.mark.gpu

# per warp: 32 squares (one rounding each) added in a tree of depth 5
TOL = {"fp64": 6 * 2.0 ** -53, "fp32": 6 * 2.0 ** -24, "bf16": 6 * 2.0 ** -24}


def _check(var, m, prec):
    want = m.var(axis=1)
    # variance = mean square - mean^2: both carry the relative error of the sums; 2^-50 for the FP64 part
    bound = 2 * (TOL[prec] + 2.0 ** -50) * (m ** 2).mean(axis=1)
    assert (np.abs(var - want) <= bound).all(), np.abs(var - want) / bound


@pytest.mark.parametrize("prec", ["fp64", "fp32", "bf16"])
@pytest.mark.parametrize("Q,dims", [(9, (2, 3, 1)), (9, (33, 36, 1)), (9, (32, 1216, 1)), (9, (95, 700, 1)),
                                    (19, (1, 2, 3)), (19, (31, 9, 4)), (19, (33, 20, 30)), (19, (64, 50, 40)),
                                    (19, (100, 70, 60))])
def test_mode_variance(Q, dims, prec):
    with Context(Q, dims, 1.1, kT=1e-4, seed=3, precision=prec) as c:
        c.init(thermal=True)
        c.step(2)
        m = c.moments(MODES).copy()
        # the sums are of the density deviation; rho - 1 would lose an FP64 state's
        # last digits, which the state itself has
        if prec == "fp64":
            g = torch.empty((Q, c.V), dtype=torch.float64, device="cuda")
            c.get_state_device(g.data_ptr())
            m[0] = g.sum(0).cpu().numpy()
        else:
            m[0] -= 1.0
        _check(c.moments(MODE_VAR), m, prec)


def test_mode_variance_of_a_batch():
    dims = [(32, 32, 32), (48, 5, 7), (3, 2, 1), (96, 64, 40), (31, 33, 2)]
    kw = dict(kT=1e-4, seed=9)
    with Batch(dims, [1.1] * 5, [1e-4] * 5, [9] * 5) as b:
        b.init(thermal=True)
        b.step(3)
        var = b.mode_variance()
    for r, d in enumerate(dims):
        with Context(19, d, 1.1, replica=r, **kw) as c:
            c.init(thermal=True)
            c.step(3)
            m = c.moments(MODES).copy()
        m[0] -= 1.0
        _check(var[r], m, "fp32")
