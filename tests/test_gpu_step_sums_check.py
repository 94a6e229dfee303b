"""flb_step_sums with check_every: the check of the totals after a step shares
its buffer of partial sums with the sums of several steps that wait to be added
up, and must neither change them nor keep them back when the run diverges."""
import numpy as np
import pytest
import torch

from paper_1012_3632_gb300 import Context, inputs
from paper_1012_3632_gb300.flb import FLB_EDIVERGED, FLBError

pytestmark = pytest.mark.gpu

EXCESS = dict(A=-0.01, B=0.1, rho_c=1.0, kappa=0.02)
TOTAL = dict(A=-0.025, B=0.4, rho_c=0.75, kappa=0.08, total=True)

# reductions before the step; rows of the density pass, X % 4 == 0 (16 states wait)
# and X % 4 == 2 (4 and 7 wait, their rows begin inside what a check writes)
CASES = [(9, (20, 12), None, "fp64"), (19, (8, 6, 5), None, "fp32"), (19, (33, 20, 31), None, "bf16"),
         (19, (12, 10, 9), TOTAL, "fp32"), (19, (9, 7, 5), EXCESS, "fp32"), (19, (16, 8, 6), EXCESS, "fp64"),
         (19, (16, 8, 6), EXCESS, "bf16"), (19, (62, 64, 64), EXCESS, "fp32"), (19, (50, 50, 50), EXCESS, "bf16")]


def _context(Q, dims, fe, prec, check_every):
    c = Context(Q, dims, 1.1, kT=1e-6, free_energy=fe, seed=3, precision=prec, check_every=check_every)
    c.init(rho=inputs.uniform_density((*dims, 1)[:3], seed=4))
    return c


@pytest.mark.parametrize("Q,dims,fe,prec", CASES)
@pytest.mark.parametrize("every", [1, 3])
def test_sums_are_those_without_checks(Q, dims, fe, prec, every):
    n = 10
    with _context(Q, dims, fe, prec, 0) as a:
        want = a.step_sums(n)
        fa = a.get_populations()
    pinned = torch.empty((n, 4), dtype=torch.float64, pin_memory=True).numpy()
    with _context(Q, dims, fe, prec, every) as b:
        got = b.step_sums(n)  # pageable memory
        fb = b.get_populations()
    with _context(Q, dims, fe, prec, every) as d:
        d.step_sums(n, out=pinned)  # page-locked: written in place
    assert np.array_equal(got, want)
    assert np.array_equal(pinned, want)
    assert np.array_equal(fa, fb)


@pytest.mark.parametrize("Q,dims,fe,prec", [c for c in CASES if c[0] == 19])
@pytest.mark.parametrize("every", [1, 3])
def test_sums_up_to_the_failing_check_are_delivered(Q, dims, fe, prec, every):
    """A population near the largest float: the state it belongs to has finite
    sums, the step from it overflows, and the first check stops the run."""
    n, unset = 8, -7.0
    pinned = torch.full((n, 4), unset, dtype=torch.float64, pin_memory=True).numpy()
    with _context(Q, dims, fe, prec, 0) as a:
        f = a.get_populations()
        f[1, 0] = 3e38 if prec != "fp64" else 1.5e308
        a.set_populations(f)
        first = a.step_sums(1)[0]
    with _context(Q, dims, fe, prec, every) as b:
        b.set_populations(f)
        with pytest.raises(FLBError) as e:
            b.step_sums(n, out=pinned)
        assert e.value.code == FLB_EDIVERGED
        assert b.step_count == every
    assert np.array_equal(pinned[0], first, equal_nan=True)
    assert not (pinned[:every] == unset).any()
    assert (pinned[every:] == unset).all()
