"""Mass deviation and momentum (k_cons_partials) against sums in exact
arithmetic, and their batches of several states in one column sum."""
import math

import numpy as np
import pytest

import oracle
from paper_1012_3632_gb300 import Context, inputs

pytestmark = pytest.mark.gpu


# around a block of 256 sites, below and above the largest grid (456 blocks)
@pytest.mark.parametrize("Q,dims", [(9, (1, 1)), (9, (51, 5)), (9, (16, 16)), (9, (257, 1)), (19, (3, 5, 17)),
                                    (19, (16, 4, 4)), (19, (48, 48, 51)), (19, (61, 53, 37))])
@pytest.mark.parametrize("prec", ["fp64", "fp32", "bf16"])
def test_totals_are_those_of_the_populations(Q, dims, prec):
    dims3 = (*dims, 1)[:3]
    lat = oracle.lattice(Q)
    f = inputs.random_populations(Q, dims3)
    with Context(Q, dims, 1.0, precision=prec) as c:
        c.set_populations(f)
        got = c.conservation()
        g = c.get_populations().reshape(Q, -1) - lat.w[:, None]  # the stored values, rho0 = 1
    if prec != "fp64":
        g = g.astype(np.float32).astype(np.float64)  # w + g was rounded to FP64 on its way out
    V = g.shape[1]
    for k in range(4):
        c_k = np.ones(Q) if k == 0 else (lat.c[:, k - 1] if k - 1 < lat.c.shape[1] else np.zeros(Q))
        want = math.fsum((c_k[:, None] * g).ravel()) + (V if k == 0 else 0.0)
        # (hi, lo) pairs: 2^-46 of the magnitudes summed; FP64 sums of V terms in
        # blocks of fewer than 2^10 per thread and a tree: 2^-42; get_populations
        # rounds every FP64 value to 2^-53
        scale = np.abs(c_k[:, None] * g).sum()
        assert abs(got[k] - want) <= 2.0 ** -42 * scale + 2.0 ** -50 * V


@pytest.mark.parametrize("Q,dims,prec,n", [(19, (8, 6, 5), "fp32", 40), (19, (33, 20, 31), "bf16", 21),
                                           (9, (40, 30), "fp64", 19), (9, (1, 1), "fp32", 5)])
def test_batches_equal_single_reductions(Q, dims, prec, n):
    kw = dict(kT=1e-5, seed=8, precision=prec)
    want = []
    with Context(Q, dims, 1.0, **kw) as a:
        for _ in range(n):
            want.append(a.conservation())
            a.step(1)
        fa = a.get_populations()
    with Context(Q, dims, 1.0, **kw) as b:
        got = np.asarray(b.step_sums(n))
        fb = b.get_populations()
    assert np.array_equal(got, np.asarray(want))
    assert np.array_equal(fa, fb)
