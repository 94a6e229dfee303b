"""Mode variances of lattices around the lines at which their sums are split
differently (csrc/flb_internal.h, mode_blocks): 608 groups of 32 sites fill 304
blocks of two warps, from 1216 groups on the blocks have eight warps."""
import pytest

from test_gpu_mode_sums import _check

import numpy as np
import torch
from paper_1012_3632_gb300 import MODE_VAR, MODES, Context

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("prec", ["fp64", "fp32", "bf16"])
@pytest.mark.parametrize("Q,dims", [(19, (3, 1, 1)), (19, (32, 1, 607)), (19, (31, 32, 19)), (19, (33, 3, 101)),
                                    (19, (32, 405, 3)), (19, (20, 64, 19)), (19, (32, 1217, 1)), (9, (40, 303, 1)),
                                    (9, (40, 608, 1))])
def test_mode_variance(Q, dims, prec):
    with Context(Q, dims, 1.1, kT=1e-4, seed=3, precision=prec) as c:
        c.init(thermal=True)
        c.step(1)
        m = c.moments(MODES).copy()
        if prec == "fp64":
            g = torch.empty((Q, c.V), dtype=torch.float64, device="cuda")
            c.get_state_device(g.data_ptr())
            m[0] = g.sum(0).cpu().numpy()
        else:
            m[0] -= 1.0
        _check(c.moments(MODE_VAR), m, prec)
        assert np.isfinite(m).all()
