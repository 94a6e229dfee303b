"""The batch step where its blocks walk several tiles each (more than 12160
tiles of 256 sites): bitwise the single lattices where rows are even, within the
rounding of another order of operations where they are odd."""
import numpy as np
import pytest

from paper_1012_3632_gb300 import Batch, Context

pytestmark = pytest.mark.gpu


def test_blocks_that_walk_several_tiles():
    dims = [(128, 128, 128), (67, 33, 31), (128, 128, 64), (36, 20, 18)]
    seeds = [3, 4, 5, 6]
    with Batch(dims, [1.1] * 4, [1e-5] * 4, seeds) as b:
        b.init()
        b.step(5)  # graph replays of two steps and a direct launch
        got = [b.get_populations(r) for r in range(4)]
    for r, d in enumerate(dims):
        with Context(19, d, 1.1, kT=1e-5, seed=seeds[r], precision="fp32", replica=r) as c:
            c.init()
            c.step(5)
            want = c.get_populations()
        if d[0] % 2 == 0:
            assert np.array_equal(got[r], want), d
        else:
            assert np.abs(got[r] - want).max() <= 1e-6, d
