"""Which lengths the register transforms (csrc/flb_fft_reg.cuh) take: a rule on the
length, three to six of the radices 4, 2, 3, 5 and at most 1024 elements."""
import ctypes

import pytest


def _radices(n):
    out = []
    for r in (4, 2, 3, 5):
        while n % r == 0:
            out.append(r)
            n //= r
    return out if n == 1 else []


@pytest.fixture(scope="module")
def both_have_kernels():
    from paper_1012_3632_gb300 import build, lib

    build.build()
    fn = lib()._ZN3flb19swift_noise_lengthsEii  # flb::swift_noise_lengths(int, int)
    fn.restype, fn.argtypes = ctypes.c_bool, [ctypes.c_int, ctypes.c_int]
    return fn


def test_every_length_of_the_rule_and_no_other(both_have_kernels):
    want = [n for n in range(1, 1300) if n <= 1024 and 3 <= len(_radices(n)) <= 6]
    assert len(want) == 73
    assert [n for n in range(1, 1300) if both_have_kernels(n, n)] == want
    assert not both_have_kernels(0, 64) and not both_have_kernels(64, -4) and not both_have_kernels(64, 1 << 30)
