"""Host side of the library over a fake CUDA runtime (tests/fake_cudart.c): device
memory that runs out between the allocations of one call."""
import os
import subprocess
import sys

import pytest

HERE = os.path.dirname(os.path.abspath(__file__))
ROOT = os.path.dirname(HERE)


@pytest.fixture(scope="module")
def fake(tmp_path_factory):
    from paper_1012_3632_gb300 import build

    build.build()
    so = str(tmp_path_factory.mktemp("fake") / "libfake.so")
    subprocess.run(["gcc", "-shared", "-fPIC", "-O1", os.path.join(HERE, "fake_cudart.c"), "-o", so], check=True)
    return so


def _run(fake, body):
    """Run `body` in a process of its own with the fake runtime loaded first."""
    code = ("import ctypes, sys\n"
            "from paper_1012_3632_gb300 import flb\n"
            "from paper_1012_3632_gb300.flb import FLBError, FLB_ENOMEM, Batch, Context\n"
            f"fake = ctypes.CDLL({fake!r})\n"
            "num = lambda name: ctypes.c_int.in_dll(fake, name)\n") + body
    env = dict(os.environ, LD_PRELOAD=fake, PYTHONPATH=ROOT)
    r = subprocess.run([sys.executable, "-c", code], env=env, capture_output=True, text=True, timeout=300)
    assert r.returncode == 0, r.stdout + r.stderr


BATCH = """
b = Batch([(4, 4, 4), (3, 5, 2)], [1.0, 1.1], [1e-5, 1e-5], [1, 2])
have = num("fake_allocs").value
num("fake_fail_from").value = have + %d          # the n-th allocation of the call fails
before = num("fake_launches").value
for _ in range(2):                                # and fails again: nothing may be launched without it
    try:
        %s
    except FLBError as e:
        assert e.code == FLB_ENOMEM, e
    else:
        sys.exit("the call went on without its buffer")
assert num("fake_launches").value == before
num("fake_fail_from").value = 0                   # memory is there again
%s
assert num("fake_launches").value > before
"""


@pytest.mark.parametrize("nth", [1, 2])
def test_batch_mode_variance_asks_again_for_what_it_did_not_get(fake, nth):
    call = "b.mode_variance()"
    _run(fake, BATCH % (nth, call, call))


@pytest.mark.parametrize("nth", [1, 2, 3, 4])
def test_batch_structure_factor_asks_again_for_what_it_did_not_get(fake, nth):
    call = "b.structure_factor(1, 0, accumulate=True)"
    _run(fake, BATCH % (nth, call, call))


def test_batch_keeps_its_work_list_when_a_new_one_cannot_be_had(fake):
    _run(fake, """
b = Batch([(4, 4, 4), (3, 5, 2)], [1.0, 1.1], [1e-5, 1e-5], [1, 2])
num("fake_fail_from").value = num("fake_allocs").value + 1
try:
    b.autotune()
except FLBError as e:
    assert e.code == FLB_ENOMEM, e
else:
    sys.exit("tuned without memory")
num("fake_keep_arg").value = 1                    # the work list of the batch step
b.step(1)
assert ctypes.c_void_p.in_dll(fake, "fake_arg").value, "step over no work list"
""")


@pytest.mark.parametrize("field,offset,side", [(2, -1, "before its start"), (2, 256, "after its end"),
                                               (3, -1, "before its start"), (3, 256, "after its end")])
def test_fields_of_a_step_in_passes_have_guard_zones_of_their_own(fake, field, offset, side):
    """Density and chemical potential (64 sites, 256 bytes each; allocations 2 and 3,
    behind the population buffers): a write past one is not lost in the other."""
    _run(fake, f"""
c = Context(19, (4, 4, 4), 1.0, kT=1e-6, free_energy=dict(A=-0.01, B=0.1, rho_c=1.0, kappa=0.02), guard=True)
c.check_guards()
base = (ctypes.c_void_p * 256).in_dll(fake, "fake_ptr")[{field}]
ctypes.memset(base + 65536 + {offset}, 0, 1)
try:
    c.check_guards()
except FLBError as e:
    assert e.code == -7 and {side!r} in str(e), e   # FLB_EBOUNDS
    assert {"density field" if field == 2 else "chemical potential field"!r} in str(e), e
else:
    sys.exit("the write was not seen")
""")
