"""Kernels of a chain (csrc/flb_kernels.cuh, pdl_wait) may start while the kernel
before them still writes what they read.  Their sources have to keep every load
behind the wait: inline PTX that loads is volatile, and no pointer that is only
read is __restrict__ (such loads count as invariant and may be moved ahead)."""
import glob
import os
import re

import pytest

CSRC = os.path.join(os.path.dirname(os.path.dirname(os.path.abspath(__file__))), "paper_1012_3632_gb300", "csrc")
FILES = sorted(glob.glob(os.path.join(CSRC, "*.cu")) + glob.glob(os.path.join(CSRC, "*.cuh")))


def _source(path):
    src = re.sub(r"/\*.*?\*/", "", open(path).read(), flags=re.S)
    return re.sub(r"//[^\n]*", "", src)


def _kernels():
    """(name, parameters, body) of every __global__ function."""
    for path in FILES:
        src = _source(path)
        for m in re.finditer(r"__global__\s+void(?:\s+__launch_bounds__\((?:[^()]|\([^()]*\))*\))?\s+(\w+)\(", src):
            brace = src.index("{", m.end())
            depth, end = 0, brace
            while True:
                depth += {"{": 1, "}": -1}.get(src[end], 0)
                if depth == 0:
                    break
                end += 1
            yield m.group(1), src[m.end():brace], src[brace:end]


def test_every_kernel_launched_in_a_chain_waits():
    kernels = {name: body for name, _, body in _kernels()}
    assert len(kernels) >= 40
    chained = set()
    for path in FILES:
        src = _source(path)
        chained |= {n for n in re.findall(r"launch_chain(?:_smem)?\(\s*(?:[^,;]*?\b)?(k_\w+)", src)}
    assert len(chained) >= 20
    for name in chained:
        assert "pdl_wait()" in kernels[name], name


@pytest.mark.parametrize("name", sorted({n for n, _, body in _kernels() if "pdl_wait()" in body}))
def test_pointers_that_a_waiting_kernel_reads_are_not_restrict(name):
    for n, params, body in _kernels():
        if n != name:
            continue
        for p in params.split(","):
            if "__restrict__" not in p:
                continue
            assert "const" not in p.split("*")[0].split(), p.strip()


@pytest.mark.parametrize("path", FILES, ids=os.path.basename)
def test_inline_ptx_that_touches_memory_is_volatile(path):
    for m in re.finditer(r"\basm\s*(volatile)?\s*\(\s*\"([a-z_]+)\.", _source(path)):
        if m.group(2) in ("ld", "st", "atom", "red", "prefetch", "griddepcontrol", "fence", "membar"):
            assert m.group(1), _source(path)[m.start():m.start() + 90]


def test_sums_of_other_blocks_are_read_after_the_warp_is_in_order():
    """Lane 0 acquires the other blocks' sums; only a __syncwarp orders that
    before the loads of the other lanes, which have to be loads that see them."""
    body = {name: body for name, _, body in _kernels()}["k_sum_steps"]
    after = body[body.index("atom.acq_rel"):]
    assert "__ldcg" not in after
    assert after.index("__shfl_sync") < after.index("__syncwarp()") < after.index("ld_relaxed(")
