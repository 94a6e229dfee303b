"""Build the CUDA library ``libflb.so`` in-tree with nvcc for sm_103a (GB300).

Each translation unit under ``csrc/`` is compiled in parallel, then linked into
one shared library next to this file.  No CMake, no torch extension machinery:
the library exposes a plain C ABI (``include/flb.h``).
"""
from __future__ import annotations

import concurrent.futures as cf
import os
import shutil
import subprocess
import sys

HERE = os.path.dirname(os.path.abspath(__file__))
CSRC = os.path.join(HERE, "csrc")
BUILD = os.path.join(HERE, "_build")
LIB = os.path.join(HERE, "libflb.so")
SOURCES = ["flb_api.cu", "flb_fp64.cu", "flb_fp32.cu", "flb_bf16.cu", "flb_fft.cu", "flb_sums.cu", "flb_noalloc.cu", "flb_batch.cu", "flb_adjoint.cu", "flb_capillary.cu", "flb_swift.cu"]
# compiled once per part (FLB_REG_PART), a share of the transform lengths each
REG_SOURCE, REG_PARTS = "flb_fft_reg.cu", 12
ARCH = ["-gencode", "arch=compute_103a,code=sm_103a"]
# --no-compress: nvcc compresses a translation unit's device code once it is large, and
# the driver unpacks it when the first of its kernels is used (the transforms: 14 ms
# against 2)
FLAGS = ["-O3", "-std=c++17", "-lineinfo", "--no-compress", "-Xcompiler", "-fPIC", "-Xcompiler", "-O2"]


def nvcc() -> str:
    for cand in (os.environ.get("NVCC"), shutil.which("nvcc"), "/usr/local/cuda/bin/nvcc"):
        if cand and os.path.exists(cand):
            return cand
    raise RuntimeError("nvcc not found: the CUDA toolkit is required to build libflb.so")


def _deps():
    return [os.path.join(CSRC, f) for f in os.listdir(CSRC)] + [os.path.join(HERE, "..", "include", "flb.h")]


def up_to_date() -> bool:
    if not os.path.exists(LIB):
        return False
    t = os.path.getmtime(LIB)
    return all(os.path.getmtime(d) <= t for d in _deps())


def build(force: bool = False, verbose: bool = False, ptxas_info: bool = False) -> str:
    if not force and up_to_date():
        return LIB
    os.makedirs(BUILD, exist_ok=True)
    cc = nvcc()
    extra = ["-Xptxas", "-v"] if ptxas_info else []
    extra += os.environ.get("FLB_NVCC_FLAGS", "").split()

    units = [(f"{os.path.splitext(REG_SOURCE)[0]}{k}.o", REG_SOURCE, [f"-DFLB_REG_PART={k}"]) for k in range(REG_PARTS)]
    units += [(os.path.splitext(src)[0] + ".o", src, []) for src in SOURCES]

    def compile_one(unit):
        name, src, defs = unit
        obj = os.path.join(BUILD, name)
        cmd = [cc, *ARCH, *FLAGS, *extra, *defs, "-c", os.path.join(CSRC, src), "-o", obj]
        r = subprocess.run(cmd, capture_output=True, text=True)
        if r.returncode != 0:
            raise RuntimeError(f"nvcc failed for {src}:\n{r.stderr}")
        return obj, r.stderr

    with cf.ThreadPoolExecutor(max_workers=max(len(SOURCES), os.cpu_count() or 1)) as ex:
        results = list(ex.map(compile_one, units))
    if verbose or ptxas_info:
        for _, err in results:
            if err:
                sys.stderr.write(err)
    tmp = LIB + f".tmp{os.getpid()}"
    cmd = [cc, *ARCH, "-shared", "-o", tmp] + [o for o, _ in results] + ["-lcudart"]
    r = subprocess.run(cmd, capture_output=True, text=True)
    if r.returncode != 0:
        raise RuntimeError(f"link failed:\n{r.stderr}")
    os.replace(tmp, LIB)
    return LIB


if __name__ == "__main__":
    build(force="--force" in sys.argv, verbose=True, ptxas_info="--ptxas" in sys.argv)
    print(LIB)
