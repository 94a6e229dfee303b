"""The FP64 paths' Box-Muller in integer arithmetic (csrc/flb_normal64.cuh)
against numpy's long double (128 bits on the GPU's Arm host, 80 on x86):
random word pairs, the ends of the table intervals, quadrant boundaries and
words whose uniform is close to 0 and to 1."""
import ctypes
import os
import shutil
import subprocess

import numpy as np
import pytest

pytestmark = pytest.mark.gpu

HERE = os.path.dirname(os.path.abspath(__file__))


@pytest.fixture(scope="module")
def normals(tmp_path_factory):
    nvcc = shutil.which("nvcc") or "/usr/local/cuda/bin/nvcc"
    so = str(tmp_path_factory.mktemp("normals") / "libnormals64.so")
    subprocess.check_call([nvcc, "-gencode", "arch=compute_103a,code=sm_103a", "-O3", "-std=c++17", "-shared",
                           "-Xcompiler", "-fPIC", os.path.join(HERE, "normals64.cu"), "-o", so])
    lib = ctypes.CDLL(so)

    def call(words):
        w = np.ascontiguousarray(words, dtype=np.uint32)
        out, ref = np.empty((len(w), 2)), np.empty((len(w), 2))
        dp = ctypes.POINTER(ctypes.c_double)
        assert lib.normals64(w.ctypes.data_as(ctypes.POINTER(ctypes.c_uint32)), len(w), out.ctypes.data_as(dp),
                             ref.ctypes.data_as(dp)) == 0
        return out, ref

    return call


def _exact(words):
    ld = np.longdouble
    a, b = words[:, 0].astype(ld), words[:, 1].astype(ld)
    u0, u1 = (a + ld(0.5)) / ld(2) ** 32, (b + ld(0.5)) / ld(2) ** 32
    r = np.sqrt(ld(-2) * np.log(u0))
    # the angle from the nearest quarter turn, so that the argument of sin and cos is small and exact
    q = np.rint(u1 * 4)
    t = (u1 - q / 4) * (ld(2) * ld("3.14159265358979323846264338327950288"))
    s, c = np.sin(t), np.cos(t)
    q = q.astype(np.int64) & 3
    cs = np.select([q == 0, q == 1, q == 2, q == 3], [c, -s, -c, s])
    sn = np.select([q == 0, q == 1, q == 2, q == 3], [s, c, -s, -c])
    return np.stack([r * cs, r * sn], 1), r


def test_integer_normals(normals):
    rng = np.random.default_rng(12)
    rnd = rng.integers(0, 2 ** 32, (400000, 2), dtype=np.uint64)
    # word 0: both sides of the interval ends j / 256 of every octave, words next to 0 and to 2^32
    edge = [(1 << k) + (j << max(k - 8, 0)) + d for k in range(32) for j in range(256) for d in (-1, 0, 1)]
    edge += [2 ** 32 - 1 - (1 << k) + d for k in range(31) for d in (0, 1)] + [0, 1, 2, 2 ** 32 - 1, 2 ** 32 - 2]
    w0 = np.array([e % 2 ** 32 for e in edge], dtype=np.uint64)
    # word 1: both sides of the table angles and of the quadrants
    w1 = np.array([(j << 22) + d for j in range(1024) for d in (-1, 0, 1)], dtype=np.int64) % 2 ** 32
    words = np.concatenate([rnd, np.stack([w0, rng.integers(0, 2 ** 32, len(w0), dtype=np.uint64)], 1),
                            np.stack([rng.integers(0, 2 ** 32, len(w1), dtype=np.uint64), w1.astype(np.uint64)], 1)])
    got, lib = normals(words)
    want, r = _exact(words)
    err = np.abs((got - want) / r[:, None]).astype(np.float64)
    libe = np.abs((lib - want) / r[:, None]).astype(np.float64)
    # half an ulp of a result just below r (2^-53 r) and 2^-60 r of the fixed-point steps
    assert err.max() <= 2.0 ** -53 * (1 + 2.0 ** -6)
    # no further off than the library's functions
    assert np.sqrt((err ** 2).mean()) <= np.sqrt((libe ** 2).mean())
    assert err.max() <= libe.max()
