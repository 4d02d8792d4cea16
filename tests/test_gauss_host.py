"""The fixed-point Gaussian noise of csrc/gauss.cuh on the host against
extended precision: random words, words at the ends of the uniforms' range
(u next to 0 and to 1), next to the octave and table edges of the logarithm
and next to the axes and diagonals of the angle."""
import ctypes
import os
import shutil
import subprocess

import numpy as np
import pytest

HERE = os.path.dirname(os.path.abspath(__file__))


@pytest.fixture(scope="module")
def lib(tmp_path_factory):
    nvcc = shutil.which("nvcc") or "/usr/local/cuda/bin/nvcc"
    if not os.path.exists(nvcc):
        pytest.skip("nvcc not available")
    if np.finfo(np.longdouble).nmant < 63:
        pytest.skip("no extended precision")
    out = str(tmp_path_factory.mktemp("gauss") / "libgauss.so")
    subprocess.run([nvcc, "-O2", "-std=c++17", "-shared", "-Xcompiler", "-fPIC", "-o", out,
                    os.path.join(HERE, "gauss_harness.cu")], check=True, capture_output=True)
    return ctypes.CDLL(out)


def _words(kind, n, seed):
    g = np.random.default_rng(seed)
    w = g.integers(0, 2 ** 64, (n, 2), dtype=np.uint64)
    near = g.integers(0, 2 ** 20, n, dtype=np.uint64) >> g.integers(0, 20, n, dtype=np.uint64)
    sgn = g.integers(0, 2, n, dtype=np.uint64)
    if kind == "small u":
        w[:, 0] >>= g.integers(0, 64, n, dtype=np.uint64)
    elif kind == "u next to 1":
        w[:, 0] = ~(w[:, 0] >> g.integers(0, 64, n, dtype=np.uint64))
    elif kind == "octaves":
        w[:, 0] = (np.uint64(1) << g.integers(12, 64, n, dtype=np.uint64)) + (near << np.uint64(12)) * (1 - 2 * sgn)
    elif kind == "log table":
        w[:, 0] = (g.integers(512, 1024, n, dtype=np.uint64) << np.uint64(54)) + (near << np.uint64(12)) * (1 - 2 * sgn)
    elif kind == "axes":
        w[:, 1] = (g.integers(0, 8, n, dtype=np.uint64) << np.uint64(61)) + (near << np.uint64(12)) * (1 - 2 * sgn)
    elif kind == "angle table":
        w[:, 1] = (g.integers(0, 1024, n, dtype=np.uint64) << np.uint64(54)) + (near << np.uint64(12)) * (1 - 2 * sgn)
    return np.ascontiguousarray(w)


@pytest.mark.parametrize("kind", ["random", "small u", "u next to 1", "octaves", "log table", "axes", "angle table"])
def test_pairs_against_extended_precision(lib, kind):
    n = 20000
    w = _words(kind, n, 5)
    z = np.zeros((n, 2))
    lib.gauss_pairs_host(w.ctypes.data_as(ctypes.c_void_p), n, z.ctypes.data_as(ctypes.c_void_p))
    u = ((w >> np.uint64(12)).astype(np.longdouble) + np.longdouble(0.5)) * np.longdouble(2.0) ** -52
    rad = np.sqrt(-np.log(u[:, 0]))
    # 2 pi u from the nearest multiple of a quarter, so that the argument is exact next to the axes
    q = np.round(4 * u[:, 1])
    d = (u[:, 1] - q / 4) * 2 * np.arctan2(np.longdouble(0), np.longdouble(-1))
    q = q.astype(int) % 4
    c, s = np.cos(d), np.sin(d)
    cs = np.choose(q, [c, -s, -c, s])
    sn = np.choose(q, [s, c, -s, -c])
    # the radius to 2^-52 relative, the angle to 2^-59, one rounding of the product: 1.5 + 1/64 units of 2^-52
    err = np.maximum(np.abs(z[:, 0] - rad * cs), np.abs(z[:, 1] - rad * sn))
    assert float(np.max(err / rad)) < 1.6 * 2.0 ** -52
