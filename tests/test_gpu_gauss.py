"""The fixed-point Gaussian pairs of csrc/gauss.cuh on the device (which takes
the root's starting value from rsqrtf) against extended precision."""
import ctypes
import os
import shutil
import subprocess

import numpy as np
import pytest
import torch

from tests.test_gauss_host import _words

pytestmark = pytest.mark.gpu

HERE = os.path.dirname(os.path.abspath(__file__))


@pytest.fixture(scope="module")
def lib(tmp_path_factory):
    nvcc = shutil.which("nvcc") or "/usr/local/cuda/bin/nvcc"
    if not os.path.exists(nvcc) or np.finfo(np.longdouble).nmant < 63:
        pytest.skip("nvcc or extended precision not available")
    out = str(tmp_path_factory.mktemp("gauss") / "libgauss.so")
    subprocess.run([nvcc, "-gencode", "arch=compute_103a,code=sm_103a", "-O3", "-std=c++17", "-shared", "-Xcompiler",
                    "-fPIC", "-o", out, os.path.join(HERE, "gauss_harness.cu")], check=True, capture_output=True)
    return ctypes.CDLL(out)


@pytest.mark.parametrize("kind", ["random", "small u", "u next to 1", "octaves", "log table", "axes", "angle table"])
def test_device_pairs_against_extended_precision(lib, kind):
    n = 50000
    w = _words(kind, n, 6)
    dev = torch.from_numpy(w.view(np.int64)).cuda()
    z = torch.zeros(n, 2, dtype=torch.float64, device="cuda")
    torch.cuda.synchronize()
    assert lib.gauss_pairs_device(ctypes.c_void_p(dev.data_ptr()), n, ctypes.c_void_p(z.data_ptr())) == 0
    z = z.cpu().numpy()
    u = ((w >> np.uint64(12)).astype(np.longdouble) + np.longdouble(0.5)) * np.longdouble(2.0) ** -52
    rad = np.sqrt(-np.log(u[:, 0]))
    # 2 pi u from the nearest multiple of a quarter, so that the argument is exact next to the axes
    q = np.round(4 * u[:, 1])
    d = (u[:, 1] - q / 4) * 2 * np.arctan2(np.longdouble(0), np.longdouble(-1))
    q = q.astype(int) % 4
    c, s = np.cos(d), np.sin(d)
    err = np.maximum(np.abs(z[:, 0] - rad * np.choose(q, [c, -s, -c, s])),
                     np.abs(z[:, 1] - rad * np.choose(q, [s, c, -s, -c])))
    # as on the host: 1.5 units of 2^-52 and a little (the two steps take any start within 2^-20 to 2^-52)
    assert float(np.max(err / rad)) < 1.6 * 2.0 ** -52
