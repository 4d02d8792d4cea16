"""The fixed-point hops of csrc/fixed.cuh on the host against exact rational
arithmetic (python integers): the error of a site's sum of hops is below that
of the same sum in FP64, over SU(3), interpolated and general links, spinors
of one scale, of very different scales between neighbours and between
components, zeros, and the ends of the range."""
import ctypes
import os
import shutil
import subprocess
from fractions import Fraction

import numpy as np
import pytest

from oracle import gauge

HERE = os.path.dirname(os.path.abspath(__file__))
T = np.array([-1, 1] * 4, dtype=np.int32)  # D: t = -1 forward, +1 backward


@pytest.fixture(scope="module")
def lib(tmp_path_factory):
    nvcc = shutil.which("nvcc") or "/usr/local/cuda/bin/nvcc"
    if not os.path.exists(nvcc):
        pytest.skip("nvcc not available")
    out = str(tmp_path_factory.mktemp("fx") / "libfx.so")
    subprocess.run([nvcc, "-O2", "-std=c++17", "-shared", "-Xcompiler", "-fPIC", "-o", out,
                    os.path.join(HERE, "fixed_point_harness.cu")], check=True, capture_output=True)
    return ctypes.CDLL(out)


def _e(mu, d):
    """e_mu d on two spin components (e_0 = -1, e_k = -i sigma_k)."""
    if mu == 0:
        return [-d[0], -d[1]]
    if mu == 1:
        return [-1j * d[1], -1j * d[0]]
    if mu == 2:
        return [-d[1], d[0]]
    return [-1j * d[0], 1j * d[1]]


def _edag(mu, w):
    if mu == 0:
        return [-w[0], -w[1]]
    if mu == 1:
        return [1j * w[1], 1j * w[0]]
    if mu == 2:
        return [w[1], -w[0]]
    return [1j * w[0], -1j * w[1]]


def _hops(u, psi, t):
    """Sum of the eight hops in FP64 numpy: u[n, 8, 3, 3], psi[n, 8, 4, 3]."""
    out = np.zeros((len(u), 4, 3), dtype=np.complex128)
    for d in range(8):
        mu = d >> 1
        up, dn = psi[:, d, :2], psi[:, d, 2:]
        h = up + t[d] * np.stack(_e(mu, [dn[:, 0], dn[:, 1]]), 1)
        m = u[:, d] if d % 2 == 0 else np.conj(np.swapaxes(u[:, d], -1, -2))
        w = np.einsum("nab,nsb->nsa", m, h)
        out[:, :2] += w
        out[:, 2:] += t[d] * np.stack(_edag(mu, [w[:, 0], w[:, 1]]), 1)
    return out


class _Q:
    """Exact complex rationals, with the operations _e, _edag and the sums need."""

    def __init__(self, re, im=0):
        self.re, self.im = Fraction(re), Fraction(im)

    def __add__(self, o):
        return _Q(self.re + o.re, self.im + o.im)

    def __neg__(self):
        return _Q(-self.re, -self.im)

    def __rmul__(self, z):
        z = complex(z)
        a, b = Fraction(z.real), Fraction(z.imag)
        return _Q(a * self.re - b * self.im, a * self.im + b * self.re)

    def mul(self, o):
        return _Q(self.re * o.re - self.im * o.im, self.re * o.im + self.im * o.re)

    def conj(self):
        return _Q(self.re, -self.im)


def _exact(u, psi, t):
    out = []
    for n in range(len(u)):
        acc = [[_Q(0) for _ in range(3)] for _ in range(4)]
        for d in range(8):
            mu = d >> 1
            p = [[_Q(psi[n, d, s, c].real, psi[n, d, s, c].imag) for c in range(3)] for s in range(4)]
            m = [[_Q(u[n, d, a, b].real, u[n, d, a, b].imag) for b in range(3)] for a in range(3)]
            if d % 2:
                m = [[m[b][a].conj() for b in range(3)] for a in range(3)]
            for a in range(3):
                w = []
                for s in range(2):
                    z = _Q(0)
                    for b in range(3):
                        e = _e(mu, [p[2][b], p[3][b]])[s]
                        z = z + m[a][b].mul(p[s][b] + (complex(int(t[d])) * e))
                    w.append(z)
                lo = _edag(mu, w)
                for s in range(2):
                    acc[s][a] = acc[s][a] + w[s]
                    acc[2 + s][a] = acc[2 + s][a] + (complex(int(t[d])) * lo[s])
        out.append(acc)
    return out


def _err(got, exact):
    """Sum of squared errors and of squares, from exact differences."""
    e = r = 0.0
    for n in range(len(exact)):
        for s in range(4):
            for c in range(3):
                q = exact[n][s][c]
                e += float(Fraction(got[n, s, c].real) - q.re) ** 2 + float(Fraction(got[n, s, c].imag) - q.im) ** 2
                r += float(q.re) ** 2 + float(q.im) ** 2
    return e, r


def _fixed(lib, u, psi, t, b=1.0):
    u, psi = np.ascontiguousarray(u), np.ascontiguousarray(psi)
    out = np.zeros((len(u), 4, 3), dtype=np.complex128)
    lib.fx_hops_host.argtypes = [ctypes.c_void_p] * 2 + [ctypes.c_int] * 2 + [ctypes.c_double, ctypes.c_void_p]
    left = lib.fx_hops_host(u.ctypes.data, psi.ctypes.data, int(t[0] > 0), len(u), b, out.ctypes.data)
    return out, left


def _inputs(kind, n, seed):
    g = np.random.default_rng(seed)
    u = gauge.generate_links((n, 1, 1, 2), 0.5, seed).reshape(n, 8, 3, 3)
    psi = (g.standard_normal((n, 8, 4, 3)) + 1j * g.standard_normal((n, 8, 4, 3))) / np.sqrt(2)
    if kind == "interp":
        u = 0.3 * u + 0.7 * gauge.generate_links((n, 1, 1, 2), 0.5, seed + 1).reshape(n, 8, 3, 3)
    elif kind == "general":  # entries of any size up to 5, links of different sizes
        u = 5.0 * (g.uniform(-1, 1, u.shape) + 1j * g.uniform(-1, 1, u.shape)) * 2.0 ** g.integers(-3, 4, (n, 8, 1, 1))
    elif kind == "largest":  # the bounds of the integer sums: every number 1 - 2^-53
        x = 1.0 - 2.0 ** -53
        u = x * (np.sign(g.standard_normal(u.shape)) + 1j * np.sign(g.standard_normal(u.shape)))
        u[: n // 2] = x * (1 - 1j)
        psi = x * (1 + 1j) * np.ones_like(psi)
    elif kind == "neighbours":  # neighbours of very different size
        psi = psi * 10.0 ** g.uniform(-12, 3, (n, 8, 1, 1))
    elif kind == "components":
        psi = psi * 10.0 ** g.uniform(-6, 0, psi.shape)
    elif kind == "zeros":
        psi[:, ::2] = 0
        psi[0] = 0
        u[1, 3] = 0
        psi[:, 1, 2] = 0
    elif kind == "small":
        psi = psi * 2.0 ** -700
    elif kind == "large":
        psi = psi * 2.0 ** 700
    return u, psi


@pytest.mark.parametrize("kind", ["su3", "interp", "general", "largest", "neighbours", "components", "zeros", "small",
                                  "large"])
@pytest.mark.parametrize("dag", [False, True])
def test_error_is_no_larger_than_in_fp64(lib, kind, dag):
    u, psi = _inputs(kind, 12, 7)
    t = -T if dag else T
    got, left = _fixed(lib, u, psi, t)
    assert left == 0
    scale = {"small": 2.0 ** 700, "large": 2.0 ** -700}.get(kind, 1.0)  # exact; keeps the squares in range
    exact = _exact(u, psi * scale, t)
    e_fx, norm = _err(got * scale, exact)
    e_64, _ = _err(_hops(u, psi * scale, t), exact)
    # one final rounding of each component (2^-53) is in both
    assert e_fx <= max(e_64, (2.0 ** -53) ** 2 * norm)


def test_range_and_scaling(lib):
    u, psi = _inputs("su3", 8, 9)
    a, left = _fixed(lib, u, psi, T, b=-0.5)
    assert left == 0
    b, _ = _fixed(lib, u, psi * 2.0 ** 40, T, b=-0.5)
    assert np.array_equal(a * 2.0 ** 40, b)  # powers of two move the exponent only
    for bad in (np.nan, np.inf, 1e300, 1e-300):
        q = psi * 0 if bad == 1e-300 else psi.copy()
        q[3, 4, 1, 2] = bad
        _, left = _fixed(lib, u, q, T)
        assert left == 1  # that site only
    w = u[0, 0].copy()
    out = np.zeros((3, 3), dtype=np.complex128)
    assert lib.fx_link_host(w.ctypes.data_as(ctypes.c_void_p), out.ctypes.data_as(ctypes.c_void_p)) != 0xFFFF
    assert np.abs(out - w).max() <= 2.0 ** -58 * np.abs(w).max() * 2
    w[1, 1] = 1e-290
    w[w != 1e-290] = 0  # out of range: kept as it is
    assert lib.fx_link_host(w.ctypes.data_as(ctypes.c_void_p), out.ctypes.data_as(ctypes.c_void_p)) == 0xFFFF
    assert np.array_equal(out, w)
