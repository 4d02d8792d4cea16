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

from oracle import dirac, gauge

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


def _alike(lib, psi):
    psi = np.ascontiguousarray(psi.reshape(-1, 4, 3))
    out = np.zeros(len(psi), dtype=np.int32)
    lib.fx_alike_host(psi.ctypes.data_as(ctypes.c_void_p), len(psi), out.ctypes.data_as(ctypes.c_void_p))
    return out.astype(bool)


def test_which_spinors_are_left_to_fp64(lib):
    g = np.random.default_rng(3)
    psi = (g.standard_normal((200000, 4, 3)) + 1j * g.standard_normal((200000, 4, 3))) / np.sqrt(2)
    assert (~_alike(lib, psi)).sum() <= 20  # expected: 6 of 200000 x 6 groups of four numbers below 2^-6 of the largest
    one = psi[:1000]
    for small in (0.0, 1e-12, 1e-3):
        q = one.copy()
        q[:, :, 2] *= small  # a colour
        assert not _alike(lib, q).any()
        q = one.copy()
        q[:, 2:] *= small  # a chirality
        assert not _alike(lib, q).any()
        q = one * small
        q[:, 1, 0] = 1.0  # all but one component
        assert not _alike(lib, q).any()


@pytest.mark.parametrize("kind", ["unit", "abelian", "su3"])
def test_every_output_is_as_accurate_as_its_terms(lib, kind):
    """Spinors taken in fixed point whose colours and spins differ as much as they
    may: the error of each output number against the sum of its terms' sizes."""
    n, g = 24, np.random.default_rng(4)
    u, psi = _inputs("su3", n, 6)
    if kind != "su3":
        u = np.zeros_like(u)
        for c in range(3):
            u[..., c, c] = np.exp(1j * g.uniform(0, 2 * np.pi, (n, 8))) if kind == "abelian" else 1.0
    psi = psi * 2.0 ** g.uniform(-8, 0, (n, 8, 1, 3)) * 2.0 ** g.uniform(-3, 0, (n, 8, 4, 1))
    ok = _alike(lib, psi).reshape(n, 8)
    psi[~ok] = _inputs("su3", n, 8)[1][~ok]
    assert ok.sum() > n and _alike(lib, psi).all()
    got, left = _fixed(lib, u, psi, T)
    assert left == 0
    exact = _exact(u, psi, T)
    size = np.zeros((n, 4, 3))  # of the terms of an output
    for d in range(8):
        up, dn = np.abs(psi[:, d, :2]), np.abs(psi[:, d, 2:])
        h = up + (dn if d >> 1 in (0, 3) else dn[:, ::-1])
        m = np.abs(u[:, d]) if d % 2 == 0 else np.abs(np.swapaxes(u[:, d], -1, -2))
        w = np.einsum("nab,nsb->nsa", m, h)
        size[:, :2] += w
        size[:, 2:] += w if d >> 1 in (0, 3) else w[:, ::-1]
    for i in range(n):
        for s in range(4):
            for c in range(3):
                q = exact[i][s][c]
                e = max(abs(float(Fraction(got[i, s, c].real) - q.re)), abs(float(Fraction(got[i, s, c].imag) - q.im)))
                # eight roundings of 2^-54 of the largest product, which is at most 2^8 x the smallest group's terms
                assert e <= 2.0 ** -43 * size[i, s, c]


def _lu_rows(kind, n, w, seed):
    g = np.random.default_rng(seed)
    l = g.standard_normal((n, w)) + 1j * g.standard_normal((n, w))
    u = g.standard_normal((n, w)) + 1j * g.standard_normal((n, w))
    if kind == "multipliers":  # rows of L21 after partial pivoting
        l = l / np.maximum(1.0, np.abs(l))
    elif kind == "graded":  # large multipliers meet small entries, over three decades
        s = 10.0 ** g.uniform(-3, 0, (n, w))
        l, u = l * s, u / s * 10.0 ** g.uniform(-3, 0, (n, w))
    elif kind == "positive":  # no cancellation, all errors of one sign would add up
        l, u = np.abs(l.real) + 1j * np.abs(l.imag), np.abs(u.real) + 1j * np.abs(u.imag)
    elif kind == "largest":
        x = 2.0 - 2.0 ** -52
        l, u = l * 0 + x * (1 - 1j), u * 0 + x * (1 - 1j)
        u[n // 2:] = x * (1 + 1j)
    elif kind == "factors":  # rows and columns of the LU of an even-odd reduced block operator
        scipy_linalg = pytest.importorskip("scipy.linalg")
        block, kappa = (4, 4, 2, 2), 0.156
        A = 1.0 / (2.0 * kappa)
        U = gauge.generate_links(block, 0.5, seed)
        M = dirac.dense_matrix(lambda v: dirac.apply_D_open(U, v, kappa), 64, block + (4, 3))
        odd = np.repeat((np.indices(block).sum(0) % 2).reshape(-1), 12) == 1
        S = A * np.eye(384) - M[np.ix_(odd, ~odd)] @ M[np.ix_(~odd, odd)] / A
        _, L, R = scipy_linalg.lu(S)
        for k in range(n):
            p = w * int(g.integers(0, 384 // w - 1))
            i, j = (int(v) for v in g.integers(p + w, 384, 2))
            l[k], u[k] = L[i, p:p + w], R[p:p + w, j]
    return l, u


@pytest.mark.parametrize("kind", ["gauss", "multipliers", "positive", "largest", "factors", "graded"])
@pytest.mark.parametrize("w", [8, 16])
def test_lu_update_error_is_no_larger_than_in_fp64(lib, kind, w):
    """The sums of the LU's trailing update against exact ones: rms error at most
    that of a chain of FP64 multiply-adds, and no bias.  Where a row and its
    column are graded against each other, only relative to the product of their
    largest numbers (a common exponent each)."""
    n = 200
    l, u = _lu_rows(kind, n, w, 3)
    e_fx, e_64, ulp = np.zeros((n, 2)), np.zeros((n, 2)), np.zeros((n, 2))
    for i in range(n):
        o = np.zeros(2)
        a, b = np.ascontiguousarray(l[i]), np.ascontiguousarray(u[i])
        lib.lu_sum_host(a.ctypes.data_as(ctypes.c_void_p), b.ctypes.data_as(ctypes.c_void_p), w,
                        o.ctypes.data_as(ctypes.c_void_p))
        exact, chain = [Fraction(0), Fraction(0)], [0.0, 0.0]
        for p, q in zip(l[i], u[i]):
            x, y, z, t = (Fraction(float(v)) for v in (p.real, p.imag, q.real, q.imag))
            for k, m in ((0, x * z), (0, -y * t), (1, x * t), (1, y * z)):
                exact[k] += m
                chain[k] = float(Fraction(chain[k]) + m)  # one rounding, as a fused multiply-add
        scale = Fraction(float(np.abs(l[i]).max() * np.abs(u[i]).max())) or 1  # (a zero row)
        for k in range(2):
            e_fx[i, k] = float((Fraction(float(o[k])) - exact[k]) / scale)
            e_64[i, k] = float((Fraction(chain[k]) - exact[k]) / scale)
            ulp[i, k] = abs(float(exact[k] / scale)) * 2.0 ** -53  # rounding of the result itself
    rms = np.sqrt((e_fx ** 2).mean())
    if kind == "graded":
        # 4 w numbers cut off by less than 2^-55 of 2^E, times one of at most 2 2^E; 8 + 1/2 units of 2^-54 dropped
        assert np.abs(e_fx).max() <= (8 * w + 17) * 2.0 ** -55
        return
    assert rms <= np.sqrt(np.maximum((e_64 ** 2).mean(), (ulp ** 2).mean()))
    # the mean of n errors of no sign stays within four of its own standard deviations
    if kind != "largest":
        assert np.abs(e_fx.mean(0)).max() <= 4 * rms / np.sqrt(n)
