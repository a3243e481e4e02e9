"""The fixed-point arithmetic of the FP64 kernels (csrc/dgpe_fixed.cuh), compiled for the host and
compared with exact integers and with mpmath."""
import ctypes
import os
import subprocess

import numpy as np
import pytest

from paper_1610_05329_gb300 import build

HERE = os.path.dirname(os.path.abspath(__file__))


@pytest.fixture(scope="module")
def lib(tmp_path_factory):
    so = str(tmp_path_factory.mktemp("fixed") / "fixed_host.so")
    r = subprocess.run([build.nvcc(), *build.ARCH, "-O1", "-std=c++17", "-Xcompiler", "-fPIC", "-shared", "-I", build.CSRC,
                        "-I", os.path.join(build.ROOT, "include"), os.path.join(HERE, "fixed_host.cu"), "-o", so],
                       capture_output=True, text=True)
    assert r.returncode == 0, r.stderr
    return ctypes.CDLL(so)


def pair(re, im):
    return (ctypes.c_longlong * 2)(re, im)


def hi_lo(h, low):
    return (h << 32) + low


# low words at both ends of a signed word (-2^31 has no 32-bit negative), and around zero
LOW = [-(1 << 31), -(1 << 31) + 1, (1 << 31) - 1, 0, 1, -1]


@pytest.mark.parametrize("dir", [-1, 1])
def test_twiddle_words(lib, dir):
    """a w / 2^64 within the product of the low words (four of at most 2^62, so less than one unit)
    and half a unit of rounding twice: 2 units."""
    out = pair(0, 0)
    for lo_a in LOW:
        for lo_b in LOW:
            for lo_c in LOW:
                for lo_d in LOW:
                    a = (hi_lo(-(1 << 29) + 12345, lo_a), hi_lo((1 << 29) - 99, lo_b))
                    w = (hi_lo((1 << 27) + 7, lo_c), hi_lo(-(1 << 27) + 3, lo_d))
                    lib.host_twiddle(dir, pair(*a), pair(*w), out)
                    wi = w[1] if dir < 0 else -w[1]
                    want = (a[0] * w[0] - a[1] * wi, a[0] * wi + a[1] * w[0])
                    for got, x in zip(out, want):
                        assert abs((got << 64) - x) <= 2 << 64, (a, w)


L, CL = np.longdouble, np.clongdouble


def pointer(a):
    return a.ctypes.data_as(ctypes.POINTER(ctypes.c_double))


class Sweep:
    """The real-time sweep of m interior points by the kernels' twisted factorization, r = dt / (4 h^2):
    with the fixed-point functions, and in 64 bits with the same (rounded) coefficients."""

    def __init__(self, lib, m, r):
        self.lib, self.m, self.r = lib, m, r
        c = CL(1j * L(r))
        diag, h = 1 + 2 * c, m // 2
        e, alpha = [1 + 2 * c], [CL(0)]
        for i in range(1, m):
            alpha.append(c / e[-1])
            e.append(diag - c * alpha[-1])
        self.c = c
        self.alpha = np.array(alpha).astype(np.complex128)
        self.beta2 = (2 / np.array(e)).astype(np.complex128)
        self.ginv = np.array([1 / (e[h] + e[m - 1 - h] - diag)]).astype(np.complex128)

    def fixed(self, psi):   # [m][lines]
        out = np.ascontiguousarray(psi.T.copy())
        for line in out:
            self.lib.host_sweep(self.m, ctypes.c_double(self.r), pointer(self.alpha), pointer(self.beta2),
                                pointer(self.ginv), pointer(line))
        return out.T.astype(CL)

    def exact(self, psi):
        m, h, v = self.m, self.m // 2, psi.astype(CL)
        a, b = self.alpha.astype(CL), self.beta2.astype(CL)
        y, out = [None] * m, [None] * m
        for s in range(h):
            y[s] = v[s] + (a[s] * y[s - 1] if s else 0)
        for s in range(m - 1 - h):
            y[m - 1 - s] = v[m - 1 - s] + (a[s] * y[m - s] if s else 0)
        x_h = self.ginv.astype(CL)[0] * (v[h] + a[h] * y[h - 1] + a[m - 1 - h] * y[h + 1])
        out[h] = 2 * x_h - v[h]
        for first, way, n in ((h - 1, -1, h), (h + 1, 1, m - 1 - h)):
            t = self.c * x_h
            for j in range(n):
                i, q = first + way * j, n - 1 - j
                x = y[i] + t
                out[i] = b[q] * x - v[i]
                t = a[q + 1] * x
        return np.array(out)


def clouds(m, lines, seed):
    rng = np.random.default_rng(seed)
    x = ((np.arange(m) - m // 2) * 25.0 / m)[:, None]
    return (np.exp(-0.35 * rng.uniform(0.3, 3, lines) * x * x + 1j * rng.uniform(-0.2, 0.2, lines) * x) *
            rng.uniform(0.5, 2, lines) + 1e-3 * rng.uniform(-1, 1, (m, lines))).astype(np.complex128)


@pytest.mark.parametrize("m", [62, 254])
def test_sweep_roundings_lean_to_no_side(lib, m):
    """A run of many steps repeats every rounding, so what leans to one side adds up: the error's
    projection on the result (a change of its norm and phase) must be that of independent roundings,
    whose standard deviation is sqrt(sum |w|^2 |d|^2) / sum |w|^2 for errors d of results w: within
    five of them.  The error itself: a few roundings of 2^-53."""
    s = Sweep(lib, m, 0.0125)
    psi = clouds(m, 2000, m)
    want, got = s.exact(psi), s.fixed(psi)
    d, total = got - want, np.sum(np.abs(want) ** 2)
    lean = np.sum(np.conj(want) * d) / total
    noise = np.sqrt(np.sum(np.abs(want) ** 2 * np.abs(d) ** 2)) / total
    assert abs(lean.real) < 5 * noise and abs(lean.imag) < 5 * noise, (lean, noise)
    assert np.sqrt(np.sum(np.abs(d) ** 2) / total) < 2.2e-16


def phase(lib, imag, z, theta, g):
    p = (ctypes.c_double * 2)(z.real, z.imag)
    assert lib.host_phase(int(imag), p, ctypes.c_longlong(round(theta * 2.0 ** 58)), ctypes.c_double(g))
    return p[0], p[1]


@pytest.mark.parametrize("scale", [1.0, 1e-4, 1e-12, 1e-18, 1e-60])
def test_potential_step_of_a_point(lib, scale):
    """Imaginary time: each component within 2^-52 of itself (a rounding and an exponential good to
    2^-56).  Real time: within 2^-52 of the point's magnitude."""
    rng = np.random.default_rng(3)
    for _ in range(2000):
        z = complex(rng.uniform(-1, 1), scale * rng.uniform(-1, 1))
        theta, g = rng.uniform(0, 0.5), 0.1
        k = round(theta * 2.0 ** 58)
        angle = L(k) / L(2) ** 58 + L(g) * (L(z.real) ** 2 + L(z.imag) ** 2)
        got = phase(lib, True, z, theta, g)
        for x, q in ((z.real, got[0]), (z.imag, got[1])):
            want = L(x) * np.exp(-angle)
            assert abs(L(q) - want) <= L(2) ** -52 * abs(want)
        got = phase(lib, False, z, theta, g)
        c, s = np.cos(angle), np.sin(angle)
        assert abs(L(got[0]) - (L(z.real) * c + L(z.imag) * s)) <= L(2) ** -52 * abs(z)
        assert abs(L(got[1]) - (L(z.imag) * c - L(z.real) * s)) <= L(2) ** -52 * abs(z)


@pytest.mark.parametrize("scale", [1.0, 1e-4, 1e-20])
@pytest.mark.parametrize("r", [2e-4, 0.0056])
def test_real_time_sweep_by_magnitude(lib, scale, r):
    """Complex coefficients mix the parts: a component is good relative to the point's magnitude.  On
    smooth lines 2 beta x is at most 2.1 of the result, rounded to 53 bits (1.05 eps) and subtracted
    (0.5 eps): 2 eps.  The twist point has FP64 arithmetic, two complex multiply-adds and a product
    of two to four roundings each on up to 2.1 of the result: 10 eps."""
    m = 62
    s = Sweep(lib, m, r)
    x = np.exp(-0.002 * (np.arange(m) - m // 2) ** 2)[:, None]
    psi = x * (1.0 + 1j * scale * np.cos(0.1 * np.arange(200))[None, :])
    want, got = s.exact(psi), s.fixed(psi)
    bound = np.full((m, 1), 2.0)
    bound[m // 2] = 10.0
    bound = bound * np.finfo(np.float64).eps * np.abs(want)
    assert np.all(np.abs((got - want).real) <= bound) and np.all(np.abs((got - want).imag) <= bound)


# ---- the constants ---------------------------------------------------------------------------
@pytest.mark.parametrize("reach", [1e-3, 0.125, 0.1251, 0.8, 3.2, 17.9])
def test_cis(lib, reach):
    """e^{-i theta} in absolute terms within 2^-57 (the fits of the short angles, whose remainder is
    2^-58, and the rounding of five products at 2^-60; the long ones' reduction by quarter turns)."""
    mp = pytest.importorskip("mpmath")
    rng = np.random.default_rng(7)
    out = pair(0, 0)
    with mp.workprec(120):
        for x in np.concatenate([rng.uniform(-reach, reach, 2000), [0.0, reach, -reach]]):
            th = int(round(x * 2.0 ** 58))
            lib.host_cis(ctypes.c_longlong(th), out)
            angle = mp.mpf(th) / 2 ** 58
            assert abs(mp.mpf(out[0]) / 2 ** 60 - mp.cos(angle)) < mp.mpf(2) ** -57
            assert abs(mp.mpf(out[1]) / 2 ** 60 + mp.sin(angle)) < mp.mpf(2) ** -57


@pytest.mark.parametrize("reach", [1e-3, 0.5, 4.0, 17.9])
def test_exp(lib, reach):
    """e^-theta within 2^-56 of itself: theta log2 e, up to 26, rounded twice at 2^-58 of a turn."""
    mp = pytest.importorskip("mpmath")
    lib.host_exp.restype = ctypes.c_longlong
    rng = np.random.default_rng(8)
    n = ctypes.c_int(0)
    with mp.workprec(120):
        for x in np.concatenate([rng.uniform(-reach, reach, 2000), [0.0, reach, -reach]]):
            th = int(round(x * 2.0 ** 58))
            p = lib.host_exp(ctypes.c_longlong(th), ctypes.byref(n))
            want = mp.exp(-mp.mpf(th) / 2 ** 58)
            assert abs(mp.mpf(p) * mp.mpf(2) ** (n.value - 60) - want) < mp.mpf(2) ** -56 * want


@pytest.mark.parametrize("p", range(2, 11))
@pytest.mark.parametrize("dir", [-1, 1])
def test_butterflies(lib, p, dir):
    """Against the discrete Fourier sum.  A product by a constant is off by less than a unit (half of
    rounding, less than half of the words left out), a halving or quartering by less than one; an
    output has at most 6 products (radix 7) or two levels of 2 + 2 (radices 9 and 10): 16 units."""
    mp = pytest.importorskip("mpmath")
    rng = np.random.default_rng(p)
    with mp.workprec(140):
        w = [mp.expjpi(mp.mpf(2 * dir * k) / p) for k in range(p)]
        for _ in range(50):
            v = [int(x) for x in rng.integers(-(1 << 58), 1 << 58, 2 * p)]
            z = [mp.mpc(v[2 * k], v[2 * k + 1]) for k in range(p)]
            buf = (ctypes.c_longlong * (2 * p))(*v)
            lib.host_butterfly(dir, p, buf)
            for k in range(p):
                want = mp.fsum(z[j] * w[j * k % p] for j in range(p))
                assert abs(buf[2 * k] - want.real) < 16 and abs(buf[2 * k + 1] - want.imag) < 16, k
