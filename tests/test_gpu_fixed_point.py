"""The FP64 step's kernels in fixed point.  The transforms: every supported length along each axis, tile
remainders, the ends of the exponent range, non-finite values; the sweeps: lengths around their chunks and tiles, short
and long reach; the potential step: small and large angles and factors.  All against the same
formulas in extended precision (64 or 113 bits).

Tolerances.  Transforms: three forward and three inverse passes store FP64 values (each rounding 2^-54 of a
value's size, 0.32 of that in rms) and keep at least 2^-58 of a tile's largest component: a
few 1e-16 of the field's norm in all, as transforms in FP64.  A sweep keeps at least 52 bits of
each coefficient and 2^-56 of each value, amplified by 1 / (1 - |alpha|)^2 <= 5 at the largest c
here, and rounds once or twice: 1e-15.  The potential step's angle and factor are within 2^-56
(the FP64 sine of a large angle within its rounding, 2^-53 |theta|): 3e-16 (1 + |theta|)."""
import numpy as np
import pytest

from paper_1610_05329_gb300 import abi, inputs

pytestmark = pytest.mark.gpu
L = np.longdouble
TOL = {abi.DGPE_FP64: 5e-16, abi.DGPE_DF64: 2e-13}

ALL = [n for n in range(4, 513, 2)
       if any(n == 2 ** a * 3 ** b * 5 ** c * 7 ** d
              for a in range(1, 10) for b in range(6) for c in range(4) for d in range(4))]


@pytest.fixture(scope="module", autouse=True)
def built():
    from paper_1610_05329_gb300 import build
    build.build()
    abi.load()


def exact_phi(psi, h):
    n = psi.shape
    dens = psi.real.astype(L) ** 2 + psi.imag.astype(L) ** 2
    two_pi = 8 * np.arctan(L(1))
    k = [two_pi * np.where(np.arange(m) <= m // 2, np.arange(m), np.arange(m) - m).astype(L) / (L(m) * L(d)) for m, d in zip(n, h)]
    k2 = k[0][:, None, None] ** 2 + k[1][None, :, None] ** 2 + k[2][None, None, :] ** 2
    k2[0, 0, 0] = 1
    u = 3 * k[2][None, None, :] ** 2 / k2 - 1
    u[0, 0, 0] = 0
    return np.fft.ifftn(u * np.fft.fftn(dens)).real


def phi(psi, h, precision):
    gpu = abi.Condensate(psi.shape, h, 0.01, precision=precision, g=1.0, gdd=1.0)
    gpu.set_psi(psi)
    out = gpu.phi()
    gpu.close()
    return out


def error(got, want):
    return float(np.linalg.norm((got.astype(L) - want).ravel()) / np.linalg.norm(want.ravel()))


@pytest.mark.parametrize("precision", [abi.DGPE_FP64, abi.DGPE_DF64])
@pytest.mark.parametrize("n,m", list(zip(ALL, reversed(ALL))))
def test_every_length(n, m, precision):
    for shape in ((n, m, 6), (4, 6, n)):   # x and y, z (a last tile of fewer lines)
        h = (9.0 / shape[0], 8.0 / shape[1], 7.0 / shape[2])
        psi = inputs.random_psi(shape, seed=n) * 0.3
        assert error(phi(psi, h, precision), exact_phi(psi, h)) < TOL[precision]


@pytest.mark.parametrize("shape", [(48, 50, 64), (24, 30, 250), (60, 128, 36)])
def test_trapped_cloud(shape):
    """Tails that fall by many powers of ten within a tile."""
    h = tuple(12.0 / n for n in shape)
    psi = inputs.gaussian_psi(shape, h, seed=5)
    assert error(phi(psi, h, abi.DGPE_FP64), exact_phi(psi, h)) < TOL[abi.DGPE_FP64]


@pytest.mark.parametrize("scale", [1e-140, 1e140])
def test_exponent_range(scale):
    shape, h = (24, 20, 28), (0.3, 0.4, 0.25)
    psi = inputs.random_psi(shape, seed=8) * scale
    got = phi(psi, h, abi.DGPE_FP64)
    assert error(got, exact_phi(psi, h)) < TOL[abi.DGPE_FP64]


@pytest.mark.parametrize("precision", [abi.DGPE_FP64, abi.DGPE_DF64])
@pytest.mark.parametrize("bad", [np.inf, np.nan])
def test_nonfinite(precision, bad):
    psi = inputs.random_psi((16, 24, 36), seed=8)
    psi[3, 4, 5] = bad
    assert np.all(np.isnan(phi(psi, (0.3, 0.3, 0.3), precision)))


def test_zero_state():
    psi = np.zeros((16, 24, 36), dtype=np.complex128)
    assert np.all(phi(psi, (0.3, 0.3, 0.3), abi.DGPE_FP64) == 0)


@pytest.mark.parametrize("shape", [(12, 14, 24), (64, 50, 250), (128, 6, 512), (4, 6, 36), (36, 10, 8)])
@pytest.mark.parametrize("mode", [abi.DGPE_REAL_TIME, abi.DGPE_IMAG_TIME])
def test_steps(orc, shape, mode):
    """Whole steps (the phase pass included) at lengths with and without these transforms."""
    h = tuple(10.0 / n for n in shape)
    psi = inputs.gaussian_psi(shape, h, seed=6)
    gpu = abi.Condensate(shape, h, 0.004, mode=mode, precision=abi.DGPE_FP64, nu=(1.0, 1.2, 0.8), g=20.0, gdd=10.0)
    gpu.set_psi(psi)
    gpu.step(3)
    got = gpu.get_psi()
    gpu.close()
    p = orc.make_params(shape, h, 0.004, orc.IMAG_TIME if mode else orc.REAL_TIME, (1.0, 1.2, 0.8), 20.0, 10.0)
    want = orc.step(p, psi, 3)
    assert np.linalg.norm(got - want) / np.linalg.norm(want) < 1e-12


def exact_sweep(psi, axis, r, imag):
    """2 (1 - c D)^-1 psi - psi on the interior of every line, walls zero."""
    v = np.moveaxis(psi, axis, 0)[1:-1].astype(np.clongdouble)
    c = np.clongdouble(L(r) if imag else 1j * L(r))
    m, diag = v.shape[0], 1 + 2 * c
    e, y, x = [diag], [v[0]], [None] * m
    for i in range(1, m):
        alpha = c / e[-1]
        e.append(diag - c * alpha)
        y.append(v[i] + alpha * y[-1])
    x[m - 1] = y[m - 1] / e[m - 1]
    for i in range(m - 2, -1, -1):
        x[i] = (y[i] + c * x[i + 1]) / e[i]
    out = np.zeros((m + 2,) + v.shape[1:], dtype=np.clongdouble)
    out[1:-1] = 2 * np.array(x) - v
    return np.moveaxis(out, 0, axis)


def cerror(got, want):
    return float(np.linalg.norm((got.astype(np.clongdouble) - want).ravel()) / np.linalg.norm(want.ravel()))


@pytest.mark.parametrize("n", [4, 6, 8, 10, 12, 18, 20, 36, 50, 128, 250, 512])
@pytest.mark.parametrize("mode", [abi.DGPE_REAL_TIME, abi.DGPE_IMAG_TIME])
def test_sweeps(n, mode):
    for axis, which in ((0, abi.DGPE_SUB_CN_X), (1, abi.DGPE_SUB_CN_Y), (2, abi.DGPE_SUB_CN_Z)):
        for other in ((6, 10), (10, 14)):   # 60 and 140 lines: tiles of 64, warps of 16
            shape = list(other)
            shape.insert(axis, n)
            psi = inputs.random_psi(tuple(shape), seed=n)
            psi[1::2] *= 1e-9
            for dt in (1e-6, 0.02, 0.8):
                gpu = abi.Condensate(tuple(shape), 0.3, dt, mode=mode, precision=abi.DGPE_FP64)
                gpu.set_psi(psi)
                gpu.substep(which)
                got = gpu.get_psi()
                gpu.close()
                want = exact_sweep(psi, axis, dt / (4 * L(0.3) ** 2), mode == abi.DGPE_IMAG_TIME)
                assert cerror(got, want) < 1e-15, (axis, other, dt)


def test_sweep_tails():
    """A cloud that falls to 1e-100: every value within FP64's precision of itself, not of the largest."""
    n = 256
    x = np.arange(n) - n // 2
    psi = np.zeros((n, 4, 4), dtype=np.complex128)
    psi[:, 1:3, 1:3] = np.exp(-0.014 * x * x + 0.2j * x)[:, None, None]
    gpu = abi.Condensate(psi.shape, 0.3, 0.004, mode=abi.DGPE_REAL_TIME, precision=abi.DGPE_FP64)
    gpu.set_psi(psi)
    gpu.substep(abi.DGPE_SUB_CN_X)
    got = gpu.get_psi()[1:-1, 1:3, 1:3]
    gpu.close()
    want = exact_sweep(psi, 0, 0.004 / (4 * L(0.3) ** 2), False)[1:-1, 1:3, 1:3]
    assert np.max(np.abs(got - want) / np.abs(want)) < 4e-15


@pytest.mark.parametrize("mode", [abi.DGPE_REAL_TIME, abi.DGPE_IMAG_TIME])
@pytest.mark.parametrize("shape", [(12, 14, 24), (8, 6, 250), (6, 20, 64)])
@pytest.mark.parametrize("dt,g,gdd,scale", [(1e-3, 20.0, 10.0, 1.0), (0.02, 50.0, 40.0, 1.0), (1e-3, 20.0, 10.0, 1e-30),
                                            (0.5, 20.0, 10.0, 0.3), (1e-3, 1e5, 0.0, 1.0), (1e-3, 5.0, 1e5, 0.3),
                                            (1e-3, 0.0, 0.0, 1e5)])
def test_potential_step(mode, shape, dt, g, gdd, scale):
    h = tuple(8.0 / n for n in shape)
    nu = (1.0, 1.5, 0.7)
    psi = inputs.gaussian_psi(shape, h, seed=9) * scale
    gpu = abi.Condensate(shape, h, dt, mode=mode, precision=abi.DGPE_FP64, nu=nu, g=g, gdd=gdd)
    gpu.set_psi(psi)
    gpu.substep(abi.DGPE_SUB_POTENTIAL)
    got = gpu.get_psi()
    gpu.close()
    x = [((np.arange(n) - n // 2).astype(L) * L(d)) for n, d in zip(shape, h)]
    v = [L(a) ** 2 * q * q / 2 for a, q in zip(nu, x)]
    dens = psi.real.astype(L) ** 2 + psi.imag.astype(L) ** 2
    theta = L(dt) * (v[0][:, None, None] + v[1][None, :, None] + v[2][None, None, :] + L(g) * dens)
    if gdd:
        theta = theta + L(dt) * L(gdd) * exact_phi(psi, h)
    f = np.exp(-theta) if mode == abi.DGPE_IMAG_TIME else np.cos(theta) - 1j * np.sin(theta)
    assert cerror(got, psi * f) < 3e-16 * (1 + float(np.max(np.abs(theta))))


# ---- components of very different size ---------------------------------------------------------
# Imaginary time: the real and imaginary parts are two fields under the same real factors, and each
# keeps FP64's bits: the tolerances above, of each part by itself.  (Real time mixes the parts: each is
# good relative to the point's magnitude, test_fixed_host.py.)
def two_parts(shape, scale):
    return (inputs.random_psi(shape, seed=3).real + 1j * scale * inputs.random_psi(shape, seed=4).real).astype(np.complex128)


@pytest.mark.parametrize("scale", [1e-4, 1e-12, 1e-20])
@pytest.mark.parametrize("axis,which", [(0, abi.DGPE_SUB_CN_X), (1, abi.DGPE_SUB_CN_Y), (2, abi.DGPE_SUB_CN_Z)])
def test_imaginary_time_sweep_keeps_each_component(axis, which, scale):
    for shape in ((20, 14, 36), (6, 50, 18)):
        psi = two_parts(shape, scale)
        gpu = abi.Condensate(shape, 0.3, 0.02, mode=abi.DGPE_IMAG_TIME, precision=abi.DGPE_FP64)
        gpu.set_psi(psi)
        gpu.substep(which)
        got = gpu.get_psi()
        gpu.close()
        want = exact_sweep(psi, axis, 0.02 / (4 * L(0.3) ** 2), True)
        assert error(got.real, want.real) < 1e-15 and error(got.imag, want.imag) < 1e-15


@pytest.mark.parametrize("scale", [1e-4, 1e-12, 1e-20])
@pytest.mark.parametrize("shape", [(12, 14, 24), (6, 20, 64)])
def test_imaginary_time_potential_step_keeps_each_component(shape, scale):
    psi, dt = two_parts(shape, scale), 0.02
    h = tuple(8.0 / n for n in shape)
    gpu = abi.Condensate(shape, h, dt, mode=abi.DGPE_IMAG_TIME, precision=abi.DGPE_FP64, g=5.0, gdd=2.0)
    gpu.set_psi(psi)
    gpu.substep(abi.DGPE_SUB_POTENTIAL)
    got = gpu.get_psi()
    gpu.close()
    x = [((np.arange(n) - n // 2).astype(L) * L(d)) for n, d in zip(shape, h)]
    v = sum((q * q / 2).reshape([-1 if d == e else 1 for e in range(3)]) for d, q in enumerate(x))
    theta = L(dt) * (v + 5 * (psi.real.astype(L) ** 2 + psi.imag.astype(L) ** 2) + 2 * exact_phi(psi, h))
    bound = 3e-16 * (1 + float(np.max(np.abs(theta))))
    assert error(got.real, psi.real * np.exp(-theta)) < bound and error(got.imag, psi.imag * np.exp(-theta)) < bound
