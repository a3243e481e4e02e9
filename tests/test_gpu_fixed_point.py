"""The FP64-class transforms in block fixed point: every supported length along each axis, tile
remainders, the ends of the exponent range, non-finite values, against the same transforms in
extended precision (64 or 113 bits).

Tolerance.  Three forward and three inverse passes store FP64 values (each rounding 2^-54 of a
value's size, 0.32 of that in rms) and keep at least 2^-58 of a tile's largest component: a
few 1e-16 of the field's norm in all, as transforms in FP64."""
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
