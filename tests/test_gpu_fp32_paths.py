"""FP32-mixed kernels at the line lengths and layouts where their dispatch changes, against the
FP64 oracle on the same seeded inputs.

Tolerances.  A Crank-Nicolson sweep is a product of FP32-rounded factors (each 6e-8 relative)
whose recurrences contract (|alpha| < 1), about ten roundings per point: 2e-6 of the field's
norm bounds it."""
import numpy as np
import pytest

from paper_1610_05329_gb300 import abi, inputs

pytestmark = pytest.mark.gpu

SWEEP_TOL = 2e-6


def rel(a, b):
    return float(np.linalg.norm(np.asarray(a) - np.asarray(b)) / np.linalg.norm(np.asarray(b)))


@pytest.fixture(scope="module", autouse=True)
def built():
    from paper_1610_05329_gb300 import build
    build.build()
    abi.load()


# one chunk, a last chunk of one point, 12 and 16 points per thread, every number of columns
# per tile (64, 32, 16, 8) and, beyond 16 chunks, the x lines' pairs of tiles
LENGTHS = (4, 14, 18, 20, 32, 48, 50, 96, 98, 128, 160, 192, 200, 250, 256, 270, 288, 320, 384, 392, 450, 500, 512)


@pytest.mark.parametrize("n", LENGTHS)
@pytest.mark.parametrize("mode", [abi.DGPE_REAL_TIME, abi.DGPE_IMAG_TIME])
def test_sweep_lengths(orc, n, mode):
    for axis, which in ((0, abi.DGPE_SUB_CN_X), (1, abi.DGPE_SUB_CN_Y)):
        shape = (n, 6, 10) if axis == 0 else (6, n, 10)
        psi = inputs.random_psi(shape, seed=n).astype(np.complex64)
        for dt in (0.02, 0.8):   # dt / (4 h^2) = 0.06 and 2.2: short and long reach along the line
            gpu = abi.Condensate(shape, 0.3, dt, mode=mode, precision=abi.DGPE_MIXED)
            p = orc.make_params(shape, 0.3, dt, orc.IMAG_TIME if mode else orc.REAL_TIME, (1.0, 1.0, 1.0), 0.0, 0.0)
            gpu.set_psi(psi)
            gpu.substep(which)
            got = gpu.get_psi()
            gpu.close()
            assert rel(got, orc.cn_sweep(p, psi.astype(np.complex128), axis)) < SWEEP_TOL, (axis, dt)


@pytest.mark.parametrize("shape", [(4, 6, 8), (48, 36, 50), (288, 10, 14), (512, 6, 20)])
@pytest.mark.parametrize("integration", [abi.DGPE_RECTANGLE, abi.DGPE_SIMPSON])
def test_step_norm(shape, integration):
    """The x sweep's norm sum: imaginary time renormalises by it, so the FP64 norm of the result
    is 1 within the rounding of the stored FP32 values (6e-8, averaging out over the points)."""
    gpu = abi.Condensate(shape, 0.4, 0.01, precision=abi.DGPE_MIXED, g=5.0, gdd=2.0, integration=integration)
    gpu.set_psi(inputs.gaussian_psi(shape, 0.4, seed=3))
    gpu.step(2)
    norm = gpu.observables()["norm"]
    gpu.close()
    assert norm == pytest.approx(1.0, abs=2e-7)


def test_adjoint_cotangent_of_any_alignment():
    """The cotangent is the caller's: 8-byte aligned complex64 gives the 16-byte aligned result."""
    import torch
    shape = (32, 48, 20)
    gpu = abi.Condensate(shape, 0.3, 0.01, mode=abi.DGPE_REAL_TIME, precision=abi.DGPE_MIXED, g=5.0, gdd=2.0)
    psi = torch.from_numpy(inputs.gaussian_psi(shape, 0.3, seed=4).astype(np.complex64)).cuda()
    w = torch.from_numpy(inputs.random_psi(shape, seed=5).astype(np.complex64)).cuda()
    a = w.clone()
    odd = torch.empty(w.numel() + 1, dtype=w.dtype, device=w.device)[1:]
    assert a.data_ptr() % 16 == 0 and odd.data_ptr() % 16 == 8
    odd.copy_(w.reshape(-1))
    gpu.adjoint_step(psi, a)
    gpu.adjoint_step(psi, odd)
    assert torch.equal(a.reshape(-1), odd)
    gpu.close()
