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


def exact_moments(psi, h, simpson):
    """norm and rms in extended precision (64 or 113 bits)."""
    L = np.longdouble
    n = psi.shape
    dens = psi.real.astype(L) ** 2 + psi.imag.astype(L) ** 2
    w, x2 = [], []
    for d in range(3):
        q = np.ones(n[d], dtype=L)
        if simpson:
            q[1::2], q[::2] = L(4) / 3, L(2) / 3
            q[0] = q[n[d] - 2] = L(1) / 3
            q[n[d] - 1] = 0
        w.append(q)
        x2.append(((np.arange(n[d]) - n[d] // 2).astype(L) * L(h[d])) ** 2)
    dens = dens * w[0][:, None, None] * w[1][None, :, None] * w[2][None, None, :]
    tot = dens.sum()
    rms = [np.sqrt((dens.sum(axis=tuple(k for k in range(3) if k != d)) * x2[d]).sum() / tot) for d in range(3)]
    return np.array([L(h[0]) * L(h[1]) * L(h[2]) * tot, *rms], dtype=L)


def moments(psi_d, shape, h, simpson):
    import torch
    out = torch.zeros(4, dtype=torch.float64, device="cuda")
    params = abi.make_params(shape, h, 0.01, precision=abi.DGPE_MIXED,
                             integration=abi.DGPE_SIMPSON if simpson else abi.DGPE_RECTANGLE)
    abi.dgpe_moments_noalloc(psi_d.data_ptr(), params, out.data_ptr(), torch.cuda.current_stream().cuda_stream)
    return out.cpu().numpy()


@pytest.mark.parametrize("shape", [(2, 3, 2), (5, 4, 24), (7, 9, 62), (6, 40, 250), (33, 17, 258), (40, 41, 512), (3, 4, 5),
                                   (64, 64, 64), (3, 400, 250), (300, 5, 100), (100, 90, 24), (64, 512, 4)])
@pytest.mark.parametrize("simpson", [False, True])
@pytest.mark.parametrize("scale", [1.0, 1e-24, 1e17])
def test_moments_of_fp32_states(shape, simpson, scale):
    """The FP32 moments call is an FP64-quality sum: within 2e-15 (a few roundings of 1.1e-16 in
    the totals, the quotient and the root) of extended precision, also where the squares leave
    the FP32 range and where the field spans many powers of ten."""
    import torch
    h = (0.3, 0.25, 0.2)
    psi = (inputs.random_psi(shape, seed=11) * scale).astype(np.complex64)
    decay = np.exp(-np.linspace(0.0, 60.0, shape[0] * shape[1]).reshape(shape[0], shape[1], 1))
    for field in (psi, (psi * decay).astype(np.complex64), (psi * decay[::-1, ::-1]).astype(np.complex64)):
        dev = torch.from_numpy(np.ascontiguousarray(field)).cuda()
        odd = torch.empty(dev.numel() + 1, dtype=dev.dtype, device="cuda")[1:]
        odd.copy_(dev.reshape(-1))
        want = exact_moments(field, h, simpson)
        for t in (dev, odd):   # 16- and 8-byte aligned
            got = moments(t, shape, h, simpson)
            if simpson and want[0] == 0:
                continue
            assert np.all(np.abs(got - want) <= 2e-15 * np.abs(want)), (got - want) / want


def test_moments_of_nonfinite_states():
    import torch
    shape, h = (64, 48, 64), (0.3, 0.25, 0.2)
    psi = inputs.random_psi(shape, seed=2).astype(np.complex64)
    for bad in (np.inf, np.nan):
        field = psi.copy()
        field[3, 4, 17] = bad
        got = moments(torch.from_numpy(field).cuda(), shape, h, False)
        assert (np.isinf(got[0]) if np.isinf(bad) else np.isnan(got[0])) and np.all(np.isnan(got[1:]))


# every supported length, as the x axis of one grid and the y axis of another
ALL = [n for n in range(4, 513, 2)
       if any(n == 2 ** a * 3 ** b * 5 ** c * 7 ** d
              for a in range(1, 10) for b in range(6) for c in range(4) for d in range(4))]


@pytest.mark.parametrize("nx,ny", list(zip(ALL, reversed(ALL))))
def test_dipolar_potential_of_every_length(orc, nx, ny):
    """Phi through the x and y transforms of every length.  An FP32 transform's error is a few
    6e-8 per stage of the field's norm (at most five stages, four transforms): 3e-6."""
    shape = (nx, ny, 6)
    h = (9.0 / nx, 8.0 / ny, 1.1)
    psi = (inputs.random_psi(shape, seed=nx) * 0.3).astype(np.complex64)
    for cutoff in (0.0, 3.0):
        gpu = abi.Condensate(shape, h, 0.01, precision=abi.DGPE_MIXED, g=1.0, gdd=1.0, cutoff=cutoff)
        p = orc.make_params(shape, h, 0.01, orc.IMAG_TIME, (1.0, 1.0, 1.0), 1.0, 1.0, cutoff=cutoff)
        gpu.set_psi(psi)
        got = gpu.phi()
        gpu.close()
        assert rel(got, orc.dipolar_phi(p, np.abs(psi.astype(np.complex128)) ** 2)) < 3e-6


@pytest.mark.parametrize("n", ALL)
def test_z_lines_of_every_length(orc, n):
    """The density transform, the potential step and z sweep, and the observables along z lines of
    every length, a last tile of fewer lines among them.  Two steps: two transform chains (3e-6 of
    Phi, times dt gdd Phi < 0.05), six sweeps (2e-6 each): 1.5e-5; the observables quadratic in it."""
    shape = (4, 20, n)
    h = (0.5, 0.4, 8.0 / n)
    psi = (inputs.gaussian_psi(shape, h, noise=0.05, seed=n)).astype(np.complex64)
    for mode in (abi.DGPE_REAL_TIME, abi.DGPE_IMAG_TIME):
        for kinetic in (abi.DGPE_KINETIC_LAPLACIAN3, abi.DGPE_KINETIC_GRADIENT5):
            # (Simpson in imaginary time: in real time FP32-mixed steps restore that norm, the oracle's do not)
            simpson = kinetic and mode == abi.DGPE_IMAG_TIME
            opt = {"integration": abi.DGPE_SIMPSON if simpson else abi.DGPE_RECTANGLE, "kinetic": kinetic}
            gpu = abi.Condensate(shape, h, 0.004, mode=mode, precision=abi.DGPE_MIXED, nu=(1.0, 1.2, 0.8), g=5.0, gdd=3.0, **opt)
            gpu.set_psi(psi)
            gpu.step(2)
            got, obs = gpu.get_psi(), gpu.observables()
            gpu.close()
            p = orc.make_params(shape, h, 0.004, orc.IMAG_TIME if mode else orc.REAL_TIME, (1.0, 1.2, 0.8), 5.0, 3.0, **opt)
            want = orc.step(p, psi.astype(np.complex128), 2)
            if mode == abi.DGPE_REAL_TIME:
                assert rel(got, want) < 1.5e-5
            else:
                assert rel(got / np.linalg.norm(got), want / np.linalg.norm(want)) < 1.5e-5
            ref = orc.observables(p, got.astype(np.complex128))
            for k in ("norm", "mu", "energy", "e_kin", "e_trap", "e_contact", "rms_x", "rms_y", "rms_z"):
                if k in obs and k in ref:
                    assert obs[k] == pytest.approx(ref[k], rel=1e-5), k


@pytest.mark.parametrize("simpson", [False, True])
def test_moments_of_fp32_clouds_are_fp64_sums(simpson):
    """The sums of FP32 states are FP64-class: the points' sums are exact to 2^-54 of their largest
    density, the FP64 sums above them round at 2^-54 of a partial sum (about 8e-17 of the total in rms)
    and each result once (6e-17 in rms): below 1.5e-16 over 18 fields, which FP64 terms reach too."""
    import torch
    err = []
    for n, shape in enumerate([(64, 64, 64), (64, 48, 80), (96, 70, 64), (50, 100, 108), (128, 64, 96), (112, 64, 90)]):
        h = tuple(12.5 / k for k in shape)
        for seed in range(3):
            psi = inputs.gaussian_psi(shape, h, noise=1e-3, seed=10 * n + seed).astype(np.complex64)
            want = exact_moments(psi, h, simpson)
            err.append(np.abs(moments(torch.from_numpy(psi).cuda(), shape, h, simpson) - want) / want)
    assert np.all(np.sqrt(np.mean(np.square(np.array(err, dtype=np.float64)), axis=0)) < 1.5e-16)


@pytest.mark.parametrize("nz", [10, 20, 98, 360])
def test_observables_of_another_radix_order(orc, nz):
    """The observables under each radix order: the oracle's."""
    shape = (40, 42, nz)
    h = tuple(9.0 / n for n in shape)
    psi = inputs.gaussian_psi(shape, h, noise=0.02, seed=nz).astype(np.complex64)
    gpu = abi.Condensate(shape, h, 0.004, mode=abi.DGPE_REAL_TIME, precision=abi.DGPE_MIXED, nu=(1.0, 1.2, 0.8), g=5.0, gdd=3.0)
    gpu.set_psi(psi)
    p = orc.make_params(shape, h, 0.004, orc.REAL_TIME, (1.0, 1.2, 0.8), 5.0, 3.0)
    ref = orc.observables(p, psi.astype(np.complex128))
    default = gpu.tuning()
    for style in range(3):
        gpu.set_tuning(dict(default, plan_style=(0, 0, style)))
        obs = gpu.observables()
        for k in ("norm", "mu", "energy", "e_kin", "e_trap", "e_contact", "rms_x", "rms_y", "rms_z"):
            if k in obs and k in ref:
                assert obs[k] == pytest.approx(ref[k], rel=1e-5), k
    gpu.close()


def test_observables_of_another_radix_order_take_no_longer():
    """... in a time of the order of the default's: the other orders' transform is four to five stages
    instead of three, its sums are the same work on as many threads: twice the time at most."""
    import time
    import torch
    shape = (128, 126, 360)
    gpu = abi.Condensate(shape, 0.1, 0.004, mode=abi.DGPE_REAL_TIME, precision=abi.DGPE_MIXED, g=5.0, gdd=3.0)
    gpu.set_psi(inputs.gaussian_psi(shape, 0.1, seed=1).astype(np.complex64))
    default, seconds = gpu.tuning(), []
    for style in range(3):
        gpu.set_tuning(dict(default, plan_style=(0, 0, style)))
        best = 1e30
        for _ in range(20):
            torch.cuda.synchronize()
            t = time.perf_counter()
            gpu.observables()
            best = min(best, time.perf_counter() - t)
        seconds.append(best)
    gpu.close()
    assert max(seconds) < 2 * seconds[0], seconds
