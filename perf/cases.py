"""The solver's workloads, as a user's program runs them through paper_1610_05329_gb300.abi.

Every case is one call sequence of a kind of program:
  step      hand a state to a Condensate, advance it, take it back (and its observables)
  observe   the observables and the dipolar potential Phi of the state held
  moments   norm and rms sizes of a caller's own psi (the per-step monitoring hook)
  adjoint   one adjoint step: the cotangent of psi and the parameter derivatives
  gradient  loss and gradients of a whole trajectory through torch autograd
  batch     many small independent condensates advanced together
Sizes are those of the repository's workloads, tests and timing grids, and generic ones of
the supported form (even, 2^a 3^b 5^c 7^d, at most 512 points per axis).
"""
import math
import random

import numpy as np
import torch

from paper_1610_05329_gb300 import abi

PRECISION = {"fp64": abi.DGPE_FP64, "mixed": abi.DGPE_MIXED, "df64": abi.DGPE_DF64}
MODE = {"real": abi.DGPE_REAL_TIME, "imag": abi.DGPE_IMAG_TIME}
OBS = ("norm", "mu", "energy", "e_kin", "e_trap", "e_contact", "e_dipolar")


def _case(kind, precision, mode, shape, box, dt, steps=1, name=None, nu=(1.0, 1.0, 1.0), g=20.0, gdd=10.0,
          cutoff=0.0, simpson=False, gradient5=False, observables=False, **more):
    """box: edge lengths (hx nx, hy ny, hz nz) of the grid."""
    c = {"kind": kind, "precision": precision, "mode": mode, "nx": shape[0], "ny": shape[1], "nz": shape[2],
         "lx": float(box[0]), "ly": float(box[1]), "lz": float(box[2]), "dt": dt, "steps": steps,
         "nux": nu[0], "nuy": nu[1], "nuz": nu[2], "g": float(g), "gdd": float(gdd), "cutoff": float(cutoff),
         "simpson": simpson, "gradient5": gradient5, "observables": observables}
    if name:
        c["name"] = name
    return {**c, **more}


def listed():
    return [
        # the smallest call: one step of one small grid (a scan's shortest member), where
        # launches and copies are all there is
        _case("step", "mixed", "imag", (32, 32, 32), (12.8,) * 3, 0.004, 1, "step_mixed_32"),
        # ground-state search on the 64^3 workload: a block of steps, then mu and energy
        _case("step", "fp64", "imag", (64, 64, 64), (12.8,) * 3, 0.004, 20, "ground_fp64_64", observables=True),
        # the 256^3 real-time run after a quench
        _case("step", "fp64", "real", (256, 256, 256), (25.6,) * 3, 5e-4, 4, "real_fp64_256",
              nu=(0.5, 1.0, 1.5), g=40.0, gdd=25.0),
        # one of the timing grids of the method's own programs, imaginary time, their
        # Simpson quadrature in the renormalisation
        _case("step", "fp64", "imag", (480, 480, 250), (24.0, 24.0, 12.5), 1e-3, 2, "imag_fp64_480x480x250",
              g=50.0, gdd=25.0, simpson=True),
        # the large FP32-mixed grid in real time
        _case("step", "mixed", "real", (512, 512, 384), (25.6, 25.6, 19.2), 5e-4, 4, "real_mixed_512x512x384",
              nu=(1.0, 1.0, 2.0), g=100.0, gdd=60.0),
        # FP32-mixed ground-state search on another timing grid (no power of two), with the
        # spherical cutoff of the dipolar interaction and the observables of the result
        _case("step", "mixed", "imag", (480, 480, 500), (24.0, 24.0, 25.0), 1e-3, 4, "imag_mixed_480x480x500",
              nu=(1.0, 1.0, 1.5), g=100.0, gdd=60.0, cutoff=11.0, observables=True),
        # the 256^3 run in double-float arithmetic
        _case("step", "df64", "real", (256, 256, 256), (25.6,) * 3, 5e-4, 4, "real_df64_256",
              nu=(0.5, 1.0, 1.5), g=40.0, gdd=25.0),
        # monitoring a run: observables (5-point gradient) and Phi for output
        _case("observe", "mixed", "real", (384, 360, 320), (19.2, 18.0, 16.0), 5e-4, 1, "observe_mixed_384x360x320",
              nu=(1.0, 1.0, 2.0), g=100.0, gdd=60.0, gradient5=True),
        # the allocation-free monitoring hook on the large grid
        _case("moments", "mixed", "real", (512, 512, 384), (25.6, 25.6, 19.2), 5e-4, 1, "moments_mixed_512x512x384"),
        # the 128^3 trap-schedule workload: its adjoint step in FP64 ...
        _case("adjoint", "fp64", "real", (128, 128, 128), (25.6,) * 3, 1e-3, 1, "adjoint_fp64_128", g=30.0, gdd=15.0),
        # ... and a short checkpointed trajectory's gradient in FP32 through autograd
        _case("gradient", "mixed", "real", (128, 128, 128), (25.6,) * 3, 1e-3, 5, "gradient_mixed_128",
              g=30.0, gdd=15.0, segments=4),
        # a parameter scan: independent condensates on uneven cubes in one batch
        _case("batch", "mixed", "imag", (128, 128, 128), (12.8,) * 3, 0.004, 20, "batch_mixed_16", members=16, pick=5,
              cubes="32 48 64 96 128"),
    ]


SIZES = [n for n in range(24, 513, 2)
         if any(n == 2 ** a * 3 ** b * 5 ** c * 7 ** d
                for a in range(1, 10) for b in range(6) for c in range(4) for d in range(4))]


def _shape(rng, low, high, points):
    """A shape of supported sizes, log-uniform per axis in [low, high], at most `points` points."""
    while True:
        s = tuple(min(SIZES, key=lambda n: abs(math.log(n) - t))
                  for t in (rng.uniform(math.log(low), math.log(high)) for _ in range(3)))
        if math.prod(s) <= points:
            return s


def draw(rng):
    kind = rng.choice(("step", "step", "step", "step", "observe", "moments", "adjoint", "gradient", "batch"))
    nu = tuple(round(rng.uniform(0.5, 2.0), 3) for _ in range(3))
    g = round(rng.uniform(5.0, 100.0), 3)
    gdd = round(rng.uniform(0.0, 0.9) * g, 3)
    opt = {"nu": nu, "g": g, "gdd": gdd}
    if kind == "step":
        prec = rng.choice(("mixed", "mixed", "fp64", "df64"))
        mode = rng.choice(("real", "imag"))
        shape = _shape(rng, 32, 512, {"mixed": 100_000_000, "fp64": 50_000_000, "df64": 50_000_000}[prec])
        steps = max(1, min(20, int(3e7 / math.prod(shape))))
        opt.update(simpson=rng.random() < 0.3, cutoff=8.0 if rng.random() < 0.3 else 0.0,
                   observables=rng.random() < 0.3)
    elif kind in ("observe", "moments"):
        prec, mode, steps = rng.choice(("mixed", "mixed", "fp64")), "real", 1
        shape = _shape(rng, 64, 512, 100_000_000 if prec == "mixed" else 50_000_000)
        opt.update(simpson=rng.random() < 0.5, gradient5=rng.random() < 0.5)
    elif kind == "adjoint":
        prec, mode, steps = rng.choice(("mixed", "fp64")), "real", 1
        shape = _shape(rng, 32, 256, 8_000_000)
    elif kind == "gradient":
        prec, mode, steps = rng.choice(("mixed", "mixed", "fp64")), "real", rng.randint(2, 5)
        shape = _shape(rng, 32, 160, 2_500_000)
        opt["segments"] = rng.randint(2, 4)
    else:
        prec, mode, steps = "mixed", rng.choice(("imag", "imag", "real")), rng.randint(5, 20)
        shape = (128, 128, 128)
        opt.update(members=rng.randint(4, 16), pick=rng.randrange(1, 1 << 16), cubes="32 40 48 56 64 80 96 112 120 128")
    box = tuple(round(rng.uniform(10.0, 26.0), 2) for _ in range(3))
    return _case(kind, prec, mode, shape, box, rng.choice((5e-4, 1e-3, 2e-3)), steps, **opt)


def _members(case):
    """Edge, interaction and trap of every member of a batch (part of the case, not of the seed)."""
    r = random.Random(case["pick"])
    out = []
    for _ in range(case["members"]):
        n = int(r.choice(case["cubes"].split()))
        g = r.uniform(5.0, 80.0)
        out.append({**case, "nx": n, "ny": n, "nz": n, "g": g, "gdd": r.uniform(0.0, 0.9) * g,
                    "nux": r.uniform(0.5, 2.0), "nuy": r.uniform(0.5, 2.0), "nuz": r.uniform(0.5, 2.0)})
    return out


def _geometry(case):
    n = (case["nx"], case["ny"], case["nz"])
    return n, tuple(length / k for length, k in zip((case["lx"], case["ly"], case["lz"]), n))


def _axis(n, h, device="cuda"):
    return (torch.arange(n, device=device, dtype=torch.float64) - n // 2) * h


def _psi(case, seed):
    """A trapped cloud with a seeded kick and noise, unit norm, in the boundary type."""
    n, h = _geometry(case)
    gen = torch.Generator(device="cuda").manual_seed(int(seed))
    kick = torch.rand(3, generator=gen, device="cuda", dtype=torch.float64) * 0.4 - 0.2
    line = []
    for d in range(3):
        x = _axis(n[d], h[d])
        nu = (case["nux"], case["nuy"], case["nuz"])[d]
        line.append(torch.exp(torch.complex(-0.35 * nu * x * x, kick[d] * x)))
    psi = line[0][:, None, None] * line[1][None, :, None] * line[2][None, None, :]
    psi.real.add_((torch.rand(n, generator=gen, device="cuda") * 2e-3 - 1e-3))
    psi /= math.sqrt(h[0] * h[1] * h[2]) * torch.linalg.vector_norm(torch.view_as_real(psi))
    return psi.to(torch.complex64 if case["precision"] == "mixed" else torch.complex128)


def _condensate(case):
    n, h = _geometry(case)
    return abi.Condensate(n, h, case["dt"], mode=MODE[case["mode"]], precision=PRECISION[case["precision"]],
                          nu=(case["nux"], case["nuy"], case["nuz"]), g=case["g"], gdd=case["gdd"],
                          cutoff=case["cutoff"], integration=abi.DGPE_SIMPSON if case["simpson"] else abi.DGPE_RECTANGLE,
                          kinetic=abi.DGPE_KINETIC_GRADIENT5 if case["gradient5"] else abi.DGPE_KINETIC_LAPLACIAN3)


def _schedule(case, seed):
    return np.random.RandomState(int(seed) % (1 << 31)).uniform(0.8, 1.2, case["segments"])


def _cotangent(case, psi):
    """A cotangent as later adjoint steps hand it on: 2 h^3 z^2 psi, out of phase with the state."""
    n, h = _geometry(case)
    z = _axis(n[2], h[2])
    return ((2.0 * h[0] * h[1] * h[2] * z * z * psi) * complex(math.cos(0.4), -math.sin(0.4))).to(psi.dtype)


def prepare(case, seed):
    s = {"case": case}
    if case["kind"] == "batch":
        s["members"] = [_condensate(m) for m in _members(case)]
        for i, (m, c) in enumerate(zip(_members(case), s["members"])):
            c.set_psi(_psi(m, int(seed) + 7919 * i))
        s["batch"] = abi.Batch(s["members"])
        return s
    s["psi"] = _psi(case, seed)
    if case["kind"] == "moments":
        n, h = _geometry(case)
        s["params"] = abi.make_params(n, h, case["dt"], MODE[case["mode"]], PRECISION[case["precision"]],
                                      integration=abi.DGPE_SIMPSON if case["simpson"] else abi.DGPE_RECTANGLE)
        s["out"] = torch.empty(4, dtype=torch.float64, device="cuda")
        return s
    s["solver"] = _condensate(case)
    if case["kind"] == "observe":
        s["solver"].set_psi(s["psi"])
    elif case["kind"] == "adjoint":
        s["gbar"] = _cotangent(case, s["psi"])
        s["solver"].adjoint_grads(reset=True)
    elif case["kind"] == "gradient":
        s["solver"].set_psi(s["psi"])
        s["nu"] = torch.from_numpy(_schedule(case, seed))
    return s


def run(s):
    case, kind = s["case"], s["case"]["kind"]
    if kind == "batch":
        s["batch"].step(case["steps"])
        return [c.get_psi(host=False) for c in s["members"]]
    if kind == "moments":
        abi.dgpe_moments_noalloc(s["psi"].data_ptr(), s["params"], s["out"].data_ptr(),
                                 torch.cuda.current_stream().cuda_stream)
        return s["out"]
    c = s["solver"]
    if kind == "step":
        c.set_psi(s["psi"])
        c.step(case["steps"])
        out = {"psi": c.get_psi(host=False)}
        if case["observables"]:
            out["observables"] = c.observables()
        return out
    if kind == "observe":
        return {"observables": c.observables(), "phi": c.phi(host=False)}
    if kind == "adjoint":
        gbar = s["gbar"].clone()
        c.adjoint_step(s["psi"], gbar)
        return {"gbar": gbar, "grads": c.adjoint_grads(reset=True)}
    nu = s["nu"].clone().requires_grad_()
    g = torch.tensor(case["g"], dtype=torch.float64, requires_grad=True)
    gdd = torch.tensor(case["gdd"], dtype=torch.float64, requires_grad=True)
    loss = abi.trajectory_z2(c, nu, g, gdd, case["steps"])
    loss.backward()
    return {"loss": loss.detach(), "nu": nu.grad, "g": g.grad, "gdd": gdd.grad}


def _step_flops(case):
    """One forward step, per grid point: the half-spectrum transforms, the phase, three sweeps."""
    n, _ = _geometry(case)
    points = math.prod(n)
    half = (n[2] // 2 + 1) / n[2]
    fft = 5.0 * math.log2(n[2]) + half * (10.0 * math.log2(n[0]) + 10.0 * math.log2(n[1]) + 2.0)
    return points * (fft + (38.0 + 3 * 22.0 if case["mode"] == "real" else 30.0 + 3 * 12.0))


def work(case):
    kind = case["kind"]
    if kind == "batch":
        each = [work({**m, "kind": "step"}) for m in _members(case)]
        return {k: sum(e[k] for e in each) for k in ("bytes", "flops")}
    points = case["nx"] * case["ny"] * case["nz"]
    size = 8 if case["precision"] == "mixed" else 16
    if kind == "step":
        return {"bytes": 2.0 * size * points * case["steps"], "flops": _step_flops(case) * case["steps"]}
    if kind == "observe":
        return {"bytes": 1.5 * size * points, "flops": _step_flops(case)}
    if kind == "moments":
        return {"bytes": float(size) * points, "flops": 8.0 * points}
    if kind == "adjoint":
        return {"bytes": 3.0 * size * points, "flops": 1.6 * _step_flops(case)}
    steps = case["steps"] * case["segments"]
    # the trajectory, its recomputation from checkpoints, and the adjoint steps
    return {"bytes": (2.0 + 2.0 + 3.0) * size * points * steps, "flops": 3.6 * _step_flops(case) * steps}


# ---- the same results from plain torch in 64 bits --------------------------------------
def _weights(case, n):
    w = torch.ones(n, dtype=torch.float64, device="cuda")
    if case["simpson"]:
        w[1::2], w[::2] = 4.0 / 3.0, 2.0 / 3.0
        w[0] = w[n - 2] = 1.0 / 3.0
        w[n - 1] = 0.0
    return w


class _Plain:
    """Split-step Crank-Nicolson with dense Cayley maps per axis and library transforms."""

    def __init__(self, case):
        self.case = case
        self.n, self.h = _geometry(case)
        self.x = [_axis(n, h) for n, h in zip(self.n, self.h)]
        self.dv = math.prod(self.h)
        self.w = [_weights(case, n) for n in self.n]
        k = [2.0 * math.pi * torch.fft.fftfreq(n, h, dtype=torch.float64, device="cuda") for n, h in zip(self.n, self.h)]
        k[2] = k[2][:self.n[2] // 2 + 1].abs()
        k2 = k[0][:, None, None] ** 2 + k[1][None, :, None] ** 2 + k[2][None, None, :] ** 2
        at0 = k2 == 0
        self.u = torch.where(at0, 0.0, 3.0 * (k[2] ** 2)[None, None, :] / torch.where(at0, 1.0, k2) - 1.0)
        if case["cutoff"] > 0:
            q = torch.sqrt(k2) * case["cutoff"]
            q = torch.where(at0, 1.0, q)
            series, term = torch.zeros_like(q), None
            for m in range(2, 12):
                term = (-1) ** m * 6.0 * m / math.factorial(2 * m + 1) * q ** (2 * m - 2)
                series = series + term
            self.u = self.u * torch.where(q < 0.5, series, 1.0 + 3.0 * torch.cos(q) / q ** 2 - 3.0 * torch.sin(q) / q ** 3)
        self.cayley = [self._cayley(n, h) for n, h in zip(self.n, self.h)]

    def _cayley(self, n, h):
        c = self.case["dt"] / (4.0 * h * h) * (1j if self.case["mode"] == "real" else 1.0)
        m = n - 2
        eye = torch.eye(m, dtype=torch.complex128, device="cuda")
        d = torch.diag(torch.ones(m - 1, dtype=torch.complex128, device="cuda"), 1)
        d = d + d.T - 2.0 * eye
        full = torch.zeros(n, n, dtype=torch.complex128, device="cuda")
        full[1:-1, 1:-1] = torch.linalg.solve(eye - c * d, eye + c * d)
        return full

    def phi(self, psi):
        dens = psi.real ** 2 + psi.imag ** 2
        return torch.fft.irfftn(torch.fft.rfftn(dens) * self.u, s=self.n)

    def trap(self, nuz):
        nu = (self.case["nux"], self.case["nuy"], nuz)
        v = [0.5 * a * a * x * x for a, x in zip(nu, self.x)]
        return v[0][:, None, None] + v[1][None, :, None] + v[2][None, None, :]

    def step(self, psi, nuz, g, gdd):
        dens = psi.real ** 2 + psi.imag ** 2
        theta = self.case["dt"] * (self.trap(nuz) + g * dens + gdd * self.phi(psi))
        psi = psi * (torch.exp(-1j * theta) if self.case["mode"] == "real" else torch.exp(-theta))
        n = self.n
        psi = torch.matmul(psi, self.cayley[2].T)
        psi = torch.matmul(self.cayley[1], psi)
        psi = torch.matmul(self.cayley[0], psi.reshape(n[0], -1)).reshape(n)
        return psi / torch.sqrt(self.norm(psi)) if self.case["mode"] == "imag" else psi

    def sum(self, f):
        return torch.einsum("ijk,i,j,k->", f, *self.w)

    def norm(self, psi):
        return self.dv * self.sum(psi.real ** 2 + psi.imag ** 2)

    def moments(self, psi):
        dens = psi.real ** 2 + psi.imag ** 2
        total = self.sum(dens)
        sq = []
        for d in range(3):
            shape = [1, 1, 1]
            shape[d] = -1
            sq.append(torch.sqrt(self.sum(dens * (self.x[d] ** 2).reshape(shape)) / total))
        return self.dv * total, sq

    def shifted(self, psi, d, k):
        out = torch.zeros_like(psi)
        m = self.n[d] - abs(k)
        out.narrow(d, max(0, -k), m).copy_(psi.narrow(d, max(0, k), m))
        return out

    def observables(self, psi):
        case = self.case
        dens = psi.real ** 2 + psi.imag ** 2
        kin = torch.zeros_like(dens)
        for d in range(3):
            f = {k: self.shifted(psi, d, k) for k in ((-2, -1, 1, 2) if case["gradient5"] else (-1, 1))}
            if case["gradient5"]:
                kin += 0.5 * torch.abs((f[-2] - 8.0 * f[-1] + 8.0 * f[1] - f[2]) / (12.0 * self.h[d])) ** 2
            else:
                kin -= 0.5 * (psi.conj() * (f[-1] - 2.0 * psi + f[1])).real / self.h[d] ** 2
        e_kin, e_trap = self.dv * self.sum(kin), self.dv * self.sum(self.trap(case["nuz"]) * dens)
        e_con = 0.5 * self.dv * case["g"] * self.sum(dens * dens)
        e_dip = 0.5 * self.dv * case["gdd"] * self.sum(self.phi(psi) * dens)
        norm, rms = self.moments(psi)
        got = (norm, (e_kin + e_trap + 2.0 * (e_con + e_dip)) / norm, e_kin + e_trap + e_con + e_dip, e_kin, e_trap, e_con, e_dip)
        return {**{k: float(v) for k, v in zip(OBS, got)}, "rms": tuple(float(v) for v in rms)}


def exact(case, seed):
    kind = case["kind"]
    if kind == "batch":
        out = []
        for i, m in enumerate(_members(case)):
            p, psi = _Plain(m), _psi(m, int(seed) + 7919 * i).to(torch.complex128)
            for _ in range(case["steps"]):
                psi = p.step(psi, m["nuz"], m["g"], m["gdd"])
            out.append(psi)
        return out
    p, psi = _Plain(case), _psi(case, seed)
    wide = psi.to(torch.complex128)
    if kind == "moments":
        norm, rms = p.moments(wide)
        return torch.stack([norm, *rms])
    if kind == "step":
        for _ in range(case["steps"]):
            wide = p.step(wide, case["nuz"], case["g"], case["gdd"])
        out = {"psi": wide}
        if case["observables"]:
            out["observables"] = p.observables(wide)
        return out
    if kind == "observe":
        return {"observables": p.observables(wide), "phi": p.phi(wide)}
    nu, segments = [torch.tensor(case["nuz"], dtype=torch.float64, device="cuda", requires_grad=True)], 1
    if kind == "gradient":
        nu = [torch.tensor(v, device="cuda", requires_grad=True) for v in _schedule(case, seed)]
        segments = case["segments"]
    g = torch.tensor(case["g"], dtype=torch.float64, device="cuda", requires_grad=True)
    gdd = torch.tensor(case["gdd"], dtype=torch.float64, device="cuda", requires_grad=True)
    if kind == "adjoint":
        wide.requires_grad_()
        got = p.step(wide, nu[0], g, gdd)
        # dL = Re sum conj(gbar) dpsi is torch's convention for the gradient of a real loss
        got.backward(_cotangent(case, psi).to(torch.complex128))
        return {"gbar": wide.grad, "grads": torch.stack([g.grad, gdd.grad, nu[0].grad])}
    for s in range(segments):
        for _ in range(case["steps"]):
            wide = p.step(wide, nu[s], g, gdd)
    loss = p.dv * torch.sum((wide.real ** 2 + wide.imag ** 2) * p.x[2] ** 2)
    loss.backward()
    return {"loss": loss.detach(), "nu": torch.stack([v.grad for v in nu]), "g": g.grad, "gdd": gdd.grad}
