"""Workloads for timing: the calls a user's program makes, with the sizes of this
repository's own configurations, tests and benchmark.

A pass advances a simulation by the steps between two diagnostics and reads the
state back (fields and particles, into buffers the program keeps), runs an
ensemble, or takes an objective with its gradients.  ``exact`` repeats a pass in
plain torch, 64 bits, on the same inputs.

Normalised units (c = m_e = e = 1, k0 = 1): dx1 = 2 pi/32, dx2 = dx3 = 4 dx1.
"""
from __future__ import annotations

import math

import numpy as np
import torch

from paper_2004_03754_gb300 import autodiff, coeffs, inputs
from paper_2004_03754_gb300 import pic as P

DX = (inputs.DX1, inputs.DX2, inputs.DX2)
FIELDS = ("e1", "e2", "e3", "b1", "b2", "b3")
LENV = 20 * math.pi           # pulse length: ten wavelengths (320 cells)


# ---------------------------------------------------------------------------
# the cases
# ---------------------------------------------------------------------------
def _sim(name, n, precision, pusher, ppc, steps, a0, ratio=0.5, solver="proposed16", w0=20.0,
         density=0.01, uth=0.001):
    n = tuple(n) + (0,) * (3 - len(n))
    return dict(name=name, kind="step", n1=n[0], n2=n[1], n3=n[2], precision=precision,
                pusher=pusher, ppc=ppc, steps=steps, a0=float(a0), ratio=ratio, solver=solver,
                w0=float(w0), density=density, uth=uth)


def listed():
    return [
        # the smallest grid that is used (smoke test, unit tests): launches and latency
        _sim("tiny_2d_fp64", (64, 16), "fp64", "boris", 1, 2, 1.0, w0=0.0),
        # the plain-method configuration: 512 x 128, one test electron ahead of the pulse
        _sim("single_electron_2d_fp64", (512, 128), "fp64", "boris", 0, 20, 1.0),
        # the benchmark's workload: 29 million electrons, FP32 fields and FP64 pusher
        _sim("plasma_2d_mixed", (4096, 1024), "mixed", "boris", 8, 10, 4.0),
        # the same plasma in plain FP64, at the size used for profiling
        _sim("plasma_2d_fp64", (2048, 512), "fp64", "boris", 8, 9, 4.0),
        # a strong pulse with compensated (FP32-pair) fields and the analytic pusher
        _sim("strong_2d_compensated", (2048, 512), "compensated", "analytic", 2, 9, 100.0),
        # odd row lengths, dt/dx1 = 1/4 (the current correction runs), Higuera-Cary pusher
        _sim("ragged_2d_mixed_quarter", (1501, 389), "mixed", "hc", 4, 12, 10.0, ratio=0.25),
        # the 3D workload: 84 million cold electrons, analytic pusher
        _sim("plasma_3d_mixed", (1024, 256, 256), "mixed", "analytic", 2, 2, 10.0, w0=30.0,
             density=0.005, uth=0.0),
        # a ragged 3D box in plain FP64
        _sim("ragged_3d_fp64", (301, 60, 44), "fp64", "boris", 2, 4, 4.0, w0=15.0),
        # an ensemble of uneven vacuum runs with 16 test electrons each, a0 from 3 to 100
        # (beyond that FP32 fields don't hold the electrons' energy)
        dict(name="ensemble_2d_mixed", kind="ensemble", nruns=16, sizes=inputs.DEFAULT_SEED,
             steps=1024, precision="mixed", pusher="analytic"),
        # energy objective and its laser gradients by the adjoint, 64 test electrons
        dict(name="adjoint_2d_fp64", kind="adjoint", n1=1024, n2=256, electrons=64, steps=200,
             every=50, a0=10.0, pusher="boris"),
    ]


def _log(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def _cost(c):
    """Rough seconds of a step case on a GB300, to keep drawn cases below the largest listed one."""
    n = [c[k] for k in ("n1", "n2", "n3") if c[k]]
    cell = {"mixed": 0.05e-9, "fp64": 0.6e-9, "compensated": 0.4e-9}[c["precision"]]
    push = {"mixed": 0.12e-9, "fp64": 0.8e-9, "compensated": 0.4e-9}[c["precision"]]
    push *= (4 if len(n) == 3 else 1) * {"boris": 1.0, "hc": 1.5, "analytic": 2.0}[c["pusher"]]
    return c["steps"] * math.prod(n) * (cell + c["ppc"] * push)


def draw(rng):
    kind = rng.choice(["step2", "step2", "step2", "step3", "step3", "ensemble", "adjoint"])
    pusher = rng.choice(["boris", "analytic", "hc"])
    precision = rng.choice(["mixed", "mixed", "fp64", "compensated"])
    a0 = float(_log(rng, 1, 100))
    if kind == "step2":
        n = (_log(rng, 64, 4096), _log(rng, 16, 1024))
        if rng.random() < 0.5:
            n = (n[0] // 32 * 32, n[1])
        ratio, solver = rng.choice([(0.5, "proposed16"), (0.5, "proposed16"), (0.25, "proposed16"),
                                    (0.5, "yee"), (0.5, "proposed8")])
        c = _sim("", n, precision, pusher, rng.choice([0, 1, 2, 4, 8]), rng.randint(2, 12), a0,
                 ratio=ratio, solver=solver, w0=rng.choice([0.0, 20.0]))
    elif kind == "step3":
        n = (_log(rng, 64, 768), _log(rng, 16, 192), _log(rng, 16, 192))
        if rng.random() < 0.5:
            n = (n[0] // 32 * 32, n[1], n[2])
        c = _sim("", n, precision, pusher, rng.choice([0, 1, 2]), rng.randint(1, 4), a0,
                 w0=rng.choice([0.0, 15.0]), density=0.005, uth=rng.choice([0.0, 0.001]))
    elif kind == "ensemble":
        c = dict(kind="ensemble", nruns=_log(rng, 4, 24), sizes=rng.randrange(1 << 30),
                 steps=_log(rng, 64, 512), precision="mixed", pusher=rng.choice(["boris", "analytic"]))
    else:
        c = dict(kind="adjoint", n1=_log(rng, 400, 1024), n2=_log(rng, 16, 256),
                 electrons=_log(rng, 4, 256), steps=_log(rng, 40, 200), every=rng.choice([25, 50]),
                 a0=float(_log(rng, 1, 30)), pusher=rng.choice(["boris", "analytic"]))
    while c["kind"] == "step" and _cost(c) > 0.05:
        if c["ppc"] > 1:
            c["ppc"] //= 2
        elif c["steps"] > 2:
            c["steps"] -= 1
        else:
            c["n2"] = c["n2"] // 2 + 1
    c.pop("name", None)
    return c


# ---------------------------------------------------------------------------
# inputs (on the GPU, from the seed alone)
# ---------------------------------------------------------------------------
def _device():
    return "cuda" if torch.cuda.is_available() else "cpu"


def _rng(seed):
    return torch.Generator(device=_device()).manual_seed(int(seed))


def _table(case):
    s = case.get("solver", "proposed16")
    if s == "yee":
        return np.array([1.0]), np.array([1.0])
    if s == "proposed8":
        return coeffs.load("proposed", 8, 0.5, 0.4)
    return coeffs.load("proposed", 16, case.get("ratio", 0.5), 0.3)


def _grid(case):
    n = tuple(case[k] for k in ("n1", "n2", "n3") if case.get(k))
    return n, DX[:len(n)], case.get("ratio", 0.5) * inputs.DX1


def _pulse_cells(case):
    return min(320, case["n1"] * 5 // 8)


def _step_inputs(case, seed):
    """Fields E^0, B^{-1/2} of a sin^2 pulse (continuous wave, Gaussian across) and the
    electrons: a uniform plasma from the pulse's front on, or one test electron."""
    n, dx, dt = _grid(case)
    dev, g, nd = _device(), _rng(seed), len(n)
    cells = _pulse_cells(case)
    L, front = cells * dx[0], (cells + 15 if case["n1"] > 400 else cells) * dx[0]
    phase = 2 * math.pi * float(torch.rand(1, generator=g, device=dev, dtype=torch.float64))
    x1 = torch.arange(n[0], device=dev, dtype=torch.float64) * dx[0]

    def wave(x):
        phi = front - x
        s, c = torch.sin(math.pi * phi / L), torch.cos(math.pi * phi / L)
        v = -case["a0"] * (2 * s * c * (math.pi / L) * torch.sin(phi + phase) +
                           s * s * torch.cos(phi + phase))
        return torch.where((phi > 0) & (phi < L), v, torch.zeros_like(v))

    tr = torch.ones((1,) * (nd - 1) + (1,), device=dev, dtype=torch.float64)
    if case["w0"] > 0:
        for d in range(1, nd):   # E2 and B3 sit at x2 = (j + 1/2) dx2, x3 = k dx3
            x = (torch.arange(n[d], device=dev, dtype=torch.float64) + (0.5 if d == 1 else 0.0)) * dx[d]
            t = torch.exp(-((x - n[d] * dx[d] / 2) / case["w0"]) ** 2)
            tr = tr * t.reshape((1,) * (nd - 1 - d) + (-1,) + (1,) * d)
    shape = tuple(reversed(n))
    F = [torch.zeros(shape, device=dev, dtype=torch.float64) for _ in range(6)]
    F[1] = (wave(x1) * tr).expand(shape).contiguous()
    F[5] = (wave(x1 + dx[0] / 2 + dt / 2) * tr).expand(shape).contiguous()
    if case["ppc"] == 0:
        pos = [front + 16 * dx[0]] + [n[d] * dx[d] / 2 for d in range(1, nd)]
        X = torch.tensor([[p % (n[d] * dx[d])] for d, p in enumerate(pos)], device=dev,
                         dtype=torch.float64)
        U, W = torch.zeros((3, 1), device=dev, dtype=torch.float64), torch.zeros(1, device=dev, dtype=torch.float64)
        return F, X, U, W
    # plasma cells: from the pulse's front, vacuum before the box ends
    lo = min(int(round(front / dx[0])), n[0] - 8) if case["n1"] > 400 else 0
    hi = n[0] - 256 if case["n1"] >= 1500 else (896 if n[0] == 1024 else n[0])
    ppc, ncell = case["ppc"], (hi - lo) * math.prod(n[1:])
    c = torch.arange(ncell, device=dev, dtype=torch.int64).repeat_interleave(ppc)
    X = torch.rand((nd, ncell * ppc), generator=g, device=dev, dtype=torch.float64)
    X[0] += lo + c % (hi - lo)
    c = torch.div(c, hi - lo, rounding_mode="floor")
    for d in range(1, nd):
        X[d] += c % n[d]
        c = torch.div(c, n[d], rounding_mode="floor")
    for d in range(nd):
        X[d] *= dx[d]
        X[d].clamp_(max=math.nextafter(n[d] * dx[d], 0.0))
    U = torch.zeros((3, ncell * ppc), device=dev, dtype=torch.float64)
    if case["uth"] > 0:
        U.normal_(0.0, case["uth"], generator=g)
    W = torch.full((ncell * ppc,), -case["density"] / ppc, device=dev, dtype=torch.float64)
    return F, X, U, W


def _ensemble_inputs(case, seed):
    n1, n2, _ = inputs.ensemble(case["nruns"], case["sizes"])   # the grids are the case's
    _, _, a0 = inputs.ensemble(case["nruns"], seed)
    at = inputs.rng(seed + 1).random((case["nruns"], 16, 2))
    runs, x = [], []
    for r in range(case["nruns"]):
        cells = min(320, int(n1[r]) // 2)
        front = (cells + 4) * DX[0]
        runs.append(dict(a0=float(a0[r]) ** 0.5, L=cells * DX[0], front=front))
        x.append([[front + (16 + 2 * (i + at[r, i, 0])) * DX[0], (i + at[r, i, 1]) * n2[r] * DX[1] / 16]
                  for i in range(16)])
    X = np.ascontiguousarray(np.array(x).reshape(-1, 2).T)
    return n1, n2, runs, X


def _adjoint_inputs(case, seed):
    g = inputs.rng(seed)
    cells, k = _pulse_cells(case), case["electrons"]
    front = (cells + 10) * DX[0]
    room = min(200, case["n1"] - cells - 20)
    x = np.concatenate([(cells + 10 + room * g.random(k)) * DX[0], g.random(k) * case["n2"] * DX[1]])
    return cells * DX[0], front, x, np.zeros(3 * k), float(g.uniform(0, 2 * np.pi))


# ---------------------------------------------------------------------------
# the calls
# ---------------------------------------------------------------------------
_STREAM = []


def _stream():
    """One stream for all work, as a program with one simulation loop has."""
    if not _STREAM:
        _STREAM.append(torch.cuda.Stream())
    return _STREAM[0].cuda_stream


def prepare(case, seed):
    if case["kind"] == "step":
        n, dx, dt = _grid(case)
        F, X, U, W = _step_inputs(case, seed)
        cE, cB = _table(case)
        sim = P.Simulation(n, dx, dt, cE, cB, precision=case["precision"], pusher=case["pusher"],
                           stream=_stream())
        torch.cuda.synchronize()
        for name, f in zip(FIELDS, F):
            sim.load_field(name, f)
        P.pic_load_particles(sim.ctx, W.numel(), X, U, W, -1.0)
        sim.sync()
        out = {name: torch.empty_like(F[0]) for name in FIELDS}
        out["x"], out["u"] = torch.empty_like(X), torch.empty_like(U)
        torch.cuda.synchronize()
        return dict(kind="step", sim=sim, steps=case["steps"], out=out)
    if case["kind"] == "ensemble":
        n1, n2, runs, X = _ensemble_inputs(case, seed)
        cE, cB = _table(case)
        ens = P.Ensemble(n1, n2, DX[:2], inputs.DT, cE, cB, precision=case["precision"],
                         pusher=case["pusher"], stream=_stream())
        ens.load_lasers([P.pic_laser(r["a0"], 1.0, 0.0, r["L"], r["front"], 0.0, 0.0, 0.0) for r in runs])
        k = X.shape[1]
        ens.load_particles([16] * case["nruns"], [X[0], X[1]], [np.zeros(k)] * 3, np.zeros(k))
        ens.set_steps([case["steps"]] * case["nruns"])
        return dict(kind="ensemble", ens=ens)
    L, front, x, u, phase = _adjoint_inputs(case, seed)
    n, dx, dt = _grid(case)
    cE, cB = _table(case)
    sim = P.Simulation(n, dx, dt, cE, cB, precision="fp64", pusher=case["pusher"], stream=_stream())
    laser = dict(L_env=L, x_front=front, x2c=n[1] * dx[1] / 2)
    return dict(kind="adjoint", sim=sim, laser=laser, x=x, u=u, a0=case["a0"], phase=phase,
                steps=case["steps"], every=case["every"])


def run(state):
    if state["kind"] == "step":
        sim, out = state["sim"], state["out"]
        sim.step(state["steps"])
        for name in FIELDS:
            sim.read_field(name, out[name])
        P.pic_read_particles(sim.ctx, out["x"], out["u"], None)
        return out
    if state["kind"] == "ensemble":
        ens = state["ens"]
        ens.run()
        x, u, _ = ens.read_particles()
        return dict(x=x, u=u, e2=[ens.read_field(r, "e2") for r in range(ens.nruns)],
                    b3=[ens.read_field(r, "b3") for r in range(ens.nruns)])
    a0 = torch.tensor(state["a0"], dtype=torch.float64, requires_grad=True)
    phase = torch.tensor(state["phase"], dtype=torch.float64, requires_grad=True)
    J = autodiff.LaserEnergy.apply(a0, phase, state["sim"], state["laser"], state["x"], state["u"],
                                   state["steps"], state["every"])
    J.backward()
    return dict(J=J.detach(), a0=a0.grad, phase=phase.grad)


def work(case):
    if case["kind"] == "step":
        n, _, _ = _grid(case)
        nd, cells, s = len(n), math.prod(n), case["steps"]
        ts = 4 if case["precision"] == "mixed" else 8
        if case["ppc"] == 0:
            parts = 1
        else:
            lo = min(_pulse_cells(case) + 15, n[0] - 8) if n[0] > 400 else 0
            hi = n[0] - 256 if n[0] >= 1500 else (896 if n[0] == 1024 else n[0])
            parts = (hi - lo) * math.prod(n[1:]) * case["ppc"]
        # per step: E and B read and written, the current written and read; x, u read and
        # written, w read.  Then the read-back in 64 bits.
        step = cells * 18 * ts + parts * 8 * (2 * (nd + 3) + 1)
        back = cells * 6 * (ts + 8) + parts * 16 * (nd + 3)
        push = {"boris": 70, "hc": 110, "analytic": 300}[case["pusher"]]
        interp = {2: 2 * 6 * 12 + 200, 3: 2 * 6 * 39 + 700}[nd]
        return {"bytes": s * step + back, "flops": s * (cells * {2: 214, 3: 226}[nd] + parts * (push + interp))}
    if case["kind"] == "ensemble":
        n1, n2, _ = inputs.ensemble(case["nruns"], case["sizes"])
        cells = float((n1 * n2).sum())
        return {"bytes": case["steps"] * cells * 48.0 + cells * 16.0, "flops": case["steps"] * cells * 208.0}
    cells = case["n1"] * case["n2"]
    # forward and reverse: the field step each way, and the states that the reverse reads
    return {"bytes": case["steps"] * cells * 8.0 * (12 + 6 + 18), "flops": case["steps"] * cells * 3.0 * 208}


# ---------------------------------------------------------------------------
# a pass in plain torch, 64 bits
# ---------------------------------------------------------------------------
class _Box:
    """Grid, stencils and the update of Eq. (1) on arrays (x1 last); boxes uniform across
    may hold one row (n2 = 1) with the true length L2 of the axis."""

    def __init__(self, n, dx, dt, cE, cB, L=None):
        self.n, self.dx, self.dt, self.nd = n, dx, dt, len(n)
        self.cE, self.cB = [float(v) for v in cE], [float(v) for v in cB]
        self.L = L or [a * b for a, b in zip(n, dx)]
        self.mat = None
        if n[0] <= 2048 and math.prod(n) * n[0] <= 1 << 30:   # circulant matrices
            self.mat = [torch.zeros((n[0], n[0]), device=_device(), dtype=torch.float64) for _ in range(2)]
            i = torch.arange(n[0], device=_device())
            for m, c in enumerate(self.cE, 1):
                self._tap(0, i, i + m, c)
                self._tap(0, i, i - m + 1, -c)
            for m, c in enumerate(self.cB, 1):
                self._tap(1, i, i + m - 1, c)
                self._tap(1, i, i - m, -c)

    def _tap(self, which, i, j, c):
        self.mat[which].index_put_((j % self.n[0], i), torch.full_like(self.mat[which][0], c / self.dx[0]),
                                   accumulate=True)

    def d1(self, f, which):
        if self.mat is not None:
            return f @ self.mat[which]
        o = torch.zeros_like(f)
        for m, c in enumerate((self.cE, self.cB)[which], 1):
            a, b = (m, m - 1) if which == 0 else (m - 1, m)
            o.add_(torch.roll(f, -a, -1) - torch.roll(f, b, -1), alpha=c / self.dx[0])
        return o

    def d(self, f, axis, which):
        """Derivative along axis 2 or 3: forward on E (which 0), backward on B."""
        if axis == 3 and self.nd == 2:
            return 0.0
        a = -axis
        return (torch.roll(f, -1, a) - f if which == 0 else f - torch.roll(f, 1, a)) / self.dx[axis - 1]

    def curl(self, f, w):
        return [self.d(f[2], 2, w) - self.d(f[1], 3, w), self.d(f[0], 3, w) - self.d1(f[2], w),
                self.d1(f[1], w) - self.d(f[0], 2, w)]

    def correct(self, J1):
        """J1 times [k]_Yee/[k]_B1 per x1 mode."""
        if self.cB[0] == 1.0 and not any(self.cB[1:]):
            return J1
        k = 2 * math.pi * torch.arange(self.n[0] // 2 + 1, device=J1.device, dtype=torch.float64) / self.L[0]
        kB = sum(c * torch.sin((2 * j - 1) * k * self.dx[0] / 2) for j, c in enumerate(self.cB, 1))
        r = torch.sin(k * self.dx[0] / 2) / kB
        r[0] = 1.0 / sum((2 * j - 1) * c for j, c in enumerate(self.cB, 1))
        return torch.fft.irfft(torch.fft.rfft(J1) * r, n=self.n[0])

    def flat(self, node):
        """Flat index of the nodes (one tensor per axis), broadcast."""
        q = node[0] % self.n[0]
        m = self.n[0]
        for d in range(1, self.nd):
            q = q + (node[d] % self.n[d]) * m
            m *= self.n[d]
        return q


def _spline(s):
    """Nearest node and the three weights of the quadratic B-spline."""
    i = torch.floor(s + 0.5)
    d = s - i
    return i.to(torch.int64), torch.stack([0.5 * (0.5 - d) ** 2, 0.75 - d * d, 0.5 * (0.5 + d) ** 2])


def _gather(box, f, X, half):
    ax = [_spline(X[d] / box.dx[d] - 0.5 * half[d]) for d in range(box.nd)]
    acc = 0.0
    for k in range(3 if box.nd == 3 else 1):
        for j in range(3):
            for i in range(3):
                node, w = [ax[0][0] + i - 1, ax[1][0] + j - 1], ax[0][1][i] * ax[1][1][j]
                if box.nd == 3:
                    node.append(ax[2][0] + k - 1)
                    w = w * ax[2][1][k]
                acc = acc + w * f.reshape(-1)[box.flat(node)]
    return acc


def _cross(a, b):
    return torch.stack([a[1] * b[2] - a[2] * b[1], a[2] * b[0] - a[0] * b[2], a[0] * b[1] - a[1] * b[0]])


def _boris(E, B, u, qm, dt):
    h = 0.5 * qm * dt
    um = u + h * E
    t = h * B / torch.sqrt(1 + (um * um).sum(0))
    up = um + _cross(um + _cross(um, t), 2 * t / (1 + (t * t).sum(0)))
    return up + h * E


def _hc(E, B, u, qm, dt):
    h = 0.5 * qm * dt
    um, b = u + h * E, h * B
    b2, us = (b * b).sum(0), (um * b).sum(0)
    sigma = 1 + (um * um).sum(0) - b2
    t = b / torch.sqrt(0.5 * (sigma + torch.sqrt(sigma ** 2 + 4 * (b2 + us ** 2))))
    w = (um + (um * t).sum(0) * t + _cross(um, t)) / (1 + (t * t).sum(0))
    return w + _cross(w, t) + h * E


def _analytic(E, B, u, qm, dt):
    """exp(L tau) U by its power series in tau, t(tau) = dt by Newton."""
    e, b = qm * E, qm * B
    V = [torch.cat([torch.sqrt(1 + (u * u).sum(0, keepdim=True)), u])]
    for _ in range(40):
        v = V[-1]
        V.append(torch.cat([(e * v[1:]).sum(0, keepdim=True), v[0] * e + _cross(v[1:], b)]))
    tau = dt / V[0][0]
    for _ in range(12):
        t, c = torch.zeros_like(tau), torch.ones_like(tau)
        gam = torch.zeros_like(tau)
        for k, v in enumerate(V):
            gam = gam + v[0] * c
            c = c * tau / (k + 1)
            t = t + v[0] * c
        tau = tau - (t - dt) / gam
    out, c = torch.zeros_like(u), torch.ones_like(tau)
    for k, v in enumerate(V):
        out = out + v[1:] * c
        c = c * tau / (k + 1)
    return out


_PUSH = {"boris": _boris, "hc": _hc, "analytic": _analytic}
_HALF = ((1, 0, 0), (0, 1, 0), (0, 0, 1), (0, 1, 1), (1, 0, 1), (1, 1, 0))


def _deposit(box, J, W, X, delta, v3):
    """Esirkepov current of the moves X -> X + delta dx (delta in cells)."""
    nd, base, S0, dS = box.nd, [], [], []
    for d in range(nd):
        s = X[d] / box.dx[d]
        i0, w0 = _spline(s)
        i1, w1 = _spline(s + delta[d])
        b = torch.minimum(i0, i1) - 1
        z = torch.zeros((4,) + s.shape, device=s.device, dtype=torch.float64)
        at = torch.arange(3, device=s.device).reshape(3, 1)
        a0 = z.scatter(0, at + (i0 - 1 - b), w0)
        dS.append(z.scatter(0, at + (i1 - 1 - b), w1) - a0)
        base.append(b)
        S0.append(a0)

    def add(c, node, v):
        J[c].reshape(-1).index_add_(0, box.flat([base[d] + node[d] for d in range(nd)]), v)

    third = 1.0 / 3.0
    if nd == 2:
        for q in range(4):
            for d, a in ((0, 1), (1, 0)):
                run = 0.0
                for m in range(3):
                    run = run - W * (box.dx[d] / box.dt) * dS[d][m] * (S0[a][q] + 0.5 * dS[a][q])
                    add(d, (m, q) if d == 0 else (q, m), run)
            for p in range(4):
                w3 = (S0[0][p] * S0[1][q] + 0.5 * dS[0][p] * S0[1][q] + 0.5 * S0[0][p] * dS[1][q] +
                      third * dS[0][p] * dS[1][q])
                add(2, (p, q), W * v3 * w3)
        return
    for d in range(3):
        a, c = (d + 1) % 3, (d + 2) % 3
        for q in range(4):
            for p in range(4):
                pre = (S0[a][p] * S0[c][q] + 0.5 * dS[a][p] * S0[c][q] + 0.5 * S0[a][p] * dS[c][q] +
                       third * dS[a][p] * dS[c][q])
                run = 0.0
                for m in range(3):
                    run = run - W * (box.dx[d] / box.dt) * dS[d][m] * pre
                    node = [0, 0, 0]
                    node[d], node[a], node[c] = m, p, q
                    add(d, node, run)


def _advance(box, F, X, U, W, pusher, steps, qm=-1.0, chunk=1 << 22):
    """`steps` full steps; F = [E1..B3]; X, U in load order."""
    E, B = list(F[:3]), list(F[3:])
    plasma = W is not None and bool((W != 0).any())
    for _ in range(steps):
        curl = box.curl(E, 0)
        bbar = [b - 0.5 * box.dt * c for b, c in zip(B, curl)]
        J = [torch.zeros_like(E[0]) for _ in range(3)] if plasma else [0.0] * 3
        xs, us = [], []
        for k in range(0, X.shape[1], chunk):
            x, u = X[:, k:k + chunk], U[:, k:k + chunk]
            eb = [_gather(box, f, x, h) for f, h in zip(E + bbar, _HALF)]
            u = _PUSH[pusher](torch.stack(eb[:3]), torch.stack(eb[3:]), u, qm, box.dt)
            v = u / torch.sqrt(1 + (u * u).sum(0))
            if plasma:
                delta = [box.dt * v[d] / box.dx[d] for d in range(box.nd)]
                _deposit(box, J, W[k:k + chunk], x, delta, v[2])
            x = torch.stack([x[d] + box.dt * v[d] for d in range(box.nd)])
            L = torch.tensor(box.L[:box.nd], device=x.device, dtype=torch.float64).reshape(-1, 1)
            xs.append(x - L * torch.floor(x.detach() / L))
            us.append(u)
        X, U = torch.cat(xs, 1), torch.cat(us, 1)
        if plasma:
            J[0] = box.correct(J[0])
        B = [b - box.dt * c for b, c in zip(B, curl)]
        E = [e + box.dt * (c - j) for e, c, j in zip(E, box.curl(B, 1), J)]
    return E + B, X, U


def _laser_rows(n1, dt, cE, cB, a0, phase, L, front):
    """x1 profiles of E2^0 and its discrete forward partner B3^{-1/2} (Eq. (8))."""
    dev, dx = _device(), DX[0]
    i = torch.arange(n1, device=dev, dtype=torch.float64)
    phi = torch.remainder(front - i * dx, n1 * dx)
    s, c = torch.sin(math.pi * phi / L), torch.cos(math.pi * phi / L)
    e = -a0 * (2 * s * c * (math.pi / L) * torch.sin(phi + phase) + s * s * torch.cos(phi + phase))
    e = torch.where((phi > 0) & (phi < L), e, torch.zeros_like(e))
    k = 2 * math.pi * torch.arange(n1 // 2 + 1, device=dev, dtype=torch.float64) / (n1 * dx)
    kE, kB = (sum(float(v) * torch.sin((2 * j - 1) * k * dx / 2) for j, v in enumerate(t, 1)) * 2 / dx
              for t in (cE, cB))
    om = 2 / dt * torch.asin(torch.clamp(0.5 * dt * torch.sqrt(kE * kB), max=1.0))
    ratio = kE / (torch.sin(om * dt / 2) * 2 / dt)
    ratio[0] = 1.0
    if n1 % 2 == 0:
        ratio[-1] = 0.0
    b = torch.fft.irfft(torch.fft.rfft(e) * ratio * torch.exp(1j * (k * dx / 2 + om * dt / 2)), n=n1)
    return e, b


def _exact_ensemble(case, seed):
    # the runs are uniform across, so one row each, all rows in one array
    n1, n2, runs, X = _ensemble_inputs(case, seed)
    cE, cB = _table(case)
    dev, dt, R = _device(), inputs.DT, case["nruns"]
    off = np.concatenate([[0], np.cumsum(n1)])
    rows = [_laser_rows(int(n1[r]), dt, cE, cB, runs[r]["a0"], 0.0, runs[r]["L"], runs[r]["front"])
            for r in range(R)]
    e2, b3 = (torch.cat([r[k] for r in rows]) for k in range(2))
    start = torch.as_tensor(np.repeat(off[:-1], n1), device=dev)
    width = torch.as_tensor(np.repeat(n1, n1), device=dev)
    i = torch.arange(int(off[-1]), device=dev) - start
    m = torch.arange(1, len(cE) + 1, device=dev)

    def at(j):
        return start[:, None] + (i[:, None] + j) % width[:, None]

    tabE, tabB = (at(m), at(1 - m)), (at(m - 1), at(-m))
    wE, wB = (torch.as_tensor(np.array(c), device=dev) / DX[0] for c in (cE, cB))
    po, pw = (torch.as_tensor(np.repeat(a, 16).astype(np.int64), device=dev) for a in (off[:-1], n1))
    x, u = torch.as_tensor(X, device=dev).clone(), torch.zeros((3, X.shape[1]), device=dev, dtype=torch.float64)
    L = torch.stack([pw * DX[0], torch.as_tensor(np.repeat(n2, 16), device=dev) * DX[1]])
    z = torch.zeros_like(u[0])
    for _ in range(case["steps"]):
        d = (e2[tabE[0]] - e2[tabE[1]]) @ wE
        bb = b3 - 0.5 * dt * d
        node, w = _spline(x[0] / DX[0])
        E = sum(w[q] * e2[po + (node + q - 1) % pw] for q in range(3))
        node, w = _spline(x[0] / DX[0] - 0.5)
        B = sum(w[q] * bb[po + (node + q - 1) % pw] for q in range(3))
        u = _PUSH[case["pusher"]](torch.stack([z, E, z]), torch.stack([z, z, B]), u, -1.0, dt)
        x = x + dt * u[:2] / torch.sqrt(1 + (u * u).sum(0))
        x = x - L * torch.floor(x / L)
        b3 = b3 - dt * d
        e2 = e2 - dt * ((b3[tabB[0]] - b3[tabB[1]]) @ wB)

    def rows_of(f):
        f = f.cpu().numpy()
        return [np.ascontiguousarray(np.broadcast_to(f[off[r]:off[r + 1]], (int(n2[r]), int(n1[r]))))
                for r in range(R)]

    return dict(x=[v.cpu().numpy() for v in x], u=[v.cpu().numpy() for v in u], e2=rows_of(e2), b3=rows_of(b3))


def exact(case, seed):
    if case["kind"] == "step":
        n, dx, dt = _grid(case)
        F, X, U, W = _step_inputs(case, seed)
        box = _Box(n, dx, dt, *_table(case))
        with torch.no_grad():
            F, X, U = _advance(box, F, X, U, W, case["pusher"], case["steps"])
        return dict(zip(FIELDS, F), x=X, u=U)
    if case["kind"] == "ensemble":
        with torch.no_grad():
            return _exact_ensemble(case, seed)
    # the objective by a forward run and torch's own reverse mode: a plane wave, one row
    L, front, x, u, ph = _adjoint_inputs(case, seed)
    n, dx, dt = _grid(case)
    cE, cB = _table(case)
    a0 = torch.tensor(case["a0"], dtype=torch.float64, device=_device(), requires_grad=True)
    phase = torch.tensor(ph, dtype=torch.float64, device=_device(), requires_grad=True)
    e2, b3 = (v.reshape(1, -1) for v in _laser_rows(n[0], dt, cE, cB, a0, phase, L, front))
    z = torch.zeros_like(e2)
    box = _Box((n[0], 1), dx, dt, cE, cB, L=[n[0] * dx[0], n[1] * dx[1]])
    X = torch.as_tensor(x, device=_device()).reshape(2, -1)
    U = torch.as_tensor(u, device=_device()).reshape(3, -1)
    _, _, U = _advance(box, [z, e2, z, z, z, b3], X, U, None, case["pusher"], case["steps"])
    J = (torch.sqrt(1 + (U * U).sum(0)) - 1).mean()
    J.backward()
    return dict(J=J.detach().cpu(), a0=a0.grad.cpu(), phase=phase.grad.cpu())
