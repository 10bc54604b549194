"""Performance cases of the Stokes-IB solver: the calls that its users make, at the sizes they make them.

A case is a dict of plain values:
  call       what one pass does: "solve" (one linear solve of a solver that is set up), "differentiate"
             (set-up, solve, adjoint solve and gradients through autograd), "march" (time steps: set-up,
             solve, move the markers), "vcycle" (one V-cycle as a preconditioner) or "coupling"
             (interpolation, spreading and the operator, FP64)
  N          the grid is N x N (the library takes powers of two; the odd and ragged sizes are the marker and
             spring counts), periodic unless the smoother is "cavity"
  shape      "ellipse", "disk", "disk_and_ellipse" (half-cell marker spacing, springs of stiffness `kappa`),
             or the paper's "annulus" and "circle" (stiffness `gamma` in units of its explicit limit)
  fluid      "stokes" (rho = 0, mu = 1, dt = 1e-2), "re" (rho = 1, mu = 1e-2, dt = 1e-3) or "paper"
             (rho = 0, mu = 1, dt = 0.32 h)
  smoother   a key of SMOOTHERS
  fp32       the V-cycle runs in FP32 (else FP64)
  kappa_hi   > 0: one stiffness per spring, LogUniform(kappa, kappa_hi)
  steps      time steps of a "march"

Solves stop at the paper's relative tolerance 1e-12, where the answer no longer depends on the path of
the iteration.  Inputs (forcing, loss gradient, position of the structure within a cell, stiffnesses)
come from the seed.
"""
import math

import numpy as np
import torch

from paper_1612_02208_gb300 import autograd, inputs, sib

DEVICE = "cuda"
RTOL = 1e-12
SMOOTHERS = {
    "vanka": {},
    "sc_wrapped": dict(smoother=sib.SMOOTHER_SC, smooth_krylov=1),
    "ras4": dict(smoother=sib.SMOOTHER_RAS, box=4, box_overlap=1),
    "ras8": dict(smoother=sib.SMOOTHER_RAS, box=8, box_overlap=2),
    "ras16": dict(smoother=sib.SMOOTHER_RAS, box=16, box_overlap=4),
    "cavity": dict(domain=sib.DOMAIN_CAVITY),
}


def _case(call, N, shape, fluid, smoother, fp32=True, kappa=0.0, kappa_hi=0.0, gamma=0.0, steps=0):
    return dict(call=call, N=N, shape=shape, fluid=fluid, smoother=smoother, fp32=fp32, kappa=kappa,
                kappa_hi=kappa_hi, gamma=gamma, steps=steps)


def listed():
    cases = {
        # the smallest problem: a script's first solve, a unit test, one of many small systems
        "solve_ellipse_32": _case("solve", 32, "ellipse", "stokes", "vanka", kappa=1e2),
        # the ordinary Stokes solve, default smoother, a thick body
        "solve_disk_128": _case("solve", 128, "disk", "stokes", "vanka", kappa=1e2),
        # a caller who wants the preconditioner in FP64 too, at a Reynolds number
        "solve_ellipse_512_fp64": _case("solve", 512, "ellipse", "re", "vanka", fp32=False, kappa=1e2),
        # the paper's thick annulus with the box smoother
        "solve_annulus_128_ras4": _case("solve", 128, "annulus", "paper", "ras4", gamma=50.0),
        # the paper's stiff thin membrane, which needs its largest boxes
        "solve_circle_128_ras16": _case("solve", 128, "circle", "paper", "ras16", gamma=50.0),
        # the paper's lid-driven cavity
        "solve_cavity_128": _case("solve", 128, "annulus", "paper", "cavity", gamma=5.0),
        # identification of a stiffness field: every pass is a new set-up, two solves and the gradients
        "differentiate_ellipse_256": _case("differentiate", 256, "ellipse", "stokes", "vanka", kappa=1e1, kappa_hi=1e3),
        # the largest differentiated solve: 3e5 markers, stiff, the paper's smoothing
        "differentiate_disk_and_ellipse_1024": _case("differentiate", 1024, "disk_and_ellipse", "re", "sc_wrapped",
                                                     kappa=1e4),
        # a simulation: the structure moves, so every step sets up again
        "march_disk_128": _case("march", 128, "disk", "stokes", "vanka", kappa=1e2, steps=3),
        # one step of a simulation with the paper's 8 x 8 boxes
        "march_annulus_128_ras8": _case("march", 128, "annulus", "paper", "ras8", gamma=50.0, steps=1),
        # the preconditioner at a size that only HBM holds, for a caller's own Krylov loop
        "vcycle_ellipse_4096": _case("vcycle", 4096, "ellipse", "re", "vanka", kappa=1e4),
        # the coupling operators for a caller's own time stepper
        "coupling_disk_and_ellipse_1024": _case("coupling", 1024, "disk_and_ellipse", "re", "vanka", kappa=1e4),
    }
    return [dict(c, name=name) for name, c in cases.items()]


def _log(rng, lo, hi):
    return math.exp(rng.uniform(math.log(lo), math.log(hi)))


def draw(rng):
    call = rng.choice(["solve", "solve", "solve", "solve", "differentiate", "march", "vcycle", "coupling"])
    ring = rng.choice(["ellipse", "disk"])
    if call == "solve":
        which = rng.choice(["vanka", "vanka", "sc_wrapped", "ras4", "ras8", "ras16", "cavity"])
        N = rng.choice([32, 64, 128, 256, 512])
        if which == "vanka":
            fluid = rng.choice(["stokes", "re"]) if ring == "ellipse" else "stokes"
            return _case(call, N, ring, fluid, which, fp32=rng.random() < 0.75, kappa=_log(rng, 1.0, 1e2))
        if which == "sc_wrapped":
            return _case(call, N, ring, "stokes", which, fp32=rng.random() < 0.75, kappa=_log(rng, 1.0, 1e3))
        N = rng.choice([64, 128])
        if which == "cavity":
            return _case(call, N, "annulus", "paper", which, gamma=_log(rng, 1.0, 10.0))
        if which == "ras16":
            return _case(call, N, rng.choice(["annulus", "circle"]), "paper", which, gamma=_log(rng, 5.0, 50.0))
        if which == "ras8":
            return _case(call, N, "annulus", "paper", which, gamma=_log(rng, 5.0, 500.0))
        return _case(call, N, "annulus", "paper", which, gamma=_log(rng, 5.0, 50.0))
    if call == "differentiate":
        if rng.random() < 0.5:
            lo = _log(rng, 1.0, 1e1)
            return _case(call, rng.choice([32, 64, 128, 256]), "ellipse", "stokes", "vanka", kappa=lo,
                         kappa_hi=lo * _log(rng, 1e1, 1e2))
        return _case(call, rng.choice([64, 128, 256, 512]), "disk_and_ellipse", "re", "sc_wrapped",
                     kappa=_log(rng, 1e2, 1e4))
    if call == "march":
        if rng.random() < 0.25:
            return _case(call, 64, "annulus", "paper", "ras8", gamma=_log(rng, 5.0, 50.0), steps=1)
        return _case(call, rng.choice([32, 64, 128, 256]), ring, "stokes", "vanka", kappa=_log(rng, 1.0, 1e2),
                     steps=rng.randint(1, 4))
    if call == "vcycle":
        which = rng.choice(["vanka", "vanka", "sc_wrapped", "ras4"])
        return _case(call, rng.choice([128, 256, 512, 1024, 2048]), "ellipse", "re", which,
                     fp32=rng.random() < 0.75, kappa=_log(rng, 1.0, 1e4))
    return _case(call, rng.choice([64, 128, 256, 512, 1024]), rng.choice(["ellipse", "disk", "disk_and_ellipse"]), "re",
                 "vanka", kappa=_log(rng, 1.0, 1e4))


def _fluid(case):
    return {"stokes": (0.0, 1.0, 1e-2), "re": (1.0, 1e-2, 1e-3), "paper": (0.0, 1.0, 0.32 / case["N"])}[case["fluid"]]


def _structure(case):
    N, kappa = case["N"], case["kappa"]
    if case["shape"] == "ellipse":
        return inputs.thin_interface(N, kappa=kappa)
    if case["shape"] == "disk":
        return inputs.elastic_disk(N, kappa=kappa)
    if case["shape"] == "disk_and_ellipse":
        return inputs.merge(inputs.elastic_disk(N, center=(0.3, 0.5), R=0.15, kappa=kappa),
                            inputs.thin_interface(N, center=(0.7, 0.5), axes=(0.15, 0.10), r0=0.125, kappa=kappa))
    return (inputs.thick_annulus if case["shape"] == "annulus" else inputs.thin_circle)(N, case["gamma"])


def _inputs(case, seed):
    """Structure and fields on the GPU, from the seed alone."""
    N, s = case["N"], _structure(case)
    rng = np.random.default_rng(seed)
    gen = torch.Generator(device=DEVICE).manual_seed(seed)
    X = torch.as_tensor(s.X + rng.uniform(-0.5, 0.5, 2) / N, device=DEVICE)
    kappa = torch.as_tensor(s.kappa, device=DEVICE)
    if case["kappa_hi"] > 0:
        kappa = torch.as_tensor(inputs.loguniform_kappa(s.E, case["kappa"], case["kappa_hi"], seed), device=DEVICE)

    def field(dtype=torch.float64, pressure=False):
        x = torch.randn(3 * N * N, generator=gen, device=DEVICE, dtype=dtype)
        if not pressure:
            x[2 * N * N:] = 0
        return x

    return X, torch.as_tensor(s.edges, device=DEVICE), kappa, field


def prepare(case, seed):
    X, edges, kappa, field = _inputs(case, seed)
    solver = sib.Solver(case["N"])
    solver.set_fluid(*_fluid(case))
    opts = dict(SMOOTHERS[case["smoother"]], omega=-1.0, rtol=RTOL, vcycle_fp32=int(case["fp32"]))
    if case["call"] in ("vcycle", "coupling"):
        opts.update(restart=1, max_it=1)   # no Krylov space is wanted
    solver.set_options(**opts)
    state = dict(call=case["call"], solver=solver, X=X, edges=edges, kappa=kappa, steps=case["steps"])
    if case["call"] in ("solve", "vcycle", "coupling"):
        solver.set_structure(X, edges, kappa)
        solver.setup()
    if case["call"] == "vcycle":
        state["b"] = field(torch.float32 if case["fp32"] else torch.float64, pressure=True)
    else:
        state["g"] = field()
    if case["call"] == "differentiate":
        state["dw"] = field()
        state["leaves"] = [t.clone().requires_grad_(True) for t in (state["g"], kappa, X)]
    if case["call"] == "coupling":
        state["F"] = field()[: 2 * len(X)].reshape(-1, 2).contiguous()
        state["x"] = field(pressure=True)
    return state


def run(state):
    solver, call = state["solver"], state["call"]
    if call == "solve":
        return solver.solve(state["g"])
    if call == "differentiate":
        g, kappa, X = state["leaves"]
        w = autograd.stokes_ib_solve(solver, g, kappa, X, state["edges"])
        return (w.detach(), *torch.autograd.grad(w, (g, kappa, X), state["dw"]))
    if call == "march":
        ws, Xs = sib.time_loop(solver, state["g"], state["X"], state["edges"], state["kappa"], state["steps"])
        return ws + Xs[1:]
    if call == "vcycle":
        return solver.vcycle(state["b"])
    u = state["g"][: 2 * solver.N ** 2]
    return solver.interp(u), solver.spread(state["F"]), solver.apply_operator(solver.num_levels - 1, state["x"])


def work(case):
    """Inputs once and outputs once; the operations of one residual and one Vanka correction per unknown
    and level for a V-cycle's smoothing (2 + 2 sweeps), once per pass at least."""
    N, s = case["N"], _structure(case)
    n3 = 3 * N * N
    structure = 16 * s.M + 16 * s.E
    if case["call"] == "vcycle":
        w = 4 if case["fp32"] else 8
        return dict(bytes=2 * n3 * w + structure, flops=4 * 4 / 3 * 30 * n3)
    if case["call"] == "coupling":
        return dict(bytes=8 * (2 * N * N + 2 * s.M) * 2 + 16 * n3 + structure, flops=4 * 64 * s.M * 2 + 12 * n3)
    passes = dict(solve=1, differentiate=2, march=case["steps"])[case["call"]]
    return dict(bytes=passes * (16 * n3 + structure), flops=passes * 4 * 4 / 3 * 30 * n3)


# ---- the answers in 64 bits: FFT Stokes solves, and conjugate gradients for the springs' tensions ----

def _phi(r):
    a = r.abs()
    near, far = a.clamp(max=1.0), a.clamp(1.0, 2.0)
    inner = (3 - 2 * near + torch.sqrt(1 + 4 * near - 4 * near * near)) / 8
    outer = (5 - 2 * far - torch.sqrt((-7 + 12 * far - 4 * far * far).clamp(min=1e-300))) / 8
    return torch.where(a < 1, inner, torch.where(a < 2, outer, torch.zeros_like(a)))


class _Problem:
    """The periodic Stokes-IB system at one configuration of the structure, in plain torch."""

    def __init__(self, N, fluid, X, edges, kappa):
        self.N, self.h, (self.rho, self.mu, self.dt) = N, 1.0 / N, fluid
        self.X, self.kappa = X, kappa
        self.a, self.b = edges[:, 0].long(), edges[:, 1].long()
        theta = 2 * math.pi * torch.arange(N, device=X.device, dtype=torch.float64) / N
        d = (1 - torch.exp(-1j * theta)) / self.h
        self.gx, self.gy = d[None, :], d[:, None]
        self.lap = self.gx.abs() ** 2 + self.gy.abs() ** 2
        self.idx, self.wgt = zip(*(self.stencil(X, c) for c in (0, 1)))

    def stencil(self, X, c):
        off = (0.0, 0.5) if c == 0 else (0.5, 0.0)
        k = torch.arange(4, device=X.device)
        at, w = [], []
        for q in (0, 1):
            s = X[:, q] / self.h - off[q]
            first = torch.floor(s.detach()).long() - 1
            at.append(first[:, None] + k)
            w.append(_phi(at[-1] - s[:, None]))
        idx = (at[1] % self.N)[:, :, None] * self.N + (at[0] % self.N)[:, None, :]
        return idx.reshape(len(X), 16), (w[1][:, :, None] * w[0][:, None, :]).reshape(len(X), 16)

    def interp(self, u):
        u = u.reshape(2, -1)
        return torch.stack([(u[c][self.idx[c]] * self.wgt[c]).sum(1) for c in (0, 1)], 1)

    def spread(self, F):
        f = torch.zeros(2, self.N ** 2, device=F.device, dtype=F.dtype)
        for c in (0, 1):
            f[c].index_add_(0, self.idx[c].reshape(-1), (self.wgt[c] * F[:, c:c + 1]).reshape(-1) / self.h ** 2)
        return f

    def stretch(self, Y):
        return Y[self.a] - Y[self.b]

    def force(self, t):
        """Marker forces of spring tensions t: -stretch^T t."""
        F = torch.zeros_like(self.X)
        return F.index_add_(0, self.b, t).index_add_(0, self.a, -t)

    def stokes(self, f, pressure=False):
        fx, fy = torch.fft.fft2(f.reshape(2, self.N, self.N))
        lap = self.lap.clone()
        lap[0, 0] = 1
        p = -(-self.gx.conj() * fx - self.gy.conj() * fy) / lap
        p[0, 0] = 0
        A = self.rho / self.dt + self.mu * lap
        u = torch.stack([(fx - self.gx * p) / A, (fy - self.gy * p) / A])
        u[:, 0, 0] = u[:, 0, 0] * A[0, 0] * self.dt / self.rho if self.rho > 0 else 0
        u = torch.fft.ifft2(u).real.reshape(2, -1)
        return (u, torch.fft.ifft2(p).real.reshape(-1)) if pressure else u

    def solve(self, f, positions):
        """[u | v | p] for the force f on the faces and spring positions `positions` + dt J u."""
        f = f[: 2 * self.N ** 2].reshape(2, -1)
        op = lambda t: t / self.kappa[:, None] - self.dt * self.stretch(  # noqa: E731
            self.interp(self.stokes(self.spread(self.force(t)))))
        t = torch.zeros(len(self.kappa), 2, device=f.device, dtype=torch.float64)
        r = self.stretch(positions + self.dt * self.interp(self.stokes(f)))
        stop = 1e-14 * float((r * r * self.kappa[:, None]).sum().sqrt())
        d, rz = torch.zeros_like(r), None
        for _ in range(4000):
            z = r * self.kappa[:, None]
            new = float((r * z).sum())
            if math.sqrt(new) <= stop:
                break
            d = z if rz is None else z + (new / rz) * d
            rz = new
            q = op(d)
            step = rz / float((d * q).sum())
            t, r = t + step * d, r - step * q
        u, p = self.stokes(f + self.spread(self.force(t)), pressure=True)
        return torch.cat([u.reshape(-1), p])

    def apply(self, x):
        u, v, p = x.reshape(3, self.N, self.N)
        h = self.h
        Y = self.interp(x[: 2 * self.N ** 2])
        f = self.dt * self.spread(self.force(self.kappa[:, None] * self.stretch(Y))).reshape(2, self.N, self.N)

        def momentum(q):
            lap = q.roll(1, 0) + q.roll(-1, 0) + q.roll(1, 1) + q.roll(-1, 1) - 4 * q
            return self.rho / self.dt * q - self.mu * lap / h ** 2

        return torch.stack([momentum(u) - f[0] + (p - p.roll(1, 1)) / h, momentum(v) - f[1] + (p - p.roll(1, 0)) / h,
                            -(u.roll(-1, 1) - u + v.roll(-1, 0) - v) / h]).reshape(-1)

    def gradients(self, w, lam):
        """d/d(kappa, X) of lam . (right-hand side - L w), the discrete adjoint."""
        n2 = 2 * self.N ** 2
        with torch.enable_grad():
            kappa, X = (t.detach().clone().requires_grad_(True) for t in (self.kappa, self.X))
            U, Lam = [], []
            for c in (0, 1):
                idx, wgt = self.stencil(X, c)
                U.append((w[:n2].reshape(2, -1)[c][idx] * wgt).sum(1))
                Lam.append((lam[:n2].reshape(2, -1)[c][idx] * wgt).sum(1) / self.h ** 2)
            Y, Lam = X + self.dt * torch.stack(U, 1), torch.stack(Lam, 1)
            q = -(kappa[:, None] * self.stretch(Y) * self.stretch(Lam)).sum()
            return torch.autograd.grad(q, (kappa, X))


def exact(case, seed):
    if case["call"] == "vcycle" or case["smoother"] == "cavity":
        # a V-cycle's result is defined by its algorithm alone; a walled Stokes solve at 128^2 needs a sparse
        # direct solver or minutes of dense elimination
        return None
    state_X, edges, kappa, field = _inputs(case, seed)
    N, fluid = case["N"], _fluid(case)
    g = field()
    P = _Problem(N, fluid, state_X, edges, kappa)
    if case["call"] == "solve":
        return P.solve(g, state_X)
    if case["call"] == "differentiate":
        dw = field()
        w, lam = P.solve(g, state_X), P.solve(dw, torch.zeros_like(state_X))
        return (w, lam, *P.gradients(w, lam))
    if case["call"] == "march":
        ws, Xs, X = [], [], state_X
        for _ in range(case["steps"]):
            P = _Problem(N, fluid, X, edges, kappa)
            ws.append(P.solve(g, X))
            X = X + P.dt * P.interp(ws[-1][: 2 * N * N])
            Xs.append(X)
        return ws + Xs
    F = field()[: 2 * len(state_X)].reshape(-1, 2)
    x = field(pressure=True)
    return P.interp(g[: 2 * N * N]), P.spread(F).reshape(-1), P.apply(x)
