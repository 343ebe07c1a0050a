"""Workloads of the least-action propagator whose speed is tracked, each as one pass through the public
Python entry points (Context, step_batch, autograd.propagate, lfa_maps).

A case is a dict of plain values.  ``listed`` holds the standing ones, ``draw`` more of the same ranges,
``prepare`` builds what a program holds before the call (contexts with their Hamiltonian set, states),
``run`` is the call, ``work`` its unavoidable bytes and flops, ``exact`` the outputs in plain 64-bit torch
(the converged solution of every step's linear system, by GMRES on the finite-difference operator).
"""
from __future__ import annotations

import dataclasses
import math

import numpy as np
import torch

from paper_1111_4363_gb300 import autograd
from paper_1111_4363_gb300 import binding as B
from paper_1111_4363_gb300 import workloads as wl


def listed():
    return [
        # the 1D harmonic problem as configured: 256 unknowns, 20 steps; launches and latency
        dict(name="1d_harmonic", kind="propagate", dim=1, nx=64, ny=1, nz=1, K=4, sub="8", levels=1, nu=1,
             precision=0, trial=0, steps=20, tol=1e-12),
        # one small grid of the batched family stepped by itself, multigrid as configured
        dict(name="2d_64_mixed", kind="propagate", dim=2, nx=64, ny=64, nz=1, K=4, sub="4x4", levels=4, nu=2,
             precision=1, trial=3, steps=8, tol=1e-10),
        # the 2D laser problem in its production schedule, both precisions
        dict(name="2d_256_fp64", kind="propagate", dim=2, nx=256, ny=256, nz=1, K=6, sub="4x4", levels=4, nu=3,
             precision=0, trial=3, steps=4, tol=1e-10),
        dict(name="2d_256_mixed", kind="propagate", dim=2, nx=256, ny=256, nz=1, K=6, sub="4x4", levels=4, nu=3,
             precision=1, trial=3, steps=8, tol=1e-10),
        # the 3D laser problem: full size in mixed precision (the benchmark's headline), 64^3 in FP64
        dict(name="3d_128_mixed", kind="propagate", dim=3, nx=128, ny=128, nz=128, K=4, sub="4x4x4", levels=4, nu=3,
             precision=1, trial=3, steps=3, tol=1e-10),
        dict(name="3d_64_fp64", kind="propagate", dim=3, nx=64, ny=64, nz=64, K=4, sub="4x4x4", levels=4, nu=3,
             precision=0, trial=3, steps=2, tol=1e-10),
        # many independent 2D grids stepped together in their tuned single-level schedule
        dict(name="batch_48_mixed", kind="batch", members=48, K=4, precision=1, steps=4),
        # forward and backward of a pulse-shaping gradient through torch.autograd, ragged z extent
        dict(name="adjoint_3d_mixed", kind="adjoint", dim=3, nx=48, ny=48, nz=44, K=4, sub="4x4x4", levels=3, nu=3,
             precision=1, steps=4, ncomp=8),
        # the paper's own square local problem, red-black
        dict(name="square_2d_256", kind="propagate", dim=2, nx=256, ny=256, nz=1, K=6, sub="4x4", levels=1, nu=2,
             precision=0, trial=3, steps=2, tol=1e-10, square=True),
        # a new potential and the first step under it, as in a scan over potentials
        dict(name="hamiltonian_3d_96", kind="hamiltonian", dim=3, nx=96, ny=96, nz=96, K=4, sub="4x4x4", levels=4,
             nu=3, precision=1, tol=1e-10),
        # action residual and norm of given coefficients on the full 3D grid (checking a trial function)
        dict(name="residual_3d_128", kind="residual", dim=3, nx=128, ny=128, nz=128, K=4, weight="dual"),
        # convergence maps of the plane-wave experiment in the Legendre-element basis
        dict(name="lfa_maps", kind="lfa", cases=24, nk=128, nw=128),
    ]


def _log_int(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def _mult(n, m):
    return max(m, n // m * m)


# subvolume shapes that programs choose, with the largest K each allows on the finest level
_SUBS = {1: [("4", 8), ("8", 8), ("16", 8)], 2: [("2x2", 8), ("4x2", 8), ("4x4", 8), ("8x4", 4), ("8x8", 4)],
         3: [("2x2x2", 8), ("4x4x2", 4), ("4x4x4", 4)]}


def draw(rng):
    kind = rng.choice(["propagate"] * 6 + ["batch", "adjoint", "square", "hamiltonian", "residual", "lfa"])
    if kind == "lfa":
        return dict(kind="lfa", cases=rng.randint(4, 32), nk=_log_int(rng, 32, 200), nw=_log_int(rng, 32, 200))
    if kind == "batch":
        return dict(kind="batch", members=_log_int(rng, 4, 48), K=rng.choice([3, 4]), precision=rng.choice([0, 1]),
                    steps=rng.randint(2, 4))
    if kind == "square":
        K = rng.choice([3, 4, 5, 6])
        return dict(kind="propagate", dim=2, nx=_log_int(rng, 24, 256), ny=_log_int(rng, 24, 256), nz=1, K=K,
                    sub=rng.choice(["2x2", "4x2", "4x4"]), levels=1, nu=2, precision=0, trial=rng.randint(0, 3),
                    steps=2, tol=1e-10, square=True)
    if kind == "residual":
        dim = rng.choice([1, 2, 3])
        hi = {1: 100000, 2: 1024, 3: 112}[dim]
        n = [_log_int(rng, 9, hi) if a < dim else 1 for a in range(3)]
        return dict(kind="residual", dim=dim, nx=n[0], ny=n[1], nz=n[2], K=rng.randint(1, 8 if dim < 3 else 5),
                    weight=rng.choice(["dual", "literal", "identity"]))
    dim = rng.choice([2, 3]) if kind != "propagate" else rng.choice([1, 2, 2, 2, 3, 3, 3])
    sub, kmax = rng.choice(_SUBS[dim])
    K = rng.randint(2, kmax)
    if dim == 3 and sub == "4x4x4":
        K = rng.choice([3, 4, 4])
    levels = rng.choice([1, 2, 3, 4]) if dim > 1 else 1
    m = 1 << (levels - 1)
    precision = rng.choice([0, 1])
    hi = {1: 512, 2: 256, 3: 96 if precision else 44}[dim]
    if kind == "adjoint":
        hi = {2: 128, 3: 48 if precision else 32}[dim]
    if dim == 3 and sub == "4x4x2" or K > 4 and dim == 3:
        hi = min(hi, 40)
    lo = {1: 24, 2: 24, 3: 12}[dim]
    n = [_mult(_log_int(rng, lo, hi), m) if a < dim else 1 for a in range(3)]
    c = dict(kind=kind, dim=dim, nx=n[0], ny=n[1], nz=n[2], K=K, sub=sub, levels=levels, nu=rng.choice([2, 3]),
             precision=precision)
    if kind == "adjoint":
        c.update(steps=rng.randint(2, 4), ncomp=rng.randint(1, 16))
    elif kind == "hamiltonian":
        c.update(tol=1e-10)
    else:
        c.update(trial=rng.randint(0, 3), steps=rng.randint(2, 4) if dim > 1 else rng.randint(2, 12), tol=1e-10)
    return c


# ------------------------------------------------------------------------------------ inputs
def _workload(case, seed):
    """The problem of a case: this package's own 1D, 2D and 3D problems at the case's sizes, with a seeded
    Gaussian initial state."""
    dim, K = case["dim"], case["K"]
    n = (case["nx"], case["ny"], case["nz"])
    sub = [int(s) for s in case.get("sub", "x".join(["4"] * dim)).split("x")] + [1, 1]
    base = {1: wl.harmonic_1d, 2: wl.softcore_2d, 3: wl.hydrogen_3d}[dim]()
    levels, nu = case.get("levels", 1), case.get("nu", 1)
    coarse = tuple(2 if a < dim else 1 for a in range(3)) if levels > 1 else None
    return dataclasses.replace(
        base, n=n, nt=K, sub=tuple(sub[:3]), levels=levels, nu1=1, nu2=nu - 1,
        coarse_sweeps=1, coarse_sub=coarse, coarse_nu=(1, 0) if levels > 2 and nu == 3 else None, max_cycles=200,
        tol=case.get("tol", 1e-10), trial=case.get("trial", 3), seed=seed,
        psi_kind="displaced_noisy" if dim == 1 else "gaussian", weight=case.get("weight", "dual"),
        local_form="square" if case.get("square") else "lsq")


# start time of every propagation: inside the pulse
_T0 = 10.0


def _dev(x):
    return torch.from_numpy(np.ascontiguousarray(x).ravel()).cuda()


def _context(w, precision, **kw):
    V0 = _dev(wl.potential(w))
    ctx = B.Context(B.config_from_workload(w, precision=precision, **kw))
    ctx.set_hamiltonian(V0, w.pulse)
    return ctx, V0


def _batch_members(case, seed):
    """Grids of the batched family (seeded extents, field strengths and potentials) in the schedule its
    autotuner picks for K = 4: one level, 4 x 2 subvolumes, two sweeps per cycle.  The extents belong to
    the case; the fields, potentials and states come from the seed."""
    out = []
    for i in range(case["members"]):
        n = wl.batched_2d(i).n
        m = wl.batched_2d(1000 * (seed % 100000) + i)
        out.append(dataclasses.replace(m, n=n, nt=case["K"], sub=(4, 2, 1), levels=1, nu1=1, nu2=1, max_cycles=200,
                                       trial=3))
    return out


def _lfa_grid(case, seed):
    """Element sizes and the (kappa, nu) pairs of the paper's figures, all three methods; wavenumbers and
    frequencies over [-8, 8], shifted by the seed within one grid cell."""
    pairs = [(1.0, 0.0), (1.0, 1.0), (2.0, 2.0), (4.0, 1.0), (0.5, 4.0)]
    kinds = [(m, s) for s in (3, 4, 6, 8) for m in ("one", "two", "transfer")]
    cases = []
    for i in range(case["cases"]):
        m, s = kinds[i % len(kinds)]
        ka, nu = pairs[(i // len(kinds)) % len(pairs)]
        cases.append((m, s, s, ka, nu))
    u = np.random.default_rng(seed).uniform(0.2, 0.8, 2)
    k = -8.0 + 16.0 * (np.arange(case["nk"]) + u[0]) / case["nk"]
    w = -8.0 + 16.0 * (np.arange(case["nw"]) + u[1]) / case["nw"]
    return cases, k, w


def prepare(case, seed):
    kind = case["kind"]
    if kind == "lfa":
        cases, k, w = _lfa_grid(case, seed)
        out = torch.empty((len(cases), 2, len(w), len(k)), dtype=torch.float64, device="cuda")
        return dict(kind=kind, cases=cases, k=k, w=w, out=out)
    if kind == "batch":
        ws = _batch_members(case, seed)
        ctxs = [_context(w, case["precision"])[0] for w in ws]
        return dict(kind=kind, ctxs=ctxs, psi0=[_dev(wl.initial_state(w)) for w in ws], steps=case["steps"],
                    t0=[_T0] * len(ws))
    w = _workload(case, seed)
    psi0 = _dev(wl.initial_state(w))
    if kind == "propagate":
        return dict(kind=kind, ctx=_context(w, case["precision"])[0], psi0=psi0, steps=case["steps"])
    if kind == "residual":
        c = _dev(wl.random_state((w.npoints, w.nt), seed + 1))
        return dict(kind=kind, ctx=_context(w, 0)[0], psi0=psi0, c=c, r=torch.empty_like(c))
    if kind == "hamiltonian":
        w = _scan_member(w, seed)
        return dict(kind=kind, ctx=B.Context(B.config_from_workload(w, precision=case["precision"])),
                    V0=_dev(wl.potential(w)), pulse=w.pulse, psi0=psi0)
    w = _adjoint_workload(case, w)
    ctx, V0 = _context(w, case["precision"], ckpt_every=2, cache_factors=1)
    x = _dev(wl.laser_coordinate(w))
    vol = float(np.prod(w.h[: w.dim]))
    return dict(kind=kind, ctx=ctx, V0=V0, pulse=w.pulse, amp=torch.tensor(w.pulse.amp, dtype=torch.float64),
                psi0=psi0, x=x * vol, steps=case["steps"])


def _scan_member(w, seed):
    a = float(np.random.default_rng(seed).uniform(0.5, 2.0))
    return dataclasses.replace(w, potential="softcore", softcore_a=a)


def _adjoint_workload(case, w):
    """Gaussian-enveloped components spread over the propagated time."""
    nc, T = case["ncomp"], case["steps"] * w.dt
    rng = np.random.default_rng(7)
    pulse = wl.Pulse(amp=list(rng.normal(0.0, 0.1, nc)), omega=list(rng.uniform(0.05, 2.0, nc)),
                     t_center=list(_T0 + np.linspace(0.0, T, nc)), sigma=[max(T / nc, 0.05)] * nc, axis=0)
    return dataclasses.replace(w, pulse=pulse)


# ------------------------------------------------------------------------------------ the call
def run(state):
    kind = state["kind"]
    if kind == "lfa":
        return {"maps": B.lfa_maps(state["cases"], state["k"], state["w"], state["out"])}
    if kind == "batch":
        psis = [p.clone() for p in state["psi0"]]
        B.step_batch(state["ctxs"], psis, state["steps"], state["t0"])
        return psis
    ctx = state["ctx"]
    if kind == "propagate":
        psi = state["psi0"].clone()
        ctx.step(psi, state["steps"], _T0)
        return {"psi": psi}
    if kind == "residual":
        N = ctx.residual(state["psi0"], _T0, state["c"], state["r"])
        return {"r": state["r"], "N": N}
    if kind == "hamiltonian":
        ctx.set_hamiltonian(state["V0"], state["pulse"])
        psi = state["psi0"].clone()
        ctx.step(psi, 1, _T0)
        return {"psi": psi}
    amp = state["amp"].clone().requires_grad_(True)
    psi0 = state["psi0"].clone().requires_grad_(True)
    psi = autograd.propagate(ctx, state["V0"], state["pulse"], amp, psi0, state["steps"], _T0)
    dipole = (state["x"] * (psi.real ** 2 + psi.imag ** 2)).sum()
    ga, gp = torch.autograd.grad(dipole, [amp, psi0])
    return {"psi": psi.detach(), "amp": ga, "psi0": gp}


# ------------------------------------------------------------------------------------ work
def _step_work(w, sweeps, square=False):
    """One time step of the relaxation: one factorisation of every finest subvolume and `sweeps` passes of two
    triangular solves with it, counted dense; the state in and out once."""
    n = 1.0
    nsub = 1.0
    for a in range(w.dim):
        n *= min(w.sub[a], w.n[a])
        nsub *= w.n[a] / min(w.sub[a], w.n[a])
    n *= w.nt
    return nsub * ((8.0 if square else 4.0) / 3.0 * n ** 3 + sweeps * 8.0 * n * n)


def work(case):
    kind = case["kind"]
    if kind == "lfa":
        pts, fl = float(case["nk"]) * case["nw"], 0.0
        for m, s, _, _, _ in _lfa_grid(case, 0)[0]:
            e = 1 if m == "one" else 2
            fl += 8.0 * 4.0 * (e * s * s) * (e * s)
        return dict(bytes=16.0 * case["cases"] * pts, flops=fl * pts)
    if kind == "batch":
        ws = _batch_members(case, 0)
        return dict(bytes=32.0 * sum(w.npoints for w in ws),
                    flops=case["steps"] * sum(_step_work(w, 4) for w in ws))
    w = _workload(case, 0)
    if kind == "residual":
        return dict(bytes=w.npoints * (24.0 + 32.0 * w.nt),
                    flops=w.npoints * w.nt * (16.0 * w.nt + 4.0 * (2 * w.dim + 1)))
    nu = case["nu"]
    per = _step_work(w, 2 * nu, bool(case.get("square")))
    base = w.npoints * 40.0
    if kind == "hamiltonian":
        return dict(bytes=base, flops=per)
    steps = case["steps"]
    if kind == "adjoint":   # forward, its recomputation and the adjoint relaxation
        return dict(bytes=base, flops=3.0 * steps * per)
    return dict(bytes=base, flops=steps * per)


# ------------------------------------------------------------------------------------ 64-bit reference
class _System:
    """The step's linear system M c = f of one grid in torch complex128, point-major [z, y, x, K], per unit
    overlap: (M c) = i Qb c - Ub (H c) - x Eb c, f = Ub0 (H psi) + x Eb0 psi."""

    def __init__(self, w, device):
        self.w, self.dev, K = w, device, w.nt
        leg = np.polynomial.legendre
        tau, wq = leg.leggauss(48)
        eye = np.eye(K + 1)
        P = np.stack([leg.legval(tau, eye[n]) for n in range(K + 1)])
        D = np.stack([leg.legval(tau, leg.legder(eye[n])) if n else 0 * tau for n in range(K + 1)])
        s = np.array([(-1.0) ** n for n in range(1, K + 1)])
        self.tau, self.wq = tau, wq
        self.b = P[1:] - s[:, None]
        self.Ub = 0.5 * w.dt * (self.b * wq) @ self.b.T
        self.Qb = (self.b * wq) @ D[1:].T
        self.Ub0 = 0.5 * w.dt * self.b @ wq
        self.end = 1.0 - s
        self.V0 = self._t(wl.potential(w)).reshape(self._grid())
        self.x = self._t(np.broadcast_to(wl.laser_coordinate(w), w.shape).copy()).reshape(self._grid())
        self.vol = float(np.prod(w.h[: w.dim]))
        self.dsum = sum(1.0 / w.h[a] ** 2 for a in range(w.dim))

    def _grid(self):
        return tuple(self.w.n[a] if a < self.w.dim else 1 for a in (2, 1, 0))

    def _t(self, a):
        a = np.asarray(a)
        return torch.from_numpy(np.ascontiguousarray(a, dtype=np.complex128 if a.dtype.kind == "c" else np.float64)
                                ).to(self.dev)

    def field(self, t0, j=None):
        """(Eb, Eb0) of the step from t0, of pulse component j at unit amplitude or of the whole pulse."""
        p, K = self.w.pulse, self.w.nt
        t = t0 + 0.5 * (self.tau + 1.0) * self.w.dt
        E = np.zeros_like(t)
        for k in range(p.ncomp if p is not None else 0):
            if j is not None and k != j:
                continue
            env = np.exp(-((t - p.t_center[k]) / p.sigma[k]) ** 2) if p.sigma[k] > 0 else 1.0
            E = E + (p.amp[k] if j is None else 1.0) * env * np.sin(p.omega[k] * t)
        return 0.5 * self.w.dt * (self.b * self.wq * E) @ self.b.T, 0.5 * self.w.dt * self.b @ (self.wq * E)

    def H(self, v):
        """H v for v [z, y, x, m]."""
        out = (self.dsum + self.V0)[..., None] * v
        for a in range(self.w.dim):
            ax, h = 2 - a, -0.5 / self.w.h[a] ** 2
            n = v.shape[ax]
            if n > 1:
                out.narrow(ax, 0, n - 1).add_(v.narrow(ax, 1, n - 1), alpha=h)
                out.narrow(ax, 1, n - 1).add_(v.narrow(ax, 0, n - 1), alpha=h)
        return out

    def at(self, t0, adjoint=False):
        """Operator (or its adjoint) and point-block preconditioner of the step from t0."""
        Eb, Eb0 = self.field(t0)
        Q, U, E = (self._t(m + 0j) for m in (self.Qb, self.Ub, Eb))
        S = -1j * Q.T if adjoint else 1j * Q
        UT, ET = (U.T, E.T) if adjoint else (U, E)
        x = self.x[..., None]

        def M(c):
            return c @ S.T - self.H(c) @ UT.T - (x * c) @ ET.T

        d = (self.dsum + self.V0).reshape(-1, 1, 1)
        D = torch.linalg.inv(S - d * UT - self.x.reshape(-1, 1, 1) * ET)

        def prec(c):
            return (D @ c.reshape(-1, self.w.nt, 1)).reshape(c.shape)

        return M, prec, Eb0

    def solve(self, M, prec, f, tol=2e-14, restart=48, outer=6):
        """Right-preconditioned GMRES with restarts."""
        c = torch.zeros_like(f)
        r = f.clone()
        f0 = float(torch.linalg.vector_norm(f))
        if f0 == 0.0:
            return c
        for _ in range(outer):
            beta = float(torch.linalg.vector_norm(r))
            if beta <= tol * f0:
                break
            V = torch.empty((restart + 1, f.numel()), dtype=f.dtype, device=f.device)
            V[0] = r.reshape(-1) / beta
            Hm = np.zeros((restart + 1, restart), dtype=np.complex128)
            m = 0
            while m < restart:
                u = M(prec(V[m].reshape(f.shape))).reshape(-1)
                for _twice in range(2):
                    h = V[: m + 1].conj() @ u
                    u = u - V[: m + 1].T @ h
                    Hm[: m + 1, m] += h.cpu().numpy()
                nrm = float(torch.linalg.vector_norm(u))
                Hm[m + 1, m] = nrm
                m += 1
                e = np.zeros(m + 1, dtype=np.complex128)
                e[0] = beta
                y = np.linalg.lstsq(Hm[: m + 1, :m], e, rcond=None)[0]
                if nrm == 0.0 or np.linalg.norm(Hm[: m + 1, :m] @ y - e) <= 1e-8 * beta:
                    break
                V[m] = u / nrm
            c = c + prec((V[:m].T @ torch.from_numpy(y).to(f.device)).reshape(f.shape))
            r = f - M(c)
        return c

    def rhs(self, psi, Eb0):
        hp = self.H(psi[..., None])
        return hp * self._t(self.Ub0) + (self.x * psi)[..., None] * self._t(Eb0)

    def step(self, psi, t0):
        M, prec, Eb0 = self.at(t0)
        c = self.solve(M, prec, self.rhs(psi, Eb0))
        return psi + c @ self._t(self.end + 0j), c

    def state(self, w):
        return self._t(wl.initial_state(w)).reshape(self._grid())


def _exact_propagate(w, steps, device):
    s = _System(w, device)
    psi = s.state(w)
    for k in range(steps):
        psi, _ = s.step(psi, _T0 + k * w.dt)
    return psi.reshape(-1)


def exact(case, seed):
    kind = case["kind"]
    device = "cuda" if torch.cuda.is_available() else "cpu"
    if kind == "lfa":
        return None
    if kind == "batch":
        return [_exact_propagate(w, case["steps"], device) for w in _batch_members(case, seed)]
    w = _workload(case, seed)
    if kind == "propagate":
        return {"psi": _exact_propagate(w, case["steps"], device)}
    if kind == "hamiltonian":
        return {"psi": _exact_propagate(_scan_member(w, seed), 1, device)}
    if kind == "residual":
        s = _System(w, device)
        c = s._t(wl.random_state((w.npoints, w.nt), seed + 1)).reshape(s._grid() + (w.nt,))
        M, _, Eb0 = s.at(_T0)
        r = s.rhs(s.state(w), Eb0) - M(c)
        W = {"dual": np.linalg.inv(s.Ub) * s.vol, "literal": s.Ub * s.vol ** 3,
             "identity": np.eye(w.nt) * s.vol ** 2}[w.weight]
        N = float((r.conj() * (r @ s._t(W.T + 0j))).sum().real)
        return {"r": (r * s.vol).reshape(-1), "N": N}
    # adjoint: mu = M^-dagger B^T lambda per step, dJ/da_j = 2 Re mu^dagger (dF_j psi - dM_j c), lambda += F^T mu
    w = _adjoint_workload(case, w)
    s = _System(w, device)
    psis, cs = [s.state(w)], []
    for k in range(case["steps"]):
        p, c = s.step(psis[-1], _T0 + k * w.dt)
        psis.append(p)
        cs.append(c)
    lam = s.vol * s.x * psis[-1]
    grad = np.zeros(w.pulse.ncomp)
    end = s._t(s.end + 0j)
    for k in reversed(range(case["steps"])):
        t = _T0 + k * w.dt
        M, prec, Eb0 = s.at(t, adjoint=True)
        mu = s.solve(M, prec, lam[..., None] * end)
        for j in range(w.pulse.ncomp):
            Ej, Ej0 = s.field(t, j)
            v = psis[k][..., None] * s._t(Ej0 + 0j) + cs[k] @ s._t(Ej.T + 0j)
            grad[j] += 2.0 * float((s.x[..., None] * (mu.conj() * v)).sum().real)
        lam = lam + s.H((mu @ s._t(s.Ub0 + 0j))[..., None])[..., 0] + s.x * (mu @ s._t(Eb0 + 0j))
    return {"psi": psis[-1].reshape(-1), "amp": torch.from_numpy(grad), "psi0": 2.0 * lam.reshape(-1)}
