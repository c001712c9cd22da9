"""Performance cases of the solver: what programs ask of it, through its public entry points.

A program that uses this library advances a flow around immersed bodies: it
sets the markers, takes a time step, moves the bodies and takes the next.
Around that it solves single Schur systems, differentiates a step, couples the
bodies both ways, or applies single operators to compose a scheme of its own.
The listed cases are these calls at the sizes of the repository's workloads
(``workloads.config``: 32^3, 128^3, 256^3 and 384^3), of its tests (48 x 40 x 32
and other boxes that are no cubes) and of its benchmark (eight spheres with
60000 markers); ``draw`` gives further ones of the same kinds.

Tolerances: steps and solves run to 1e-11, where their results agree with the
exact ones to the 1e-10 that the repository claims; the 32^3 workload to its own
1e-10, the metric's FP64 solve to the metric's 1e-8.  Everything else is at the
library's defaults.
The FP32 V-cycle has no case by itself: as an operator it is only used inside
the mixed solves, which are measured here as a whole.

``exact`` restates every path in plain torch in 64 bits: dense cosine
transforms for the inverse Laplacian, conjugate gradients for the linear
systems, explicit index and weight lists for the marker operators.
"""
from __future__ import annotations

import math

import numpy as np
import torch

from paper_2501_15314_gb300 import workloads as wl
from paper_2501_15314_gb300._lib import (IBM_ARNOLDI_FP32, IBM_ARNOLDI_FP64, IBM_CMODE_EXACT,
                                         IBM_CMODE_SCALAR, IBM_FSI_CRIT_EULERIAN)
from paper_2501_15314_gb300.api import IBM_PREC_FP32, IBM_PREC_FP64, IBMSolver, RigidSpheres
from paper_2501_15314_gb300.autograd import body_loads, ib_step

F64 = torch.float64


def _case(kind, n, bodies=1, r_lo=0.15, r_hi=0.15, spacing=1.0, Re=100.0, dt=2e-3,
          fp64=False, rtol=1e-11, history=False, exact_c=False, **more):
    """A case: radii in units of the shortest side of the box, marker spacing
    h / ``spacing``, ``history`` false for a step from rest."""
    nx, ny, nz = (n, n, n) if isinstance(n, int) else n
    return dict(kind=kind, nx=nx, ny=ny, nz=nz, bodies=bodies, r_lo=r_lo, r_hi=r_hi,
                spacing=spacing, Re=Re, dt=dt, fp64=fp64, rtol=rtol, history=history,
                exact_c=exact_c, **more)


def listed():
    return [
        # A program that composes its own scheme: every field and marker
        # operator once, on the small box of the tests that is no cube.
        dict(_case("operators", (48, 40, 32), bodies=3, r_lo=0.12, r_hi=0.16),
             name="operators_48x40x32"),
        # The smallest time step: plain FP64 method, one sphere.
        dict(_case("step", 32, r_lo=0.2, r_hi=0.2, dt=0.01, fp64=True, rtol=1e-10),
             name="step_32_fp64"),
        # A box that is no cube, three bodies, in the middle of a run.
        dict(_case("step", (112, 80, 48), bodies=3, r_lo=0.12, r_hi=0.2, Re=150.0, dt=4e-3,
                   history=True), name="step_112x80x48"),
        # The ordinary time step: one sphere at 128^3, mixed precision, in the
        # middle of a run (moving markers, BDF2 history, convection).
        dict(_case("step", 128, history=True), name="step_128"),
        # The benchmark's step: eight spheres and about 60000 markers, from rest.
        dict(_case("step", 256, bodies=8, r_lo=0.05, r_hi=0.1, spacing=1.38, Re=200.0, dt=1e-3),
             name="step_256"),
        # The largest step: the sedimentation workload's grid and sphere.
        dict(_case("step", 384, r_lo=0.08, r_hi=0.08, Re=50.0, dt=5e-4, history=True),
             name="step_384"),
        # The metric's FP64 column: one Schur solve, V-cycle and Arnoldi in FP64.
        dict(_case("solve", 256, bodies=8, r_lo=0.05, r_hi=0.1, spacing=1.38, Re=200.0, dt=1e-3,
                   fp64=True, rtol=1e-8), name="solve_256_fp64"),
        # The exact Schur complement L + B^T C^{-1} B of the spectral theorem.
        dict(_case("solve", 64, exact_c=True), name="solve_64_exact_c"),
        # A differentiated step: drag and torque of the oscillating sphere,
        # with their gradients to the marker velocities and positions, FP64.
        dict(_case("adjoint", 128, fp64=True, rtol=1e-12), name="adjoint_128_fp64"),
        # The preconditioner as an operator of a caller's own Krylov method.
        dict(_case("precond", 192, fp64=True), name="precond_192_fp64"),
        # New body positions and the coupling operators: what a direct-forcing
        # scheme of the caller's own asks of the markers in every step.
        dict(_case("coupling", 256, bodies=8, r_lo=0.05, r_hi=0.1, spacing=1.38),
             name="coupling_256"),
        # A two-way coupled step of a falling sphere, four corrections (what a
        # step takes once the fall is under way).
        dict(_case("fsi", 128, r_lo=0.1, r_hi=0.1, Re=50.0, dt=5e-4, inner=4), name="fsi_128"),
    ]


def _box(rng, most):
    """Cell counts per axis, q 2^k with small q, at most ``most`` cells and
    spread over the logarithm of their number."""
    while True:
        target = math.exp(rng.uniform(math.log(16 ** 3), math.log(most)))
        k = rng.randint(1, 6)
        side = target ** (1.0 / 3.0) / 2 ** k
        q = [max(2, round(side * math.exp(rng.uniform(-0.4, 0.4)))) for _ in range(3)]
        n = [v * 2 ** k for v in q]
        if (min(n) >= 16 and max(q) <= 9 and max(n) <= 3 * min(n)
                and q[0] * q[1] * q[2] <= 512 and n[0] * n[1] * n[2] <= most):
            return tuple(n)


def draw(rng):
    kind = rng.choice(["step", "step", "step", "solve", "solve", "operators", "coupling",
                       "adjoint", "precond", "fsi"])
    most = {"step": 256 ** 3, "solve": 224 ** 3, "operators": 256 ** 3, "coupling": 256 ** 3,
            "adjoint": 112 ** 3, "precond": 224 ** 3, "fsi": 160 ** 3}[kind]
    n = _box(rng, most)
    bodies = rng.choice([1, 1, 2, 3, 5])
    r = rng.uniform(0.1, 0.16) if bodies > 1 else rng.uniform(0.12, 0.22)
    r = max(r, 2.0 / min(n)) if bodies == 1 else max(r, 1.5 / min(n))
    if bodies > 1 and min(n) < 40:
        bodies = 1
    h = 1.0 / max(n)
    # time steps at CFL numbers of 0.1 to 0.4
    dt = rng.uniform(0.1, 0.4) * h
    c = _case(kind, n, bodies=bodies, r_lo=r, r_hi=1.15 * r, spacing=rng.uniform(1.0, 1.4),
              Re=math.exp(rng.uniform(math.log(50.0), math.log(300.0))), dt=dt,
              fp64=rng.random() < 0.25, history=rng.random() < 0.7)
    if kind == "solve" and n[0] * n[1] * n[2] <= 64 ** 3 and rng.random() < 0.5:
        c.update(exact_c=True, spacing=1.0)
    if kind == "adjoint":
        c.update(fp64=True, rtol=1e-12, history=False)
    if kind == "precond":
        c.update(fp64=True)
    if kind == "fsi":
        c.update(inner=rng.randint(2, 4), spacing=1.0, bodies=1)
    return c


# ---- inputs ---------------------------------------------------------------

def _dev(a):
    return torch.from_numpy(np.ascontiguousarray(a)).cuda()


class _Geometry:
    """Grid, spheres, markers and their rigid velocities, from the seed alone."""

    def __init__(self, case, seed):
        self.n = (case["nx"], case["ny"], case["nz"])
        self.h = 1.0 / max(self.n)
        self.side = np.array(self.n) * self.h
        rng = np.random.default_rng([7, seed])
        self.rng = rng
        short = self.side.min()
        gap = 3.0 * self.h
        # the radii, and with them the marker counts, belong to the case; the
        # seed places the spheres
        radii = np.linspace(case["r_lo"], case["r_hi"], case["bodies"]) * short
        while True:
            centers = []
            for r in radii:
                for _ in range(2000):
                    c = rng.uniform(r + gap, self.side - r - gap)
                    if all(np.linalg.norm(c - d) >= r + s + gap for d, s in zip(centers, radii)):
                        centers.append(c)
                        break
                else:
                    break
            if len(centers) == len(radii):
                break
        self.radii, self.centers = radii, np.array(centers)
        X, ids = [], []
        for b, (c, r) in enumerate(zip(self.centers, radii)):
            k = wl.markers_for_spacing(r, self.h / case["spacing"])
            X.append(wl.fibonacci_sphere(k, r, c))
            ids.append(np.full(k, b, dtype=np.int32))
        self.X = np.concatenate(X, axis=1)
        self.body_id = np.concatenate(ids)
        self.U = wl.rigid_velocities(self.X, self.body_id, self.centers, rng)

    def coords(self, d):
        """Coordinates (z, y, x) of the d-faces (d = 3: of the cells)."""
        out = []
        for e in range(3):
            k = torch.arange(self.n[e] + (1 if e == d else 0), device="cuda", dtype=F64)
            out.append((k + (0.0 if e == d else 0.5)) * self.h)
        return out[2][:, None, None], out[1][None, :, None], out[0][None, None, :]

    def pack(self, comps):
        """One packed face vector, 0 on the walls."""
        for d, c in enumerate(comps):
            c.select(2 - d, 0).zero_()
            c.select(2 - d, -1).zero_()
        return torch.cat([c.reshape(-1) for c in comps])

    def body_force(self):
        """The smooth forcing of the workloads: eight sine modes of amplitude 1."""
        comps = []
        for d in range(3):
            z, y, x = self.coords(d)
            f = 0.0
            for _ in range(8):
                k = self.rng.integers(1, 5, 3)
                ph = self.rng.uniform(0.0, 2.0 * np.pi)
                f = f + torch.sin(2.0 * np.pi * (k[0] * x + k[1] * y + k[2] * z) + ph)
            comps.append(f)
        return self.pack(comps)

    def flow(self, modes=4):
        """A smooth velocity field of size about 1, divergence-free and
        tangential at the walls."""
        comps = [0.0, 0.0, 0.0]
        for _ in range(modes):
            k = self.rng.integers(1, 5, 3) * np.pi / self.side
            a = np.cross(k, self.rng.uniform(-1.0, 1.0, 3))
            a /= np.linalg.norm(a) * math.sqrt(modes)
            for d in range(3):
                z, y, x = self.coords(d)
                fn = [torch.sin if e == d else torch.cos for e in range(3)]
                comps[d] = comps[d] + a[d] * (fn[0](k[0] * x) * fn[1](k[1] * y) * fn[2](k[2] * z))
        return self.pack(comps)

    def pressure(self):
        z, y, x = self.coords(3)
        p = 0.0
        for _ in range(4):
            k = self.rng.integers(1, 4, 3) * np.pi / self.side
            p = p + self.rng.uniform(-1, 1) * (torch.cos(k[0] * x) * torch.cos(k[1] * y)
                                               * torch.cos(k[2] * z))
        return p.reshape(-1).contiguous()


def _options(case):
    o = dict(rtol=case["rtol"], helm_rtol=case["rtol"],
             precond_prec=IBM_PREC_FP64 if case["fp64"] else IBM_PREC_FP32,
             arnoldi=IBM_ARNOLDI_FP64 if case["fp64"] else IBM_ARNOLDI_FP32,
             c_mode=IBM_CMODE_EXACT if case["exact_c"] else IBM_CMODE_SCALAR)
    if case["exact_c"]:
        o["c_maxit"] = 2000
    return o


def _inputs(case, seed):
    """The tensors of a call (and host values), without the solver."""
    g = _Geometry(case, seed)
    kind = case["kind"]
    m = g.n[0] * g.n[1] * g.n[2]
    nf = sum((g.n[d] + 1) * (m // g.n[d]) for d in range(3))
    nmk = g.X.size
    s = dict(geometry=g, X=_dev(g.X), U=_dev(g.U.ravel()))
    gen = torch.Generator(device="cuda")
    gen.manual_seed(int(seed))
    normal = lambda k: torch.randn(k, generator=gen, device="cuda", dtype=F64)  # noqa: E731
    if kind in ("step", "adjoint", "fsi"):
        if case["history"] or kind == "fsi":
            s["u_n"] = g.flow()
            s["u_nm1"] = 0.98 * s["u_n"] + 0.02 * g.flow(1)
            s["p_n"] = g.pressure()
            s["F_n"] = 5.0 * s["U"]
        else:
            s["u_n"] = torch.zeros(nf, device="cuda", dtype=F64)
            s["u_nm1"] = s["u_n"]
            s["p_n"] = torch.zeros(m, device="cuda", dtype=F64)
            s["F_n"] = torch.zeros(nmk, device="cuda", dtype=F64)
        s["f_body"] = g.body_force()
    if kind == "fsi":
        # the falling sphere: velocity and rotation of the moment, a little
        # heavier than the fluid
        s["velocity"] = g.rng.uniform(-0.2, 0.2, (1, 3)) + np.array([[0.0, 0.0, -0.5]])
        s["omega"] = g.rng.uniform(-0.5, 0.5, (1, 3))
        s["L0"] = _dev(g.X - g.centers[0][:, None])
        s["body_id"] = _dev(g.body_id)
    if kind == "adjoint":
        s["body_id"] = _dev(g.body_id)
        s["centers"] = torch.from_numpy(g.centers)
        w = torch.zeros((g.centers.shape[0], 6), dtype=F64)
        w[:, 2] = -1.0   # drag and torque about z: the bodies feel minus the loads
        w[:, 5] = -1.0
        s["w"] = w
    if kind == "solve":
        # right-hand side of a step's form: divergence of a smooth momentum
        # imbalance and the markers' slip
        s["momentum"] = 1.5 / case["dt"] * (g.flow() + case["dt"] * g.body_force())
        s["slip"] = 1.5 / case["dt"] * s["U"]
    if kind in ("operators", "precond"):
        s["v"] = normal(m)   # a Krylov vector
    if kind in ("operators", "coupling"):
        s["u"] = g.flow()
        s["F"] = normal(nmk)
    return s


def prepare(case, seed):
    s = _inputs(case, seed)
    g = s["geometry"]
    s["kind"], s["case"], s["opts"] = case["kind"], case, _options(case)
    solver = IBMSolver(*g.n, h=g.h, Re=case["Re"], dt=case["dt"])
    s["solver"] = solver
    if case["kind"] in ("solve", "operators"):
        solver.set_markers(s["X"])
    if case["kind"] == "solve":
        s["b"] = solver.gradient_t(s["momentum"] + solver.spread(2.0 * s["slip"]))
    return s


def run(s):
    solver, kind = s["solver"], s["kind"]
    if kind == "step":
        solver.set_markers(s["X"])
        out, _ = solver.step(s["u_n"], s["u_nm1"], s["p_n"], s["F_n"], s["U"], s["f_body"],
                             **s["opts"])
        return out
    if kind == "solve":
        p, _ = solver.solve_schur(s["b"], **s["opts"])
        return dict(p=p)
    if kind == "adjoint":
        X = s["X"].clone().requires_grad_(True)
        U = s["U"].clone().requires_grad_(True)
        F, u, p = ib_step(solver, X, U, {k: s[k] for k in ("u_n", "u_nm1", "p_n", "F_n", "f_body")},
                          **s["opts"])
        loads = body_loads(solver, F, X, s["body_id"], s["centers"])
        X_bar, U_bar = torch.autograd.grad((s["w"] * loads).sum(), (X, U))
        return dict(loads=loads.detach(), u=u, p=p, F=F.detach(), X_bar=X_bar, U_bar=U_bar)
    if kind == "precond":
        return dict(z=solver.precond(s["v"], prec=IBM_PREC_FP64))
    if kind == "operators":
        return dict(G=solver.gradient(s["v"]), GT=solver.gradient_t(s["u"]),
                    L=solver.apply_laplacian(s["v"]), S=solver.apply_schur(s["v"]),
                    interp=solver.interp(s["u"]), spread=solver.spread(s["F"]),
                    F_corr=solver.force_correction(s["v"], s["F"]))
    if kind == "coupling":
        solver.set_markers(s["X"])
        return dict(interp=solver.interp(s["u"]), spread=solver.spread(s["F"]))
    if kind == "fsi":
        g = s["geometry"]
        spheres = RigidSpheres(g.radii, 1.05, g.centers, s["velocity"], s["omega"])
        out, _ = solver.fsi_step(spheres, s["L0"], s["body_id"], s["u_n"], s["u_nm1"], s["p_n"],
                                 s["F_n"], s["f_body"], gravity=(0.0, 0.0, -10.0), tol=0.0,
                                 max_inner=s["case"]["inner"], criterion=IBM_FSI_CRIT_EULERIAN,
                                 **s["opts"])
        return dict(out, xc=spheres.get("xc"), us=spheres.get("us"), om=spheres.get("om"),
                    rot=spheres.get("rot"))
    raise ValueError(kind)


def work(case):
    """Each input read once and each output written once, and the operations
    of one evaluation of the formulas (an iterative solve's iterations are not
    what the path cannot do without)."""
    n = (case["nx"], case["ny"], case["nz"])
    m = n[0] * n[1] * n[2]
    nf = sum((n[d] + 1) * (m // n[d]) for d in range(3))
    side = min(n) / max(n)
    r = 0.5 * (case["r_lo"] + case["r_hi"]) * side
    markers = case["bodies"] * 4.0 * math.pi * (r * max(n) * case["spacing"]) ** 2
    kind = case["kind"]
    if kind in ("step", "fsi"):
        # u^n, u^{n-1}, f, p^n in, u, p out; X, U, F^n in, F out
        return dict(bytes=8.0 * (4 * nf + 2 * m + 12 * markers), flops=60.0 * nf + 1500.0 * markers)
    if kind == "adjoint":
        # the step and, once more, u^{n+1} with the marker arrays and gradients
        return dict(bytes=8.0 * (5 * nf + 2 * m + 24 * markers), flops=70.0 * nf + 4000.0 * markers)
    if kind == "solve":
        return dict(bytes=16.0 * m, flops=13.0 * m)
    if kind == "precond":
        return dict(bytes=16.0 * m, flops=60.0 * m)
    if kind == "operators":
        # v, u, F in; G v, L v, S v, G^T u, R F and three marker vectors out
        return dict(bytes=8.0 * (3 * nf + 4 * m + 12 * markers), flops=2.0 * nf + 25.0 * m)
    # coupling: X, u, F in, R F and R^T u out
    return dict(bytes=8.0 * (2 * nf + 12 * markers), flops=1000.0 * markers)


# ---- the same in plain torch, 64 bits ---------------------------------------

def _phi(r):
    a = r.abs()
    inner = (1 + (1 - 3 * a * a).clamp(min=0).sqrt()) / 3
    outer = (5 - 3 * a - (1 - 3 * (1 - a) ** 2).clamp(min=0).sqrt()) / 6
    return torch.where(a <= 0.5, inner, torch.where(a <= 1.5, outer, torch.zeros_like(a)))


def _dphi(r):
    a = r.abs()
    inner = -r / (1 - 3 * r * r).clamp(min=1e-300).sqrt()
    q = 1 - a
    outer = -torch.sign(r) * 0.5 * (1 + q / (1 - 3 * q * q).clamp(min=1e-300).sqrt())
    return torch.where(a <= 0.5, inner, torch.where(a < 1.5, outer, torch.zeros_like(a)))


class _Exact:
    """The operators of the method on one grid with one set of markers."""

    def __init__(self, case, g, X):
        self.n, self.h, self.N = g.n, g.h, X.shape[1]
        self.shapes = [tuple(self.n[e] + (e == d) for e in (2, 1, 0)) for d in range(3)]
        self.cells = (self.n[2], self.n[1], self.n[0])
        self.a, self.nu = 1.5 / case["dt"], 1.0 / case["Re"]
        self.dt = case["dt"]
        # taps and weights of the markers: idx[d], w[d] (N, 27), and the
        # weights differentiated with respect to the marker's coordinates
        self.idx, self.w, self.dw = [], [], []
        for d in range(3):
            j, f, df = [], [], []
            for e in range(3):
                t = X[e] / self.h - (0.0 if e == d else 0.5)
                k = torch.floor(t + 0.5)[:, None] + torch.arange(-1, 2, device="cuda", dtype=F64)
                r = k - t[:, None]
                j.append(k.long())
                f.append(_phi(r))
                df.append(-_dphi(r) / self.h)
            nz, ny, nx = self.shapes[d]
            self.idx.append(((j[2][:, :, None, None] * ny + j[1][:, None, :, None]) * nx
                             + j[0][:, None, None, :]).reshape(self.N, 27))

            def outer(p):
                return (p[2][:, :, None, None] * p[1][:, None, :, None]
                        * p[0][:, None, None, :]).reshape(self.N, 27)

            self.w.append(outer(f))
            self.dw.append([outer([df[q] if q == e else f[q] for q in range(3)])
                            for e in range(3)])
        # cosine modes of the Neumann Laplacian
        self.Q, lam = [], []
        for e in range(3):
            i = torch.arange(self.n[e], device="cuda", dtype=F64)
            Q = torch.cos(math.pi / self.n[e] * (i[:, None] + 0.5) * i[None, :])
            self.Q.append(Q / Q.norm(dim=0))
            lam.append((2 - 2 * torch.cos(math.pi * i / self.n[e])) / self.h ** 2)
        ev = lam[2][:, None, None] + lam[1][None, :, None] + lam[0][None, None, :]
        ev[0, 0, 0] = math.inf
        self.inv_ev = 1.0 / ev

    def split(self, u):
        return [c.view(s) for c, s in zip(u.split([math.prod(s) for s in self.shapes]),
                                          self.shapes)]

    def G(self, p):
        p = p.view(self.cells)
        out = []
        for d in range(3):
            ax = 2 - d
            c = torch.zeros(self.shapes[d], device="cuda", dtype=F64)
            c.narrow(ax, 1, self.n[d] - 1).copy_(torch.diff(p, dim=ax) / self.h)
            out.append(c.view(-1))
        return torch.cat(out)

    def GT(self, u):
        out = 0.0
        for d, c in enumerate(self.split(u)):
            ax = 2 - d
            c = c.clone()
            c.select(ax, 0).zero_()
            c.select(ax, -1).zero_()
            out = out - torch.diff(c, dim=ax) / self.h
        return out.reshape(-1)

    def L(self, p):
        return self.GT(self.G(p))

    def L_inv(self, b):
        x = b.view(self.cells)
        for sign in (0, 1):
            if sign:
                x = x * self.inv_ev
            for e in range(3):
                Q = self.Q[e] if sign else self.Q[e].T
                x = torch.movedim(torch.tensordot(Q, x, dims=([1], [2 - e])), 0, 2 - e)
        return x.reshape(-1)

    def RT(self, u):
        return torch.cat([(c.reshape(-1)[i] * w).sum(1)
                          for c, i, w in zip(self.split(u), self.idx, self.w)])

    def R(self, F):
        out = []
        for d, f in enumerate(F.view(3, -1)):
            c = torch.zeros(math.prod(self.shapes[d]), device="cuda", dtype=F64)
            out.append(c.index_add_(0, self.idx[d].reshape(-1),
                                    (self.w[d] * f[:, None]).reshape(-1)))
        return torch.cat(out)

    def dR(self, f, m):
        """f^T (dR/dX) m for each marker and axis, (3, N)."""
        out = 0.0
        for c, i, dw, md in zip(self.split(f), self.idx, self.dw, m.view(3, -1)):
            v = c.reshape(-1)[i]
            out = out + torch.stack([(v * dw[e]).sum(1) * md for e in range(3)])
        return out

    def B(self, p):
        return self.RT(self.G(p))

    def BT(self, F):
        return self.GT(self.R(F))

    def C_factor(self):
        """Cholesky factors of the three blocks of C = R^T R."""
        out = []
        for d in range(3):
            rows = torch.arange(self.N, device="cuda")[:, None].expand(-1, 27)
            taps, inv = torch.unique(self.idx[d], return_inverse=True)
            M = torch.zeros((self.N, taps.numel()), device="cuda", dtype=F64)
            M[rows, inv] = self.w[d]
            out.append(torch.linalg.cholesky(M @ M.T))
        return out

    def schur_solve(self, b, exact_c=False):
        """Mean-zero p of S p = b by conjugate gradients with the exact L^+."""
        if exact_c:
            fac = self.C_factor()

            def c_inv(t):
                return torch.cat([torch.cholesky_solve(v[:, None], f)[:, 0]
                                  for v, f in zip(t.view(3, -1), fac)])
        else:
            def c_inv(t):
                return 2.0 * t
        S = lambda p: self.L(p) + self.BT(c_inv(self.B(p)))  # noqa: E731
        return _cg(S, b, self.L_inv, 1e-14)

    def advection(self, u):
        """div(u u_d) on the interior faces, central, no flux through walls."""
        uc = self.split(u)
        out = []
        for d in range(3):
            ad, nd = 2 - d, self.n[d]
            ud = uc[d]
            acc = torch.zeros(self.shapes[d], device="cuda", dtype=F64)
            inner = acc.narrow(ad, 1, nd - 1)
            for e in range(3):
                ae = 2 - e
                if e == d:
                    cc = 0.5 * (ud.narrow(ad, 0, nd) + ud.narrow(ad, 1, nd))
                    inner += torch.diff(cc * cc, dim=ad) / self.h
                    continue
                ne = self.n[e]
                ue = 0.5 * (uc[e].narrow(ad, 0, nd - 1) + uc[e].narrow(ad, 1, nd - 1))
                flux = torch.zeros_like(ue)
                v = 0.5 * (ud.narrow(ae, 0, ne - 1) + ud.narrow(ae, 1, ne - 1))
                flux.narrow(ae, 1, ne - 1).copy_(ue.narrow(ae, 1, ne - 1)
                                                 * v.narrow(ad, 1, nd - 1))
                inner += torch.diff(flux, dim=ae) / self.h
            out.append(acc.view(-1))
        return torch.cat(out)

    def mask(self, u):
        for d, c in enumerate(self.split(u)):
            c.select(2 - d, 0).zero_()
            c.select(2 - d, -1).zero_()
        return u

    def helmholtz(self, u):
        """a u - nu Lap u with no-slip walls, on the interior faces."""
        out = torch.empty_like(u)
        s = self.nu / self.h ** 2
        for d, (c, o) in enumerate(zip(self.split(u), self.split(out))):
            torch.mul(c, self.a + 6.0 * s, out=o)
            for e in range(3):
                ax, k = 2 - e, c.shape[2 - e]
                o.narrow(ax, 1, k - 1).sub_(c.narrow(ax, 0, k - 1), alpha=s)
                o.narrow(ax, 0, k - 1).sub_(c.narrow(ax, 1, k - 1), alpha=s)
                if e != d:   # ghost value beyond the wall: minus the first one
                    for q in (0, k - 1):
                        o.select(ax, q).add_(c.select(ax, q), alpha=s)
        return self.mask(out)

    def step(self, s):
        rhs = ((4.0 * s["u_n"] - s["u_nm1"]) / (2.0 * self.dt) - self.G(s["p_n"])
               + self.R(s["F_n"]) + s["f_body"] - self.advection(s["u_n"]))
        us = _cg(self.helmholtz, self.mask(rhs), None, 1e-14)
        rhs_F = self.a * (self.RT(us) - s["U"])
        p = self.schur_solve(self.a * self.GT(us) + 2.0 * self.BT(rhs_F))
        F = 2.0 * (self.B(p) - rhs_F)
        u = us + (2.0 * self.dt / 3.0) * (self.R(F) - self.G(p))
        return dict(u=u, p=s["p_n"] + p, F=s["F_n"] + F), F

    def precond(self, b, pre=2, post=2):
        """One V-cycle: Chebyshev smoothing on D^{-1} L with roots on [0.3, 2],
        8-cell averages down, trilinear interpolation up, pseudo-inverse at
        the coarsest level."""
        def weights(p):
            return [1.0 / (1.15 + 0.85 * math.cos((2 * i + 1) * math.pi / (2 * p)))
                    for i in range(p)]

        def lap(x, h):
            out = torch.zeros_like(x)
            for ax in range(3):
                k = x.shape[ax]
                g = torch.diff(x, dim=ax)
                out.narrow(ax, 0, k - 1).sub_(g)
                out.narrow(ax, 1, k - 1).add_(g)
            return out / h ** 2

        def diag(x, h):
            nn = torch.zeros_like(x)
            for ax in range(3):
                k = x.shape[ax]
                nn.narrow(ax, 0, k - 1).add_(1.0)
                nn.narrow(ax, 1, k - 1).add_(1.0)
            return nn / h ** 2

        def up(x):
            for ax in range(3):
                k = x.shape[ax]
                lo = torch.cat([x.narrow(ax, 0, 1), x.narrow(ax, 0, k - 1)], ax)
                hi = torch.cat([x.narrow(ax, 1, k - 1), x.narrow(ax, k - 1, 1)], ax)
                x = torch.stack([0.75 * x + 0.25 * lo, 0.75 * x + 0.25 * hi], ax + 1).flatten(
                    ax, ax + 1)
            return x

        def cycle(b, h):
            s = b.shape
            if any(k % 2 or k < 4 for k in s) or b.numel() <= 64:
                eye = torch.eye(b.numel(), device="cuda", dtype=F64).view(-1, *s)
                A = torch.stack([lap(v, h).reshape(-1) for v in eye])
                one = 1.0 / b.numel()
                return ((torch.linalg.inv(A + one) - one) @ b.reshape(-1)).view(s)
            D = diag(b, h)
            x = torch.zeros_like(b)
            for w in weights(pre):
                x = x + w * (b - lap(x, h)) / D
            r = (b - lap(x, h)).view(s[0] // 2, 2, s[1] // 2, 2, s[2] // 2, 2).mean((1, 3, 5))
            x = x + up(cycle(r, 2 * h))
            for w in weights(post):
                x = x + w * (b - lap(x, h)) / D
            return x

        return cycle(b.view(self.cells), self.h).reshape(-1)


def _cg(A, b, M, rtol, most=120):
    """Preconditioned conjugate gradients to the last digits."""
    x = torch.zeros_like(b)
    r = b.clone()
    z = M(r) if M else r
    p, rz, stop = z.clone(), torch.dot(r, z), rtol * torch.linalg.vector_norm(b)
    for _ in range(most):
        q = A(p)
        alpha = rz / torch.dot(p, q)
        x += alpha * p
        r -= alpha * q
        if torch.linalg.vector_norm(r) <= stop:
            break
        z = M(r) if M else r
        new = torch.dot(r, z)
        p.mul_(new / rz).add_(z)
        rz = new
    return x - x.mean() if M else x


def exact(case, seed):
    kind = case["kind"]
    if kind == "fsi":
        return None   # the bodies' volume fractions and corrections have no short restatement
    s = _inputs(case, seed)
    E = _Exact(case, s["geometry"], s["X"])
    if kind == "step":
        return E.step(s)[0]
    if kind == "solve":
        b = E.GT(s["momentum"] + E.R(2.0 * s["slip"]))
        return dict(p=E.schur_solve(b, case["exact_c"]))
    if kind == "precond":
        return dict(z=E.precond(s["v"]))
    if kind == "operators":
        return dict(G=E.G(s["v"]), GT=E.GT(s["u"]), L=E.L(s["v"]),
                    S=E.L(s["v"]) + 2.0 * E.BT(E.B(s["v"])), interp=E.RT(s["u"]),
                    spread=E.R(s["F"]), F_corr=2.0 * (E.B(s["v"]) - s["F"]))
    if kind == "coupling":
        return dict(interp=E.RT(s["u"]), spread=E.R(s["F"]))
    # adjoint, from rest (F^n = 0)
    out, F_corr = E.step(s)
    F, X, h3 = out["F"].view(3, -1), s["X"], E.h ** 3
    bid = s["body_id"].long()
    arm = X - s["centers"].cuda().T[:, bid]
    per_marker = torch.cat([F, torch.linalg.cross(arm, F, dim=0)])
    loads = torch.zeros((s["w"].shape[0], 6), device="cuda", dtype=F64)
    loads.index_add_(0, bid, h3 * per_marker.T.contiguous())
    wF, wT = s["w"].cuda()[bid].T.reshape(2, 3, -1)
    F_bar = (h3 * (wF + torch.linalg.cross(wT, arm, dim=0))).reshape(-1)
    lam = E.schur_solve(2.0 * E.BT(F_bar))
    U_bar = 2.0 * E.a * (F_bar - E.B(lam))
    X_bar = (E.dR(E.R(F_corr) - E.a * out["u"], U_bar / E.a) - E.dR(E.G(lam), F_corr)
             + h3 * torch.linalg.cross(F, wT, dim=0))
    return dict(out, loads=loads, X_bar=X_bar, U_bar=U_bar)
