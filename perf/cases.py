"""Performance cases of the solver: the work that its users have it do, through its public entry points.

A case is a dict of plain values.  ``listed()`` gives the fixed ones, ``draw(rng)`` one more of the
same ranges, ``prepare(case, seed)`` what a program has in hand before the call (initial state,
solver context), ``run(state)`` one pass, ``work(case)`` the bytes and operations that a pass cannot
do without, and ``exact(case, seed)`` the pass in plain torch in 64 bits, without the library.

Every pass starts from the same initial state: a call advances its state in place, so ``run``
first copies the initial state into the working one, as a program that runs a study from one
initial state does.
"""
from __future__ import annotations

import math

import numpy as np
import torch

import paper_2306_05002_gb300 as dg
from paper_2306_05002_gb300 import adjoint as A
from paper_2306_05002_gb300 import workloads as W

# Kinds of cases, each one entry point in its own use:
#   step      Solver.dg_step: SSP-RK3 steps of one problem on a device state
#   host      Solver.dg_step on a page-locked host state
#   batch     BatchSolver.dg_batch_step: many problems of mixed size and order
#   rhs       adjoint.DGRHS: one right-hand side and its gradient
#   traj      adjoint.DGTrajectory: a checkpointed trajectory and its gradient
#   kin       KinematicSolver.dg_kin_step on rectangles ("quad") or triangles ("tri")
#   reinit    Solver.dg_reinit: level-set re-initialisation


def listed():
    return [
        # The 1D slab advection (100 elements, p = 3): the smallest problem there is, where a step is
        # launches and latency.
        dict(name="slab1d_fp32", kind="step", problem="slab", n=100, p=3, precision="fp32bulk", steps=50),
        # The 2D drop on 64 x 64 elements, p = 3, the benchmark's own problem, in both precisions.
        dict(name="drop64p3_fp32", kind="step", problem="drop", n=64, p=3, precision="fp32bulk", steps=20),
        dict(name="drop64p3_fp64", kind="step", problem="drop", n=64, p=3, precision="fp64", steps=10),
        # Viscous Rayleigh-Taylor with gravity, surface tension and walls on 256 x 256 elements, p = 4:
        # the largest single problem of the benchmark.
        dict(name="rt256p4_fp32", kind="step", problem="rt", n=256, p=4, precision="fp32bulk", steps=10),
        # The rising bubble on 20 x 40 elements, p = 4: every term of the model and the pressure
        # boundary in full precision, a mesh that fills no more than a part of the GPU.
        dict(name="bubble20p4_fp64", kind="step", problem="bubble", n=20, p=4, precision="fp64", steps=10),
        # An ensemble of drops and bubbles of uneven sizes (16 to 128 elements a side) and orders 2 to 5.
        dict(name="ensemble32_fp32", kind="batch", count=32, nmin=16, nmax=128, mix=4, steps=4),
        # One right-hand side with its gradient, as a term of a larger differentiable program.
        dict(name="rhs64p3_grad", kind="rhs", n=64, p=3),
        # Gradient of a trajectory with respect to its initial state: 20 steps, a checkpoint every 10.
        dict(name="traj128p3_grad", kind="traj", n=128, p=3, steps=20, every=10),
        # The Rider-Kothe vortex in the kinematic mode, rectangles and triangles.
        dict(name="vortex64p3_quad", kind="kin", elem="quad", n=64, p=3, steps=20),
        dict(name="vortex32p3_tri", kind="kin", elem="tri", n=32, p=3, steps=20),
        # Level-set re-initialisation with the paper's 50 iterations.
        dict(name="reinit64p3", kind="reinit", n=64, p=3, niter=50),
        # One step on a page-locked host state, read and written back by the call: a host program that
        # looks at every step's result.
        dict(name="drop64p3_host", kind="host", problem="drop", n=64, p=3, precision="fp32bulk", steps=1),
    ]


def _log_int(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def draw(rng):
    kind = rng.choice(["step", "step", "step", "step", "batch", "rhs", "traj", "kin", "kin", "reinit", "host"])
    if kind == "step":
        problem = rng.choice(["slab", "drop", "rt", "bubble"])
        precision = rng.choice(["fp32bulk", "fp64"])
        p = rng.randint(1, 5)
        big = 200 if precision == "fp32bulk" else 120
        n = {"slab": _log_int(rng, 10, 1000), "drop": _log_int(rng, 8, big), "rt": _log_int(rng, 12, big),
             "bubble": _log_int(rng, 6, 40)}[problem]
        return dict(kind=kind, problem=problem, n=n, p=p, precision=precision, steps=rng.randint(1, 12))
    if kind == "batch":
        lo = _log_int(rng, 8, 32)
        return dict(kind=kind, count=rng.randint(2, 32), nmin=lo, nmax=lo * rng.randint(1, 4),
                    mix=rng.randint(0, 9999), steps=rng.randint(1, 4))
    if kind == "rhs":
        return dict(kind=kind, n=_log_int(rng, 8, 160), p=rng.randint(1, 5))
    if kind == "traj":
        steps = rng.randint(2, 12)
        return dict(kind=kind, n=_log_int(rng, 8, 100), p=rng.randint(1, 4), steps=steps, every=rng.randint(1, steps))
    if kind == "kin":
        elem = rng.choice(["quad", "tri"])
        return dict(kind=kind, elem=elem, n=_log_int(rng, 8, 128 if elem == "quad" else 64),
                    p=rng.randint(1, 5 if elem == "quad" else 4), steps=rng.randint(1, 20))
    if kind == "reinit":
        return dict(kind=kind, n=_log_int(rng, 8, 160), p=rng.randint(1, 5), niter=rng.randint(5, 50))
    return dict(kind="host", problem="drop", n=_log_int(rng, 16, 96), p=rng.randint(2, 5), precision="fp32bulk",
                steps=rng.randint(1, 3))


# ---------------------------------------------------------------------------
# Problems
# ---------------------------------------------------------------------------

def _problem(case, seed):
    """The workload of a single-problem case; the seed moves the drop, the interface, the flow."""
    rng = np.random.default_rng(seed)
    kind, n, p = case["kind"], case["n"], case["p"]
    if kind == "kin":
        c = rng.uniform(-0.1, 0.1, size=2)
        return W.rider_kothe(n=n, p=p, elem=case["elem"], center=(float(c[0]), 0.25 + float(c[1])))
    if kind in ("rhs", "traj"):
        theta = rng.normal(0.0, 0.01, size=16)
        wl = W.adjoint_drop(n=n, p=p, seed=int(rng.integers(1 << 30)), theta=theta, u=float(rng.uniform(0.5, 1.5)))
        return wl
    if kind == "reinit":
        return W.drop_2d(n=n, p=p, seed=int(rng.integers(1 << 30)), R=float(rng.uniform(0.1, 0.3)))
    problem = case["problem"]
    if problem == "slab":
        wl = W.slab_1d(nx=n, p=p, u=float(rng.uniform(0.5, 1.5)), P0=float(rng.uniform(0.9e5, 1.1e5)))
        return wl
    if problem == "drop":
        return W.drop_2d(n=n, p=p, seed=int(rng.integers(1 << 30)), R=float(rng.uniform(0.1, 0.2)),
                         u=float(rng.uniform(0.5, 1.5)), v=float(rng.uniform(-1.0, 1.0)))
    if problem == "rt":
        return W.rayleigh_taylor(n=n, p=p, seed=int(rng.integers(1 << 30)), amp=float(rng.uniform(0.005, 0.02)))
    wl = W.rising_bubble(nx=n, ny=2 * n, p=p, case=int(rng.integers(1, 3)), nquad=400)
    # a bubble that already rises: a divergence-free stir that vanishes at the walls and the top
    x, y = W.node_coords(wl)
    amp = float(rng.uniform(0.02, 0.05))
    u = amp * np.sin(2 * np.pi * x) * np.cos(np.pi * y)
    v = -2.0 * amp * np.cos(2 * np.pi * x) * np.sin(np.pi * y)
    rho = wl.w[2] + wl.w[3]
    wl.w = wl.w.copy()
    wl.w[4], wl.w[5] = rho * u, rho * v
    wl.w[6] += 0.5 * rho * (u * u + v * v)
    return wl


def _members(case):
    """Sizes and orders of an ensemble's problems: by the case alone, so that a case is one amount of work."""
    r = np.random.default_rng(case["mix"])
    return [(int(r.integers(case["nmin"], case["nmax"] + 1)), int(r.choice((2, 3, 4, 5)))) for _ in range(case["count"])]


def _ensemble(case, seed):
    r = np.random.default_rng(seed)
    out = []
    for n, p in _members(case):
        out.append(W.drop_2d(n=n, p=p, R=float(r.uniform(0.05, 0.2)), center=r.uniform(0.0, 1.0, size=2),
                             water_inside=bool(r.integers(0, 2))))
    return out


def prepare(case, seed):
    kind = case["kind"]
    s = dict(case=case)
    if kind == "batch":
        wls = _ensemble(case, seed)
        s["solver"] = dg.BatchSolver(wls)
        s["w0"] = [torch.from_numpy(wl.w.copy()).cuda() for wl in wls]
        s["w"] = [torch.empty_like(w) for w in s["w0"]]
        s["dt"] = [wl.dt for wl in wls]
        return s
    wl = _problem(case, seed)
    s["dt"] = wl.dt
    if kind == "kin":
        s["solver"] = dg.KinematicSolver(wl)
    else:
        s["solver"] = dg.Solver(wl, precision=case.get("precision", "fp64"))
    w0 = torch.from_numpy(np.ascontiguousarray(wl.w))
    if kind == "host":
        s["w0"] = w0.clone()
        s["w"] = torch.empty_like(w0).pin_memory()
        return s
    s["w0"] = w0.cuda()
    if kind in ("rhs", "traj"):
        g = torch.Generator().manual_seed(seed)
        # the seed of the reverse sweep: the gradient of a misfit, in the scale of each variable
        scale = 1.0 / w0.abs().amax(dim=1, keepdim=True).clamp_min(1e-3)
        s["lam"] = (torch.randn(w0.shape, generator=g, dtype=torch.float64) * scale).cuda()
        s["w0"].requires_grad_()
    else:
        s["w"] = torch.empty_like(s["w0"])
    return s


def run(s):
    case = s["case"]
    kind = case["kind"]
    solver = s["solver"]
    if kind == "batch":
        torch._foreach_copy_(s["w"], s["w0"])
        solver.dg_batch_step(s["w"], s["dt"], case["steps"])
        return s["w"]
    if kind in ("rhs", "traj"):
        w0 = s["w0"]
        if kind == "rhs":
            out = A.DGRHS.apply(w0, solver)
        else:
            out = A.DGTrajectory.apply(w0, solver, s["dt"], case["steps"], case["every"])
        (grad,) = torch.autograd.grad(out, w0, s["lam"])
        return [out.detach(), grad]
    w = s["w"]
    w.copy_(s["w0"])
    if kind == "kin":
        return solver.dg_kin_step(w, 0.0, s["dt"], case["steps"])
    if kind == "reinit":
        return solver.dg_reinit(w, case["niter"])
    return solver.dg_step(w, s["dt"], case["steps"])


# ---------------------------------------------------------------------------
# Necessary work
# ---------------------------------------------------------------------------

def _model_flops(dim, p, viscous, st):
    """Operations per node and right-hand side: closure, gradients, normal, a_1, fluxes, flux divergence,
    transport; half of a face's numerical fluxes per side (they are shared), their lifting, the update."""
    P1 = p + 1
    face = 2 * dim / P1 if dim == 2 else 2.0 / P1  # face nodes per node
    f = 25 + 4 * dim * P1 + 6 + 10 + 40 + 12 * dim * P1 + 8 + face * (5 + 0.5 * 130) + 16 * dim + 14
    if viscous:
        f += 4 * dim * P1 + 32 + face * 15
    if st:
        f += 2 * dim * P1 + 8
    return f


def work(case):
    kind = case["kind"]
    if kind == "batch":
        nb = fl = 0.0
        for n, p in _members(case):
            N = n * n * (p + 1) ** 2
            nb += 2 * 56.0 * N
            fl += 3.0 * case["steps"] * N * _model_flops(2, p, False, False)
        return {"bytes": nb, "flops": fl}
    n, p = case["n"], case["p"]
    P1 = p + 1
    if kind == "kin":
        if case["elem"] == "quad":
            N = n * n * P1 * P1
            f = 8 * P1 + 4 * P1 + 35 + 4.0 / P1 * 20 + 12 + 6
        else:
            npt, nq, ne = P1 * (P1 + 1) // 2, (p + 2) ** 2, 3 * (p + 2)
            N = 2 * n * n * npt
            per = nq * (10 * npt + 45) + ne * (6 * P1 + 4 * npt + 25) + npt * (8 * nq + 2 * ne + 4 * (p + 2)) + 4 * npt * npt
            f = per / npt
        return {"bytes": 2 * 16.0 * N, "flops": 4.0 * case["steps"] * N * f}
    if kind == "reinit":
        N = n * n * P1 * P1
        return {"bytes": 8.0 * N * 2, "flops": 3.0 * case["niter"] * N * (8 * P1 + 10 + 4.0 / P1 * 5 + 12)}
    slab = case.get("problem") == "slab"
    bubble = case.get("problem") == "bubble"
    full = case.get("problem") in ("rt", "bubble")
    dim = 1 if slab else 2
    N = n * P1 if slab else (2 if bubble else 1) * n * n * P1 * P1
    f = _model_flops(dim, p, full, full)
    if kind == "rhs":      # the state and the seed in, the right-hand side and the gradient out
        return {"bytes": 4 * 56.0 * N, "flops": 4.0 * N * f}
    if kind == "traj":     # forward, and about three times that for the gradient
        return {"bytes": 4 * 56.0 * N, "flops": 3.0 * case["steps"] * N * 4.0 * f}
    return {"bytes": 2 * 56.0 * N, "flops": 3.0 * case["steps"] * N * f}


# ---------------------------------------------------------------------------
# The same in plain torch, 64 bits
# ---------------------------------------------------------------------------

def _device():
    return "cuda" if torch.cuda.is_available() else "cpu"


def _t(a):
    return torch.tensor(np.asarray(a), dtype=torch.float64, device=_device())


def _gll(p):
    """Gauss-Lobatto-Legendre nodes, weights and the Lagrange derivative matrix on [-1, 1]."""
    L = np.polynomial.legendre.Legendre.basis(p)
    x = np.concatenate([[-1.0], np.sort(L.deriv().roots().real), [1.0]])
    for _ in range(3):  # polish the inner nodes: Newton on L'
        x[1:-1] -= L.deriv()(x[1:-1]) / L.deriv(2)(x[1:-1]) if p > 1 else 0.0
    w = 2.0 / (p * (p + 1) * L(x) ** 2)
    D = np.zeros((p + 1, p + 1))
    for a in range(p + 1):
        for b in range(p + 1):
            if a != b:
                D[a, b] = L(x[a]) / (L(x[b]) * (x[a] - x[b]))
    D[np.arange(p + 1), np.arange(p + 1)] = -D.sum(axis=1)
    return x, w, D


class _Grid:
    """Rectangles as tensors (..., ny, nx, j, i): derivatives, face traces, the neighbours' traces."""

    def __init__(self, dim, nx, ny, p, hx, hy, bc):
        self.dim, self.nx, self.ny, self.p, self.bc = dim, nx, ny, p, bc
        x, w, D = _gll(p)
        Dh = w[None, :] * D.T / w[:, None]
        self.x, self.w = x, w
        self.Dx, self.Dhx = _t(D * 2 / hx), _t(Dh * 2 / hx)
        self.Dy, self.Dhy = _t(D * 2 / hy), _t(Dh * 2 / hy)
        self.mx, self.my = _t(2 / (hx * w)), _t(2 / (hy * w))  # face weight times M^-1 along the normal line
        P1 = p + 1
        self.shape = (ny, nx, P1 if dim == 2 else 1, P1)

    def field(self, w):
        return w.reshape(w.shape[:-1] + self.shape)

    def dx(self, f):
        return torch.einsum("ic,...c->...i", self.Dx, f)

    def dy(self, f):
        return torch.einsum("jc,...ci->...ji", self.Dy, f)

    def div(self, fx, fy):
        r = torch.einsum("ic,...c->...i", self.Dhx, fx)
        return r + torch.einsum("jc,...ci->...ji", self.Dhy, fy) if self.dim == 2 else r

    def faces(self):
        """(axis, side, own line index, sign): west, east, south, north."""
        return [(0, 0, 0, -1.0), (0, 1, self.p, 1.0), (1, 2, 0, -1.0), (1, 3, self.p, 1.0)][: 2 * self.dim]

    def own(self, f, axis, idx):
        return f[..., idx] if axis == 0 else f[..., idx, :]

    def across(self, f, axis, idx, sg):
        """The neighbour's trace on the face; wrapped round at the ends of the mesh (walls: not used)."""
        g = self.own(f, axis, self.p - idx)
        return torch.roll(g, -int(sg), dims=-2 if axis == 0 else -3)

    def wall(self, axis, side):
        """Mask of the elements whose face is a boundary, or None when the direction is periodic."""
        if self.bc[side] in ("periodic", 0):
            return None
        m = torch.zeros((self.ny, self.nx, 1), dtype=torch.bool, device=self.Dx.device)
        if axis == 0:
            m[:, 0 if side == 0 else -1] = True
        else:
            m[0 if side == 2 else -1] = True
        return m

    def lift(self, R, axis, idx, sg, S, sym):
        """R + the face term at the face nodes and the symmetric term along the normal line, M^-1 applied."""
        if axis == 0:
            e = torch.zeros(self.p + 1, dtype=torch.float64, device=R.device)
            e[idx] = 1.0
            R = R + S[..., None] * (e * self.mx)
            return R if sym is None else R + sym[..., None] * (sg * self.Dx[idx] * self.mx)
        e = torch.zeros(self.p + 1, dtype=torch.float64, device=R.device)
        e[idx] = 1.0
        R = R + S[..., None, :] * (e * self.my)[:, None]
        return R if sym is None else R + sym[..., None, :] * (sg * self.Dy[idx] * self.my)[:, None]


def _normal(gx, gy):
    g2 = gx * gx + gy * gy
    ok = g2 >= 1e-24
    r = torch.where(ok, torch.rsqrt(torch.where(ok, g2, torch.ones_like(g2))), torch.zeros_like(g2))
    return gx * r, gy * r


class _Model:
    """The semi-discrete right-hand side of the five-equation model with the Allen-Cahn phase field."""

    def __init__(self, wl):
        self.wl = wl
        hy = wl.hy if wl.dim == 2 else 1.0
        self.g = _Grid(wl.dim, wl.nx, wl.ny, wl.p, wl.hx, hy, wl.bc)
        self.C = [wl.gamma[l] * wl.pinf[l] / (wl.gamma[l] - 1.0) for l in range(2)]
        self.i = [1.0 / (wl.gamma[l] - 1.0) for l in range(2)]
        P1 = wl.p + 1
        self.eta = (wl.c_ip * P1 * P1 / wl.hx, wl.c_ip * P1 * P1 / hy)

    def closure(self, phi, m1, m2, ru, rv, rE):
        wl = self.wl
        rho = m1 + m2
        u, v = ru / rho, rv / rho
        Cm = phi * self.C[0] + (1 - phi) * self.C[1]
        den = phi * self.i[0] + (1 - phi) * self.i[1]
        P = (rE - 0.5 * (ru * ru + rv * rv) / rho - Cm) / den
        c = torch.sqrt((P + (P + Cm) / den) / rho)
        Bp = wl.gamma[0] / (wl.gamma[0] - 1.0) - wl.gamma[1] / (wl.gamma[1] - 1.0)
        return rho, u, v, P, c, P * Bp + (self.C[0] - self.C[1])

    def rhs(self, w):
        wl, g = self.wl, self.g
        two = wl.dim == 2
        q = g.field(w)
        phi, psi, m1, m2, ru, rv, rE = q.unbind(0)
        if not two:
            rv = torch.zeros_like(rv)
        rho, u, v, P, c, B = self.closure(phi, m1, m2, ru, rv, rE)
        zero = torch.zeros_like(phi)
        gpx, gsx = g.dx(phi), g.dx(psi)
        gpy, gsy = (g.dy(phi), g.dy(psi)) if two else (zero, zero)
        nx, ny = _normal(gsx, gsy)
        r1, r2 = wl.rho0
        dr = r1 - r2
        sp = phi * (1 - phi)
        ax, ay = wl.Gamma * (wl.eps * gpx - sp * nx), wl.Gamma * (wl.eps * gpy - sp * ny)
        k = 0.5 * (u * u + v * v)
        cE = dr * k + B
        txx = txy = tyy = mu = zero
        if wl.viscous:
            mu = wl.mu[0] * phi + wl.mu[1] * (1 - phi)
            gux, gvx, guy, gvy = g.dx(u), g.dx(v), g.dy(u), g.dy(v)
            d3 = (gux + gvy) / 3.0
            txx, tyy, txy = 2 * mu * (gux - d3), 2 * mu * (gvy - d3), mu * (guy + gvx)
        Fx = torch.stack([-ax, m1 * u - r1 * ax, m2 * u + r2 * ax, ru * u + P - dr * ax * u - txx,
                          rv * u - dr * ax * v - txy, (rE + P) * u - cE * ax - (txx * u + txy * v)])
        Fy = torch.stack([-ay, m1 * v - r1 * ay, m2 * v + r2 * ay, ru * v - dr * ay * u - txy,
                          rv * v + P - dr * ay * v - tyy, (rE + P) * v - cE * ay - (txy * u + tyy * v)])
        R = g.div(Fx, Fy)
        src = [-(u * gpx + v * gpy), zero, zero, zero, zero, zero]
        Rpsi = -(u * gsx + v * gsy)
        if wl.gravity:
            src[3] = src[3] + rho * wl.g[0]
            src[4] = src[4] + rho * wl.g[1]
            src[5] = src[5] + rho * (wl.g[0] * u + wl.g[1] * v)
        if wl.surface_tension:
            kappa = -(g.dx(nx) + (g.dy(ny) if two else zero))
            s = wl.sigma * kappa * torch.sqrt(gpx * gpx + gpy * gpy)
            src[3] = src[3] + s * nx
            src[4] = src[4] + s * ny
            src[5] = src[5] + s * (u * nx + v * ny)
        R = R + torch.stack(src)
        fields = torch.stack([phi, psi, m1, m2, ru, rv, rE])
        for axis, side, idx, sg in g.faces():
            normal = torch.stack([gpx, nx, txx, txy]) if axis == 0 else torch.stack([gpy, ny, txy, tyy])
            Wm, Wp = g.own(fields, axis, idx), g.across(fields, axis, idx, sg)
            Nm, Np = g.own(normal, axis, idx), g.across(normal, axis, idx, sg)
            wall = g.wall(axis, side)
            if wall is not None:
                ghost = self.ghost(Wm, axis, wl.bc[side], wl.p_bc[side])
                Wp = torch.where(wall, ghost, Wp)
                Np = torch.where(wall, Nm, Np)
            a = [t for t in Wm.unbind(0)]
            b = [t for t in Wp.unbind(0)]
            _, um, vm, Pm, cm, Bm = self.closure(a[0], *a[2:])
            _, up, vp, Pp, cp, Bq = self.closure(b[0], *b[2:])
            unm, unp = ((um, up) if axis == 0 else (vm, vp))
            unm, unp = sg * unm, sg * unp
            lam = torch.maximum(unm.abs() + cm, unp.abs() + cp)

            def flux(t, un, P_):
                f = [t[2] * un, t[3] * un, t[4] * un, t[5] * un, (t[6] + P_) * un]
                f[2 + axis] = f[2 + axis] + P_ * sg
                return torch.stack(f)
            S = -(0.5 * (flux(a, unm, Pm) + flux(b, unp, Pp)) - 0.5 * lam * (Wp[2:] - Wm[2:]))
            Sphi = (lam - unm) * 0.5 * (b[0] - a[0])
            Spsi = (lam - unm) * 0.5 * (b[1] - a[1])
            jump = b[0] - a[0]
            sharp = 0.5 * sg * (b[0] * (1 - b[0]) * Np[1] + a[0] * (1 - a[0]) * Nm[1])
            ahat = wl.Gamma * (wl.eps * (0.5 * sg * (Np[0] + Nm[0]) + self.eta[axis] * jump) - sharp)
            sym = -0.5 * wl.Gamma * wl.eps * jump
            if wall is not None:
                ahat = torch.where(wall, torch.zeros_like(ahat), ahat)
                sym = torch.where(wall, torch.zeros_like(sym), sym)
            km, kp = 0.5 * (um * um + vm * vm), 0.5 * (up * up + vp * vp)
            one = torch.ones_like(jump)
            Cq = torch.stack([one, r1 * one, -r2 * one, dr * 0.5 * (um + up), dr * 0.5 * (vm + vp),
                              0.5 * (Bm + Bq) + dr * 0.5 * (km + kp)])
            S = torch.cat([Sphi[None], S]) + Cq * ahat
            if wl.viscous:
                def mix(f):
                    return wl.mu[0] * f + wl.mu[1] * (1 - f)
                em = self.eta[axis] * 0.5 * (mix(a[0]) + mix(b[0]))
                tmx, tmy, tpx, tpy = sg * Nm[2], sg * Nm[3], sg * Np[2], sg * Np[3]
                S = S + torch.stack([0 * jump, 0 * jump, 0 * jump, 0.5 * (tmx + tpx) + em * (up - um),
                                     0.5 * (tmy + tpy) + em * (vp - vm),
                                     0.5 * (tmx * um + tmy * vm + tpx * up + tpy * vp) + em * (kp - km)])
            R = g.lift(R, axis, idx, sg, S, Cq * sym)
            Rpsi = g.lift(Rpsi, axis, idx, sg, Spsi, None)
        out = torch.cat([R[:1], Rpsi[None], R[1:]])
        if not two:
            out = out * _t([1, 1, 1, 1, 1, 0, 1]).reshape(7, 1, 1, 1, 1)
        return out.reshape(7, -1)

    def ghost(self, Wm, axis, bc, pb):
        phi, psi, m1, m2, ru, rv, rE = Wm.unbind(0)
        if bc == "pressure":
            den = phi * self.i[0] + (1 - phi) * self.i[1]
            E = pb * den + phi * self.C[0] + (1 - phi) * self.C[1]
            return torch.stack([phi, psi, m1, m2, 0 * ru, 0 * rv, E])
        flip = [axis == 0 or bc == "noslip", axis == 1 or bc == "noslip"]
        return torch.stack([phi, psi, m1, m2, -ru if flip[0] else ru, -rv if flip[1] else rv, rE])

    def step(self, w, dt):
        w1 = w + dt * self.rhs(w)
        w2 = 0.75 * w + 0.25 * (w1 + dt * self.rhs(w1))
        return w / 3.0 + 2.0 / 3.0 * (w2 + dt * self.rhs(w2))


def _kin_quad(wl, steps):
    g = _Grid(2, wl.nx, wl.ny, wl.p, wl.hx, wl.hy, ("periodic",) * 4)
    P1 = wl.p + 1
    xc = _t(wl.x0 + wl.hx * (np.arange(wl.nx)[:, None] + 0.5 * (g.x[None] + 1)))[None, :, None, :]
    yc = _t(wl.y0 + wl.hy * (np.arange(wl.ny)[:, None] + 0.5 * (g.x[None] + 1)))[:, None, :, None]
    stream = torch.sin(math.pi * (xc - wl.xc + 0.5)) ** 2 * torch.sin(math.pi * (yc - wl.yc + 0.5)) ** 2 / math.pi
    U, V = g.dy(stream), -g.dx(stream)
    eta = (P1 * P1 / wl.hx * wl.c_ip, P1 * P1 / wl.hy * wl.c_ip)

    def rhs(w, t):
        c = math.cos(math.pi * t / wl.T)
        u, v = c * U, c * V
        phi, psi = g.field(w).unbind(0)
        gpx, gpy, gsx, gsy = g.dx(phi), g.dy(phi), g.dx(psi), g.dy(psi)
        nx, ny = _normal(gsx, gsy)
        sp = phi * (1 - phi)
        ax, ay = wl.Gamma * (wl.eps * gpx - sp * nx), wl.Gamma * (wl.eps * gpy - sp * ny)
        Rp = g.div(-ax, -ay) - (u * gpx + v * gpy)
        Rs = -(u * gsx + v * gsy)
        for axis, side, idx, sg in g.faces():
            st = torch.stack([phi, psi, gpx if axis == 0 else gpy, nx if axis == 0 else ny, u if axis == 0 else v])
            a, b = g.own(st, axis, idx).unbind(0), g.across(st, axis, idx, sg).unbind(0)
            unm, unp = sg * a[4], sg * b[4]
            lam = torch.maximum(unm.abs(), unp.abs())
            jump = b[0] - a[0]
            sharp = 0.5 * sg * (b[0] * (1 - b[0]) * b[3] + a[0] * (1 - a[0]) * a[3])
            ahat = wl.Gamma * (wl.eps * (0.5 * sg * (a[2] + b[2]) + eta[axis] * jump) - sharp)
            Rp = g.lift(Rp, axis, idx, sg, (lam - unm) * 0.5 * jump + ahat, -0.5 * wl.Gamma * wl.eps * jump)
            Rs = g.lift(Rs, axis, idx, sg, (lam - unm) * 0.5 * (b[1] - a[1]), None)
        return torch.stack([Rp, Rs]).reshape(2, -1)
    return _rk4(rhs, _t(wl.w), wl.dt, steps)


def _rk4(rhs, w, dt, steps):
    for k in range(steps):
        t = k * dt
        k1 = rhs(w, t)
        k2 = rhs(w + 0.5 * dt * k1, t + 0.5 * dt)
        k3 = rhs(w + 0.5 * dt * k2, t + 0.5 * dt)
        k4 = rhs(w + dt * k3, t + dt)
        w = w + dt / 6.0 * (k1 + 2 * k2 + 2 * k3 + k4)
    return w


def _kin_tri(wl, steps):
    """Triangles: each cell's lower-right (type 0) and upper-left (type 1) one, nodal basis on the
    equispaced points, collapsed Gauss rule of (p+2)^2 points, (p+2)-point Gauss rule on the edges."""
    p, nx, ny, hx, hy = wl.p, wl.nx, wl.ny, wl.hx, wl.hy
    nodes = np.array([(-1 + 2 * i / p, -1 + 2 * j / p) for j in range(p + 1) for i in range(p + 1 - j)])
    powers = [(i, j) for j in range(p + 1) for i in range(p + 1 - j)]

    def mono(r, s, d=None):
        cols = []
        for i, j in powers:
            if d is None:
                cols.append(r ** i * s ** j)
            elif d == 0:
                cols.append(i * r ** max(i - 1, 0) * s ** j)
            else:
                cols.append(j * r ** i * s ** max(j - 1, 0))
        return np.stack(cols, axis=-1)
    Vinv = np.linalg.inv(mono(nodes[:, 0], nodes[:, 1]))

    def basis(r, s):
        return [mono(r, s, d) @ Vinv for d in (None, 0, 1)]
    gx, gw = np.polynomial.legendre.leggauss(p + 2)
    ga, gb = np.meshgrid(gx, gx)          # rows: b
    rv, sv = (0.5 * (1 + ga) * (1 - gb) - 1).ravel(), gb.ravel()
    wv = (gw[None, :] * gw[:, None] * 0.5 * (1 - gb)).ravel()
    B, Br, Bs = basis(rv, sv)
    Minv = np.linalg.inv((B * wv[:, None]).T @ B)
    re = np.stack([gx, -gx, -np.ones_like(gx)])
    se = np.stack([-np.ones_like(gx), gx, -gx])
    Be, Ber, Bes = basis(re, se)          # (3, k, n)
    verts = [np.array([[0, 0], [hx, 0], [hx, hy]]), np.array([[0, 0], [hx, hy], [0, hy]])]
    cell = np.stack(np.meshgrid(np.arange(nx), np.arange(ny)), axis=-1) * np.array([hx, hy]) + np.array([wl.x0, wl.y0])
    geo = []
    for v in verts:
        xr, xs = 0.5 * (v[1] - v[0]), 0.5 * (v[2] - v[0])
        det = xr[0] * xs[1] - xs[0] * xr[1]
        inv = np.array([[xs[1], -xs[0]], [-xr[1], xr[0]]]) / det   # rows: grad r, grad s
        edges = []
        for f in range(3):
            e = v[(f + 1) % 3] - v[f]
            ln = np.hypot(*e)
            m = np.array([e[1], -e[0]]) / ln
            he = 2.0 * (2.0 * det) / ln           # 2 |T| / |e|, |T| = 2 det
            edges.append((m, 0.5 * ln, wl.c_ip * (p + 1) * (p + 2) / he))

        def points(r, s, v=v):
            loc = v[0] + 0.5 * (1 + r)[..., None] * (v[1] - v[0]) + 0.5 * (1 + s)[..., None] * (v[2] - v[0])
            return cell[(...,) + (None,) * r.ndim + (slice(None),)] + loc

        def vel(xy):
            X, Y = xy[..., 0] - wl.xc + 0.5, xy[..., 1] - wl.yc + 0.5
            return (_t(np.sin(np.pi * X) ** 2 * np.sin(2 * np.pi * Y)), _t(-np.sin(2 * np.pi * X) * np.sin(np.pi * Y) ** 2))
        geo.append(dict(det=det, gx=_t(Br * inv[0, 0] + Bs * inv[1, 0]), gy=_t(Br * inv[0, 1] + Bs * inv[1, 1]),
                        ex=_t(Ber * inv[0, 0] + Bes * inv[1, 0]), ey=_t(Ber * inv[0, 1] + Bes * inv[1, 1]),
                        edges=edges, vol=vel(points(rv, sv)), edge=vel(points(re, se))))
    B, Be, wv, Minv, gw = _t(B), _t(Be), _t(wv), _t(Minv), _t(gw)

    def rhs(w, t):
        c = math.cos(math.pi * t / wl.T)
        q = w.reshape(2, ny, nx, 2, -1)
        tr = []
        for ty in range(2):
            G, f = geo[ty], q[:, :, :, ty]
            val = torch.einsum("fkn,vyxn->vyxfk", Be, f)
            dx, dy = torch.einsum("fkn,vyxn->vyxfk", G["ex"], f), torch.einsum("fkn,vyxn->vyxfk", G["ey"], f)
            n0, n1 = _normal(dx[1], dy[1])
            tr.append([val[0], val[1], dx[0], dy[0], n0, n1, c * G["edge"][0], c * G["edge"][1]])
        out = []
        for ty in range(2):
            G, f = geo[ty], q[:, :, :, ty]
            ph = torch.einsum("qn,yxn->yxq", B, f[0])
            gp = [torch.einsum("qn,yxn->yxq", G[d], f[0]) for d in ("gx", "gy")]
            gs = [torch.einsum("qn,yxn->yxq", G[d], f[1]) for d in ("gx", "gy")]
            n0, n1 = _normal(*gs)
            sp = ph * (1 - ph)
            ax, ay = wl.Gamma * (wl.eps * gp[0] - sp * n0), wl.Gamma * (wl.eps * gp[1] - sp * n1)
            u, v = c * G["vol"][0], c * G["vol"][1]
            wq = wv * G["det"]
            Rp = torch.einsum("yxq,qn->yxn", -wq * (u * gp[0] + v * gp[1]), B)
            Rp = Rp + torch.einsum("yxq,qn->yxn", -wq * ax, G["gx"]) + torch.einsum("yxq,qn->yxn", -wq * ay, G["gy"])
            Rs = torch.einsum("yxq,qn->yxn", -wq * (u * gs[0] + v * gs[1]), B)
            for e in range(3):
                m, hl, eta = G["edges"][e]
                a = [z[:, :, e] for z in tr[ty]]
                # the neighbour across: type 0 has bottom, right, diagonal; type 1 diagonal, top, left
                roll, oe = {(0, 0): ((1, 0), 1), (0, 1): ((0, -1), 2), (0, 2): ((0, 0), 0),
                            (1, 0): ((0, 0), 2), (1, 1): ((-1, 0), 0), (1, 2): ((0, 1), 1)}[(ty, e)]
                b = [torch.roll(z[:, :, oe], roll, dims=(0, 1)).flip(-1) for z in tr[1 - ty]]
                unm, unp = a[6] * m[0] + a[7] * m[1], b[6] * m[0] + b[7] * m[1]
                lam = torch.maximum(unm.abs(), unp.abs())
                jump = b[0] - a[0]
                gn = 0.5 * ((a[2] + b[2]) * m[0] + (a[3] + b[3]) * m[1])
                sharp = 0.5 * (a[0] * (1 - a[0]) * (a[4] * m[0] + a[5] * m[1]) + b[0] * (1 - b[0]) * (b[4] * m[0] + b[5] * m[1]))
                ahat = wl.Gamma * (wl.eps * (gn + eta * jump) - sharp)
                wf = gw * hl
                Rp = Rp + torch.einsum("yxk,kn->yxn", wf * ((lam - unm) * 0.5 * jump + ahat), Be[e])
                dn = G["ex"][e] * m[0] + G["ey"][e] * m[1]
                Rp = Rp + torch.einsum("yxk,kn->yxn", -wf * 0.5 * wl.Gamma * wl.eps * jump, dn)
                Rs = Rs + torch.einsum("yxk,kn->yxn", wf * (lam - unm) * 0.5 * (b[1] - a[1]), Be[e])
            out.append(torch.stack([Rp, Rs]) @ Minv / G["det"])
        return torch.stack(out, dim=3).reshape(2, -1)
    return _rk4(rhs, _t(wl.w), wl.dt, steps)


def _reinit(wl, niter):
    g = _Grid(2, wl.nx, wl.ny, wl.p, wl.hx, wl.hy, wl.bc)
    P1 = wl.p + 1
    eta = (wl.c_ip * P1 * P1 / wl.hx, wl.c_ip * P1 * P1 / wl.hy)
    h = min(wl.hx, wl.hy)
    q = 2 * wl.p + 1
    nu = h / (2 * P1)
    dtau = min(0.5 * h / q, 0.1 * h * h / (q * q * nu))
    w = _t(wl.w).clone()
    psi0 = g.field(w[0]) - 0.5
    gm = torch.sqrt(g.dx(psi0) ** 2 + g.dy(psi0) ** 2)
    flat = gm < 1e-12
    S = torch.where(flat, torch.sign(psi0), torch.tanh(psi0 / (2 * wl.eps * torch.where(flat, torch.ones_like(gm), gm))))

    def rhs(psi):
        gx, gy = g.dx(psi), g.dy(psi)
        R = g.div(-nu * gx, -nu * gy) + S * (1 - torch.sqrt(gx * gx + gy * gy))
        for axis, side, idx, sg in g.faces():
            d = gx if axis == 0 else gy
            jump = g.across(psi, axis, idx, sg) - g.own(psi, axis, idx)
            gn = 0.5 * sg * (g.across(d, axis, idx, sg) + g.own(d, axis, idx))
            R = g.lift(R, axis, idx, sg, nu * (gn + eta[axis] * jump), -0.5 * nu * jump)
        return R
    psi = psi0
    for _ in range(niter):
        p1 = psi + dtau * rhs(psi)
        p2 = 0.75 * psi + 0.25 * (p1 + dtau * rhs(p1))
        psi = psi / 3.0 + 2.0 / 3.0 * (p2 + dtau * rhs(p2))
    w[1] = psi.reshape(-1)
    return w


def exact(case, seed):
    kind = case["kind"]
    if kind == "batch":
        out = []
        for wl in _ensemble(case, seed):
            m, w = _Model(wl), _t(wl.w)
            for _ in range(case["steps"]):
                w = m.step(w, wl.dt)
            out.append(w)
        return out
    wl = _problem(case, seed)
    if kind == "kin":
        return (_kin_tri if case["elem"] == "tri" else _kin_quad)(wl, case["steps"])
    if kind == "reinit":
        return _reinit(wl, case["niter"])
    m, w = _Model(wl), _t(wl.w)
    if kind in ("rhs", "traj"):
        w0 = torch.from_numpy(np.ascontiguousarray(wl.w))
        g = torch.Generator().manual_seed(seed)
        scale = 1.0 / w0.abs().amax(dim=1, keepdim=True).clamp_min(1e-3)
        lam = _t((torch.randn(w0.shape, generator=g, dtype=torch.float64) * scale).numpy())

        def vjp(fn, w, lam):
            w = w.detach().requires_grad_()
            out = fn(w)
            return out.detach(), torch.autograd.grad(out, w, lam)[0]
        if kind == "rhs":
            return list(vjp(m.rhs, w, lam))
        states = [w]
        for _ in range(case["steps"]):
            states.append(m.step(states[-1], wl.dt))
        for w in reversed(states[:-1]):
            lam = vjp(lambda z: m.step(z, wl.dt), w, lam)[1]
        return [states[-1], lam]
    for _ in range(case["steps"]):
        w = m.step(w, wl.dt)
    return w
