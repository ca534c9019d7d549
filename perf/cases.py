"""The calls whose time matters to a user of this library: single time steps and short runs of every
built-in system, the limiter, misfit gradients and ensembles, each through the public binding
(`paper_1905_07987_gb300.ader`).

A case is a dict of plain values; `kind` says which entry points it goes through:

  steps     Context: set_state, `steps` calls of step (or one run_graph), get_state
  gradient  Context.misfit_gradient: forward sweep, checkpoints, adjoint sweep
  ensemble  Ensemble: set_state of every run, one step call, get_state of every run

`exact` restates the scheme in plain torch float64 (tables from numpy, no code of this
repository), for the accuracy of what `run` returns.
"""
import math
import random

import numpy as np
import torch
import torch.utils.checkpoint

from paper_1905_07987_gb300 import ader

DEV = "cuda"
F64 = torch.float64
# CFL factors per order (0.9 of the scheme's one-dimensional stability limit times 2N+1)
CFL = {1: 0.9, 2: 0.765, 3: 0.648, 4: 0.558, 5: 0.495, 6: 0.441}
NVAR = {"swe": 4, "elastic": 9}


def steps_case(name, pde, n, order, **kw):
    c = dict(name=name, kind="steps", pde=pde, nx=n[0], ny=n[1], nz=n[2] if len(n) > 2 else 0, order=order,
             precision="fp64", predictor="picard", guess="constant", iters=0, limiter=0, bc="periodic",
             steps=1, graph=False)
    c.update(kw)
    return c


def listed():
    return [
        # one step of a small 2-D grid, the latency of a single call (time loops driven from Python)
        steps_case("euler2d_small_step", "euler", (27, 27), 3),
        # the same grid through a captured graph: how short runs to a final time are made
        steps_case("euler2d_small_graph", "euler", (27, 27), 3, steps=48, graph=True),
        # the benchmark's workload: 332 M unknowns, mixed precision, Runge-Kutta guess and one iteration
        steps_case("euler3d_large_mixed", "euler", (81, 81, 81), 4, precision="mixed", guess="cerk", iters=1),
        # FP64 reference arithmetic on a ragged 3-D grid, the default predictor
        steps_case("euler3d_fp64", "euler", (41, 37, 33), 4),
        # explosion between walls with the subcell limiter (shock capturing), FP64, from t = 0
        steps_case("explosion3d_limiter", "euler", (64, 64, 64), 3, limiter=1, bc="wall", steps=2),
        # seismic wave propagation, Cauchy-Kowalevski predictor, mixed precision, 1 G unknowns
        steps_case("elastic3d_large_ck_mixed", "elastic", (81, 81, 81), 5, precision="mixed", predictor="ck", bc="absorbing"),
        # the same system with the default (Picard) predictor on a ragged grid, several steps
        steps_case("elastic3d_picard_mixed", "elastic", (57, 49, 41), 5, precision="mixed", bc="absorbing", steps=2),
        # the FP64 form of the seismic step
        steps_case("elastic3d_ck_fp64", "elastic", (40, 40, 40), 5, predictor="ck", bc="absorbing"),
        # shallow water over bathymetry, 67 M unknowns
        steps_case("swe2d_large", "swe", (1024, 1024), 3),
        # gradient of the receiver misfit (inversion), Cauchy-Kowalevski predictor, mixed precision
        dict(name="gradient_ck_mixed", kind="gradient", pde="elastic", nx=40, ny=40, nz=40, order=4,
             precision="mixed", predictor="ck", steps=4, k_ckpt=2),
        # the same for the default predictor in FP64 on a smaller, ragged grid
        dict(name="gradient_picard", kind="gradient", pde="elastic", nx=19, ny=16, nz=13, order=3,
             precision="fp64", predictor="picard", steps=4, k_ckpt=2),
        # ensemble of uneven grids, default predictor, mixed precision, advanced together
        dict(name="ensemble_mixed", kind="ensemble", pde="elastic", sides="64,48,32,24,24,24,40,24", order=4,
             precision="mixed", predictor="picard", steps=2),
    ]


def _log_int(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def draw(rng):
    kind = rng.choice(["euler2d", "euler3d_mixed", "euler3d_fp64", "explosion", "elastic", "elastic", "swe",
                       "gradient", "ensemble"])
    if kind == "euler2d":
        order = rng.randint(1, 5)
        side = _log_int(rng, 9, 240)
        c = steps_case("", "euler", (side, max(3, side - rng.randint(0, 7))), order, steps=2 * rng.randint(1, 12),
                       graph=rng.random() < 0.5, bc=rng.choice(["periodic", "wall", "absorbing"]))
    elif kind in ("euler3d_mixed", "euler3d_fp64"):
        mixed = kind == "euler3d_mixed"
        side = _log_int(rng, 8, 64 if mixed else 36)
        cerk = rng.random() < 0.5
        c = steps_case("", "euler", (side, max(3, side - rng.randint(0, 5)), max(3, side - rng.randint(0, 5))),
                       rng.randint(2, 5 if mixed else 4), precision="mixed" if mixed else "fp64",
                       guess="cerk" if cerk else "constant", iters=1 if cerk else 0,
                       bc=rng.choice(["periodic", "wall", "absorbing"]))
    elif kind == "explosion":
        side = _log_int(rng, 12, 48)
        c = steps_case("", "euler", (side, side + rng.randint(0, 3), side), rng.randint(2, 3), limiter=1, bc="wall",
                       steps=rng.randint(1, 3), precision=rng.choice(["fp64", "mixed"]))
    elif kind == "elastic":
        side = _log_int(rng, 8, 48)
        form = rng.choice(["picard/fp64", "picard/mixed", "ck/fp64", "ck/mixed", "ck/tf32x3"])
        predictor, precision = form.split("/")
        order = rng.choice([1, 3, 5]) if precision == "tf32x3" else rng.randint(1, 5)
        if form == "picard/fp64":
            side = min(side, 28)
        c = steps_case("", "elastic", (side, max(3, side - rng.randint(0, 5)), max(3, side - rng.randint(0, 5))), order,
                       precision=precision, predictor=predictor, bc=rng.choice(["absorbing", "periodic"]),
                       guess="cerk" if predictor == "picard" and rng.random() < 0.2 else "constant", steps=rng.randint(1, 3))
    elif kind == "swe":
        side = _log_int(rng, 24, 640)
        c = steps_case("", "swe", (side, max(3, side - rng.randint(0, 9))), rng.randint(1, 5), steps=rng.randint(1, 3),
                       bc=rng.choice(["periodic", "wall", "absorbing"]))
    elif kind == "gradient":
        predictor = rng.choice(["picard", "ck"])
        side = _log_int(rng, 6, 14 if predictor == "picard" else 28)
        c = dict(kind="gradient", pde="elastic", nx=side, ny=max(3, side - rng.randint(0, 3)),
                 nz=max(3, side - rng.randint(0, 3)), order=rng.randint(2, 4), precision=rng.choice(["fp64", "mixed"]),
                 predictor=predictor, steps=rng.randint(2, 5), k_ckpt=rng.randint(1, 3))
    else:
        runs = rng.randint(2, 7)
        c = dict(kind="ensemble", pde="elastic", sides=",".join(str(_log_int(rng, 8, 40)) for _ in range(runs)),
                 order=rng.randint(2, 4), precision=rng.choice(["fp64", "mixed"]), predictor=rng.choice(["picard", "ck"]),
                 steps=2 * rng.randint(1, 2))
        if c["precision"] == "fp64" and c["predictor"] == "picard":
            c["sides"] = ",".join(str(min(int(s), 20)) for s in c["sides"].split(","))
    c.pop("name", None)
    return c


# ---- inputs ---------------------------------------------------------------------------------------

def grid_of(case):
    """(cells per direction, lower corner, upper corner) of a steps or gradient case."""
    n = [case["nx"], case["ny"]] + ([case["nz"]] if case.get("nz") else [])
    if case["pde"] == "elastic":  # cells of 0.5 km
        return n, [0.0] * 3, [0.5 * k for k in n]
    if case.get("limiter"):
        return n, [-1.0] * len(n), [1.0] * len(n)
    return n, [0.0] * len(n), [k / max(n) for k in n]


def gauss(n):
    x, w = np.polynomial.legendre.leggauss(n)
    return 0.5 * (x + 1.0), 0.5 * w


def points(ncell, lo, hi, x):
    """Coordinates of the points x (per cell and direction, in [0,1]): one broadcastable tensor per
    direction over [cells (z, y, x)..., points (z, y, x)...]."""
    D, m = len(ncell), len(x)
    out = []
    for d in range(D):
        h = (hi[d] - lo[d]) / ncell[d]
        i = torch.arange(ncell[d], dtype=F64, device=DEV).view([ncell[d] if a == D - 1 - d else 1 for a in range(D)] + [1] * D)
        p = torch.as_tensor(x, dtype=F64, device=DEV).view([1] * D + [m if a == D - 1 - d else 1 for a in range(D)])
        out.append(lo[d] + h * (i + p))
    return out


def smooth(rng, X, lo, hi, modes=3):
    """A seeded smooth periodic field with values in [-1, 1]: a few plane waves."""
    f = 0.0
    for _ in range(modes):
        phase = 2 * math.pi * rng.random()
        for d, x in enumerate(X):
            k = rng.choice([-2, -1, 1, 2])
            phase = phase + 2 * math.pi * k * (x - lo[d]) / (hi[d] - lo[d])
        f = f + torch.sin(phase) / modes
    return f


def euler_state(rho, vel, p, gamma=1.4):
    E = p / (gamma - 1.0)
    for v in vel:
        E = E + 0.5 * rho * v * v
    return torch.stack(torch.broadcast_tensors(rho, *[rho * v for v in vel], E), dim=-1).contiguous()


def initial_state(case, seed):
    """(state [cells..., nodes..., nvar], material [cells..., 3] or None) of a case."""
    rng = random.Random(1000003 * seed + 17)
    ncell, lo, hi = grid_of(case)
    X = points(ncell, lo, hi, gauss(case["order"] + 1)[0])
    if case["pde"] == "euler" and case.get("limiter"):
        return euler_state(*ball(rng, X)), None
    if case["pde"] == "euler":
        f = [smooth(rng, X, lo, hi) for _ in range(len(X) + 2)]
        return euler_state(1.0 + 0.2 * f[0], [1.0 - 0.3 * d + 0.1 * f[1 + d] for d in range(len(X))], 1.0 + 0.1 * f[-1]), None
    if case["pde"] == "swe":
        b = 0.1 + 0.05 * smooth(rng, X, lo, hi)
        h = 1.0 - b + 0.02 * smooth(rng, X, lo, hi)
        hu = 0.3 * h * (1 + 0.1 * smooth(rng, X, lo, hi))
        hv = -0.2 * h * (1 + 0.1 * smooth(rng, X, lo, hi))
        return torch.stack(torch.broadcast_tensors(h, hu, hv, b), dim=-1).contiguous(), None
    # elastic: a smooth wavefield (stresses of the size rho vp v) and smooth per-cell material
    v = [1e-3 * smooth(rng, X, lo, hi) for _ in range(3)]
    s = [1e-3 * 15.0 * smooth(rng, X, lo, hi) for _ in range(6)]
    C = [c.reshape(c.shape[:3]) for c in points(ncell, lo, hi, [0.5])]
    rho = 2.75 + 0.25 * smooth(rng, C, lo, hi)
    vp = 6.0 + smooth(rng, C, lo, hi)
    mu = rho * vp * vp / 3.0
    mat = torch.stack(torch.broadcast_tensors(rho, rho * vp * vp - 2 * mu, mu), dim=-1).contiguous()
    return torch.stack(torch.broadcast_tensors(*v, *s), dim=-1).contiguous(), mat


def ball(rng, X):
    """Explosion: (rho, velocities, p) of a ball of hot gas, its centre and radius seeded."""
    r0 = 0.45 + 0.1 * rng.random()
    r2 = 0.0
    for x in X:
        c = 0.1 * (rng.random() - 0.5)
        r2 = r2 + (x - c) ** 2
    ins = r2 < r0 * r0
    rho = torch.where(ins, 1.0, 0.125).to(F64)
    return rho, [0.0 * rho] * len(X), torch.where(ins, 1.0, 0.1).to(F64)


def subcells(case, seed):
    """Subcell samples of the explosion and the cells (bytes) that the jump cuts."""
    rng = random.Random(1000003 * seed + 17)
    ncell, lo, hi = grid_of(case)
    D, ns = len(ncell), 2 * case["order"] + 1
    U = euler_state(*ball(rng, points(ncell, lo, hi, (np.arange(ns) + 0.5) / ns)))
    rho = U[..., 0].reshape(ncell[::-1] + [-1])
    return U, (rho.amax(-1) > rho.amin(-1)).to(torch.uint8).reshape(-1).contiguous()


def source_of(case, ncell, hi):
    """The point source of the elastic cases: (x0, moment tensor, f0, t0)."""
    return [0.37 * hi[0], 0.52 * hi[1], 0.61 * hi[2]], [3e-4, -2e-4, 5e-4, 1e-3, 4e-4, -6e-4], 2.0, 0.05


def receiver_points(hi):
    return np.array([[(i + 0.5) * hi[0] / 4, (j + 0.5) * hi[1] / 4, hi[2]] for j in range(4) for i in range(4)])


def elastic_dt(case):
    """A fixed step for the gradient and ensemble cases: Eq. (7) at the fastest wave (vp <= 7 km/s)."""
    return CFL[case["order"]] / (3 * (2 * case["order"] + 1)) * 0.5 / 7.0


def config_of(case, **kw):
    ncell, lo, hi = grid_of(case)
    return ader.make_config(case["pde"], len(ncell), case["order"], ncell, lo, hi, case.get("bc", "absorbing"),
                            CFL[case["order"]], picard_iters=case.get("iters", 0), limiter=case.get("limiter", 0),
                            precision=case["precision"], predictor=case["predictor"],
                            initial_guess=case.get("guess", "constant"), **kw)


def members(case):
    """The single-run cases of an ensemble case."""
    return [dict(case, kind="steps", nx=int(s), ny=int(s), nz=int(s)) for s in case["sides"].split(",")]


def prepare(case, seed):
    s = {"case": case}
    if case["kind"] == "ensemble":
        s["ens"] = ader.Ensemble([config_of(m) for m in members(case)])
        s["u0"] = []
        for i, (m, ctx) in enumerate(zip(members(case), s["ens"].runs)):
            ncell, lo, hi = grid_of(m)
            u, mat = initial_state(m, 100 * seed + i)
            ctx.set_material(mat.view(-1))
            ctx.set_point_source(*source_of(m, ncell, hi))
            s["u0"].append(u.view(-1))
        s["out"] = [torch.empty_like(u) for u in s["u0"]]
        return s
    ncell, lo, hi = grid_of(case)
    u, mat = initial_state(case, seed)
    s["u0"] = u.view(-1)
    s["ctx"] = ctx = ader.Context(config_of(case))
    if mat is not None:
        s["mat"] = mat.view(-1)
        ctx.set_material(s["mat"])
        ctx.set_point_source(*source_of(case, ncell, hi))
    if case["kind"] == "gradient":
        pts = receiver_points(hi)
        s["seismo"] = torch.zeros(case["steps"], len(pts), 3, dtype=F64, device=DEV)
        ctx.set_receivers(pts, s["seismo"], case["steps"])
        g = torch.Generator(device=DEV).manual_seed(seed)
        s["obs"] = 1e-3 * torch.randn(case["steps"], len(pts), 3, dtype=F64, device=DEV, generator=g)
        s["grad_mat"] = torch.zeros(ctx.cells * 3, dtype=F64, device=DEV)
        s["grad_M"] = torch.zeros(6, dtype=F64, device=DEV)
    else:
        s["out"] = torch.empty_like(s["u0"])
    if case.get("limiter"):
        s["sub"], s["flags"] = subcells(case, seed)
    return s


def run(state):
    case = state["case"]
    if case["kind"] == "ensemble":
        ens = state["ens"]
        for ctx, u in zip(ens.runs, state["u0"]):
            ctx.set_time(0.0)
            ctx.set_state(u)
        ens.step(case["steps"], dt=elastic_dt(case))
        for ctx, out in zip(ens.runs, state["out"]):
            ctx.get_state(out)
        return state["out"]
    ctx = state["ctx"]
    if case["kind"] == "gradient":
        J = ctx.misfit_gradient(state["u0"], 0.0, elastic_dt(case), case["steps"], case["k_ckpt"], state["obs"],
                                state["grad_mat"], state["grad_M"])
        return {"J": J, "grad_mat": state["grad_mat"], "grad_M": state["grad_M"]}
    ctx.set_time(0.0)
    ctx.set_state(state["u0"])
    if case["limiter"]:
        ctx.set_subcell_state(state["sub"], state["flags"])
    if case["graph"]:
        ctx.run_graph(2, case["steps"] // 2)
    else:
        for _ in range(case["steps"]):
            ctx.step()
    return ctx.get_state(state["out"])


# ---- what a pass cannot do without -----------------------------------------------------------------

def cell_flops(case, D):
    """Operations of one step per cell: nodal flux evaluations, derivative products by sum
    factorisation, time solve, face terms."""
    n = case["order"] + 1
    pde = case["pde"]
    nv = NVAR.get(pde, D + 2)
    ns = n ** D
    faces = 2 * D * ns * nv * 2 + 2 * D * n ** (D - 1) * nv * 6
    if pde == "elastic":  # linear: order + 1 applications of the spatial operator, whatever the predictor
        return (n + 1) * ns * (18 * 2 * n + 48) + faces
    flux = 12 * D + 10
    iters = case.get("iters") or n
    point = flux + D * nv * 2 * n
    guess = 4 * ns * point if case.get("guess") == "cerk" else ns * point
    its = iters if case.get("guess") == "cerk" else iters - 1
    total = guess + its * ns * n * (point + 2 * n * nv) + ns * n * flux + D * ns * nv * 2 * n + faces
    if case.get("limiter"):
        total += 2 * nv * D * (2 * n - 1) ** D * n  # subcell averages of the candidate
    return total


def work(case):
    if case["kind"] == "ensemble":
        w = [work(dict(m, limiter=0, graph=False)) for m in members(case)]
        return {"bytes": sum(x["bytes"] for x in w), "flops": sum(x["flops"] for x in w)}
    ncell = grid_of(case)[0]
    D, cells = len(ncell), math.prod(grid_of(case)[0])
    dofs = cells * (case["order"] + 1) ** D * NVAR.get(case["pde"], D + 2)
    f = cells * cell_flops(case, D)
    if case["kind"] == "gradient":  # per step: forward, and the adjoint with its recomputation
        return {"bytes": 16 * dofs + 48 * cells, "flops": case["steps"] * 3 * f}
    return {"bytes": 16 * dofs + (24 * cells if case["pde"] == "elastic" else 0), "flops": case["steps"] * f}


# ---- the scheme in plain float64 -------------------------------------------------------------------

def _t(a):
    return torch.as_tensor(np.asarray(a), dtype=F64, device=DEV)


def lagrange(nodes, xi):
    """phi_m(xi) for every node m, [len(xi), n]."""
    n = len(nodes)
    out = np.ones((len(xi), n))
    for m in range(n):
        for k in range(n):
            if k != m:
                out[:, m] *= (np.asarray(xi) - nodes[k]) / (nodes[m] - nodes[k])
    return out


def lagrange_dx(nodes):
    n = len(nodes)
    D = np.zeros((n, n))
    for m in range(n):
        for l in range(n):
            if l != m:
                t = np.full(n, 1.0 / (nodes[m] - nodes[l]))
                for k in range(n):
                    if k not in (m, l):
                        t *= (nodes - nodes[k]) / (nodes[m] - nodes[k])
                D[:, m] += t
    return D


def along(M, a, axis):
    """sum_m M[i, m] a[..., m, ...] along an axis."""
    return torch.tensordot(a, M, dims=([axis], [1])).movedim(-1, axis)


def ends(e, a, axis):
    return torch.tensordot(a, e, dims=([axis], [0]))


def cut(a, axis, k0, k1):
    return a.narrow(axis, k0, k1 - k0)


class Scheme:
    """One step of a steps / gradient / ensemble-member case on arrays [cells..., nodes..., nvar]."""

    def __init__(self, case, mat=None, M=None):
        self.case, self.pde, self.mat = case, case["pde"], mat
        self.nc, self.lo, self.hi = grid_of(case)
        self.D, self.n = len(self.nc), case["order"] + 1
        self.h = [(b - a) / k for a, b, k in zip(self.lo, self.hi, self.nc)]
        self.bc = case.get("bc", "absorbing")
        x, w = gauss(self.n)
        Dm = lagrange_dx(x)
        e0, e1 = lagrange(x, [0.0])[0], lagrange(x, [1.0])[0]
        K1 = np.outer(e1, e1) - (np.diag(w) @ Dm).T
        self.xn, self.x, self.w, self.Dm = x, _t(x), _t(w), _t(Dm)
        self.e0, self.e1, self.Kw = _t(e0), _t(e1), _t(np.linalg.solve(K1, np.diag(w)))
        self.Vinv = _t(np.linalg.inv(np.vander(x, increasing=True)))
        z, wz = gauss(3)
        self.path = list(zip(z.tolist(), wz.tolist()))
        self.ns = ns = 2 * case["order"] + 1
        s, sw = gauss(self.n)
        P1 = np.stack([sw @ lagrange(x, (k + s) / ns) for k in range(ns)])
        self.P1 = _t(P1)
        # least squares that keeps the cell mean
        A = np.block([[2 * P1.T @ P1, w[:, None]], [w[None, :], np.zeros((1, 1))]])
        B = np.vstack([2 * P1.T, np.full((1, ns), 1.0 / ns)])
        self.R1 = _t(np.linalg.solve(A, B)[:-1])
        self.src = None
        if self.pde == "elastic":
            x0, M0, self.f0, self.t0 = source_of(case, self.nc, self.hi)
            self.M = _t(M0) if M is None else M
            cell, xi = self.locate(x0)
            g = self.basis(xi)
            for a in range(3):
                g = g / self.w.view([self.n if b == a else 1 for b in range(3)])
            self.src = (cell, g / math.prod(self.h))

    def locate(self, p):
        cell, xi = [], []
        for d in range(self.D):
            s = (p[d] - self.lo[d]) / self.h[d]
            k = min(max(int(math.floor(s)), 0), self.nc[d] - 1)
            cell.append(k)
            xi.append(s - k)
        return tuple(cell[::-1]), xi

    def basis(self, xi):
        g = _t(lagrange(self.xn, [xi[2]])[0])[:, None, None]
        return g * _t(lagrange(self.xn, [xi[1]])[0])[None, :, None] * _t(lagrange(self.xn, [xi[0]])[0])[None, None, :]

    def ricker(self, t):
        a = (math.pi * self.f0 * (torch.as_tensor(t, dtype=F64, device=DEV) - self.t0)) ** 2
        return (1.0 - 2.0 * a) * torch.exp(-a)

    def with_source(self, a, z0, amp):
        """a + source with amplitude amp, where a covers the cell layers from z0."""
        if self.src is None:
            return a
        (k, j, i), g = self.src
        if not z0 <= k < z0 + a.shape[0]:
            return a
        S = torch.zeros_like(a)
        S[k - z0, j, i, ..., 3:] = -amp * g[..., None] * self.M
        return a + S

    # fluxes and products -------------------------------------------------------------------------
    def flux(self, q, d):
        if self.pde == "euler":
            v = q[..., 1 + d] / q[..., 0]
            p = self.pressure(q)
            f = [q[..., 1 + i] * v + (p if i == d else 0.0) for i in range(self.D)]
            return torch.stack([q[..., 1 + d]] + f + [(q[..., -1] + p) * v], dim=-1)
        u = q[..., 1 + d] / q[..., 0]
        return torch.stack([q[..., 1 + d], q[..., 1] * u, q[..., 2] * u, torch.zeros_like(u)], dim=-1)

    def pressure(self, q):
        return 0.4 * (q[..., -1] - 0.5 * (q[..., 1:-1] ** 2).sum(-1) / q[..., 0])

    def speed(self, q, d):
        if self.pde == "euler":
            return (q[..., 1 + d] / q[..., 0]).abs() + torch.sqrt((1.4 * self.pressure(q) / q[..., 0]).clamp(min=0))
        return (q[..., 1 + d] / q[..., 0]).abs() + torch.sqrt(9.81 * q[..., 0])

    def mirror(self, q, d):
        return torch.cat([q[..., :1 + d], -q[..., 1 + d:2 + d], q[..., 2 + d:]], dim=-1)

    def elastic_rows(self, dq, ir, lam, mu):
        """rows of -sum_d B_d dq[d] (dq[d] = None: direction left out)."""
        sig = [[3, 6, 7], [6, 4, 8], [7, 8, 5]]
        R = [0.0] * 9
        for d in range(3):
            if dq[d] is None:
                continue
            for i in range(3):
                R[i] = R[i] + ir * dq[d][..., sig[i][d]]
                R[3 + i] = R[3 + i] + (lam + (2.0 * mu if i == d else 0.0)) * dq[d][..., d]
                if i != d:
                    R[sig[i][d]] = R[sig[i][d]] + mu * dq[d][..., i]
        like = ir * dq[[d for d in range(3) if dq[d] is not None][0]][..., 0]
        return torch.stack([r if torch.is_tensor(r) else torch.zeros_like(like) for r in R], dim=-1)

    def operator(self, q, lead, mat):
        """Right-hand side without sources; the node axes start at `lead`."""
        out = 0.0
        dq = []
        for d in range(self.D):
            ax = lead + self.D - 1 - d
            if self.pde == "elastic":
                dq.append(along(self.Dm, q, ax) / self.h[d])
                continue
            out = out - along(self.Dm, self.flux(q, d), ax) / self.h[d]
            if self.pde == "swe":
                g = 9.81 * q[..., 0] * along(self.Dm, q[..., 0] + q[..., 3], ax) / self.h[d]
                z = torch.zeros_like(g)
                out = out - torch.stack([z, g if d == 0 else z, g if d == 1 else z, z], dim=-1)
        if self.pde == "elastic":
            m = mat.reshape([1] * (lead - 3) + list(mat.shape[:3]) + [1, 1, 1, 3])
            out = self.elastic_rows(dq, 1.0 / m[..., 0], m[..., 1], m[..., 2])
        return out

    # predictor ------------------------------------------------------------------------------------
    def predict(self, u, dt, t, z0, mat):
        """(volume change, per direction (q+, q-, F+, F-)) of the cell layers u from z0."""
        D, n = self.D, self.n
        tn = t + self.x * dt
        wt = self.w.view([n] + [1] * (2 * D + 1))
        if self.case["predictor"] == "ck":
            amp = self.Vinv @ self.ricker(tn)
            a, qbar = u, u
            for k in range(n - 1):
                a = dt / (k + 1) * self.with_source(self.operator(a, D, mat), z0, amp[k])
                qbar = qbar + a / (k + 2)
            vol = self.with_source(self.operator(qbar, D, mat), z0, (self.w * self.ricker(tn)).sum())
            q = None
        else:
            def rhs(q):
                R = self.operator(q, 1 + D, mat)
                if self.src is None:
                    return R
                return torch.stack([self.with_source(R[k], z0, self.ricker(tn[k])) for k in range(n)])
            if self.case.get("guess") == "cerk":
                def R1(q, tt):
                    return self.with_source(self.operator(q, D, mat), z0, self.ricker(tt) if self.src else 0.0)
                k1 = R1(u, t)
                k2 = R1(u + 0.5 * dt * k1, t + 0.5 * dt)
                k3 = R1(u + 0.5 * dt * k2, t + 0.5 * dt)
                k4 = R1(u + dt * k3, t + dt)
                th = self.x.view(wt.shape)
                q = u + dt * ((th - 1.5 * th ** 2 + 2 * th ** 3 / 3) * k1 + (th ** 2 - 2 * th ** 3 / 3) * (k2 + k3)
                              + (-0.5 * th ** 2 + 2 * th ** 3 / 3) * k4)
                del k1, k2, k3, k4
            else:
                q = u.unsqueeze(0).expand([n] + list(u.shape))
            for _ in range(self.case.get("iters") or n):
                q = u + dt * along(self.Kw, rhs(q), 0)
            qbar = (wt * q).sum(0)
            vol = (wt * rhs(q)).sum(0)
        faces = []
        for d in range(D):
            ax = 2 * D - 1 - d
            qp, qm = ends(self.e1, qbar, ax), ends(self.e0, qbar, ax)
            if self.pde == "elastic":
                faces.append((qp, qm, None, None))
                continue
            F = sum(self.w[k] * self.flux(q[k], d) for k in range(n))
            faces.append((qp, qm, ends(self.e1, F, ax), ends(self.e0, F, ax)))
        return dt * vol, faces

    # faces ----------------------------------------------------------------------------------------
    def riemann(self, d, qL, qR, FL, FR, mL, mR):
        D = self.D
        dq = qR - qL
        if self.pde == "elastic":
            shape = lambda m: m.reshape(list(m.shape[:3]) + [1, 1])  # noqa: E731
            sL, sR = (torch.sqrt((m[..., 1] + 2 * m[..., 2]) / m[..., 0]) for m in (mL, mR))
            G = -0.5 * shape(torch.where(sL >= sR, sL, sR))[..., None] * dq
            half = 0.0
            for z, wz in self.path:
                m = mL + z * (mR - mL)
                rows = [None] * 3
                rows[d] = dq
                half = half - 0.5 * wz * self.elastic_rows(rows, shape(1.0 / m[..., 0]), shape(m[..., 1]), shape(m[..., 2]))
            return G + half, G - half
        s = torch.maximum(self.speed(qL, d), self.speed(qR, d))
        s = s.flatten(D).amax(-1).reshape(list(s.shape[:D]) + [1] * D)
        G = 0.5 * (FL + FR) - 0.5 * s * dq
        if self.pde == "euler":
            return G, G
        half = 0.5 * 9.81 * (qL[..., 0] + 0.5 * dq[..., 0]) * (dq[..., 0] + dq[..., 3])
        z = torch.zeros_like(half)
        half = torch.stack([z, half if d == 0 else z, half if d == 1 else z, z], dim=-1)
        return G + half, G - half

    def ghost(self, d, q, F):
        if self.pde == "elastic":
            return torch.zeros_like(q), None
        if self.bc == "wall":
            return self.mirror(q, d), -self.mirror(F, d)
        return q, F

    def face_fluxes(self, faces):
        """Per direction: Phi_L on every cell's upper face, Phi_R on its lower face."""
        out = []
        for d in range(self.D):
            qp, qm, Fp, Fm = faces[d]
            ax, N = self.D - 1 - d, self.nc[d]
            first, last = (lambda a: cut(a, ax, 0, 1)), (lambda a: cut(a, ax, N - 1, N))
            nxt = lambda a, end: torch.cat([cut(a, ax, 1, N), end], dim=ax)  # noqa: E731
            m = self.mat
            if self.bc == "periodic":
                eq, eF, em = first(qm), None if Fm is None else first(Fm), None if m is None else first(m)
            else:
                eq, eF = self.ghost(d, last(qp), None if Fp is None else last(Fp))
                em = None if m is None else last(m)
            L, R = self.riemann(d, qp, nxt(qm, eq), Fp, None if Fm is None else nxt(Fm, eF), m, None if m is None else nxt(m, em))
            if self.bc == "periodic":
                R0 = last(R)
            else:
                gq, gF = self.ghost(d, first(qm), None if Fm is None else first(Fm))
                fm = None if m is None else first(m)
                R0 = self.riemann(d, gq, first(qm), gF, None if Fm is None else first(Fm), fm, fm)[1]
            out.append((L, torch.cat([R0, cut(R, ax, 0, N - 1)], dim=ax)))
        return out

    def cfl(self, u):
        if self.pde == "elastic":
            lam = float(torch.sqrt((self.mat[..., 1] + 2 * self.mat[..., 2]) / self.mat[..., 0]).max())
        else:
            lam = max(float(self.speed(u, d).max()) for d in range(self.D))
        return CFL[self.n - 1] / (self.D * (2 * self.n - 1)) * min(self.h) / lam

    def step(self, u, dt, t, rep=None):
        D = self.D
        layer = u[0].numel() * self.n
        zs = max(1, int(6e7 // layer))
        parts = []
        for z0 in range(0, u.shape[0], zs):
            parts.append(self.predict(u[z0:z0 + zs], dt, t, z0, None if self.mat is None else self.mat[z0:z0 + zs]))
        new = u + torch.cat([p[0] for p in parts])
        faces = [tuple(None if parts[0][1][d][k] is None else torch.cat([p[1][d][k] for p in parts]) for k in range(4)) for d in range(D)]
        del parts
        flux = self.face_fluxes(faces)
        for d in range(D):
            ax = 2 * D - 1 - d
            shape = [self.n if a == ax else 1 for a in range(2 * D + 1)]
            L, R = flux[d]
            if faces[d][2] is not None:
                L, R = L - faces[d][2], R - faces[d][3]
            new = new - dt / self.h[d] * ((self.e1 / self.w).view(shape) * L.unsqueeze(ax) - (self.e0 / self.w).view(shape) * R.unsqueeze(ax))
        if rep is None:
            return new
        return self.limit(new, rep, dt, flux)

    # limiter (3-D, walls) ---------------------------------------------------------------------------
    def project(self, u, M):
        for a in range(self.D):
            u = along(M, u, self.D + a)
        return u

    def shifted(self, a, d, side, fill):
        """a of the neighbour cell across `side` (+1 / -1) of direction d, `fill` outside the domain."""
        ax, N = self.D - 1 - d, self.nc[d]
        f = torch.full_like(cut(a, ax, 0, 1), fill)
        return torch.cat([cut(a, ax, 1, N), f], dim=ax) if side > 0 else torch.cat([f, cut(a, ax, 0, N - 1)], dim=ax)

    def admissible(self, q):
        ok = (q[..., 0] > 0) & (self.pressure(q) > 0) & torch.isfinite(q).all(-1)
        return ok.flatten(self.D).all(-1)

    def fv(self, rep, dt):
        """One MUSCL-Hancock step of every subcell: (averages, per direction the subface fluxes)."""
        D, ns, nv = self.D, self.ns, rep.shape[-1]
        nc = self.nc[::-1]
        G = rep.permute([k + o for k in range(D) for o in (0, D)] + [2 * D]).reshape([c * ns for c in nc] + [nv])
        for d in range(D):
            ax, N = D - 1 - d, G.shape[D - 1 - d]
            G = torch.cat([self.mirror(cut(G, ax, 0, 2).flip(ax), d), G, self.mirror(cut(G, ax, N - 2, N).flip(ax), d)], dim=ax)
        U = G[(slice(1, -1),) * D]
        sig, inc = [], 0.0
        for d in range(D):
            ax = D - 1 - d
            inner = [slice(1, -1)] * D
            inner[ax] = slice(None)
            S = G[tuple(inner)]
            N = S.shape[ax]
            a, b = cut(S, ax, 1, N - 1) - cut(S, ax, 0, N - 2), cut(S, ax, 2, N) - cut(S, ax, 1, N - 1)
            sig.append(torch.where(a * b > 0, torch.sign(a) * torch.minimum(a.abs(), b.abs()), 0.0))
            inc = inc - dt * ns / (2 * self.h[d]) * (self.flux(U + 0.5 * sig[d], d) - self.flux(U - 0.5 * sig[d], d))
            del S, a, b
        new, subface = U[(slice(1, -1),) * D], []
        for d in range(D):
            ax = D - 1 - d
            inner = [slice(1, -1)] * D
            inner[ax] = slice(None)
            Ui, si, ii = U[tuple(inner)], sig[d][tuple(inner)], inc[tuple(inner)]
            N = Ui.shape[ax]
            L, R = cut(Ui + 0.5 * si + ii, ax, 0, N - 1), cut(Ui - 0.5 * si + ii, ax, 1, N)
            s = torch.maximum(self.speed(L, d), self.speed(R, d))[..., None]
            f = 0.5 * (self.flux(L, d) + self.flux(R, d)) - 0.5 * s * (R - L)
            new = new + dt * ns / self.h[d] * (cut(f, ax, 0, N - 2) - cut(f, ax, 1, N - 1))
            subface.append(f)
        back = [k for c in nc for k in (c, ns)]
        return new.reshape(back + [nv]).permute([2 * k for k in range(D)] + [2 * k + 1 for k in range(D)] + [2 * D]), subface

    def limit(self, star, rep, dt, flux):
        D = self.D
        cand = self.project(star, self.P1)
        flat = rep.flatten(D, 2 * D - 1)
        mn, mx = flat.amin(D), flat.amax(D)
        lo, hi = mn, mx
        for d in range(D):
            for side in (-1, 1):
                lo = torch.minimum(lo, self.shifted(mn, d, side, math.inf))
                hi = torch.maximum(hi, self.shifted(mx, d, side, -math.inf))
        delta = torch.clamp(1e-3 * (hi - lo), min=1e-4)
        c = cand.flatten(D, 2 * D - 1)
        ok = ((c >= (lo - delta).unsqueeze(D)) & (c <= (hi + delta).unsqueeze(D))).flatten(D).all(-1)
        bad = ~(ok & self.admissible(star) & self.admissible(cand))
        U, subface = self.fv(rep, dt)
        pick = lambda m, a, b: torch.where(m.reshape(list(m.shape) + [1] * (D + 1)), a, b)  # noqa: E731
        new = star
        fixed = torch.zeros_like(bad)
        for d in range(D):
            ax, nax = D - 1 - d, 2 * D - 1 - d
            ns, N = self.ns, self.nc[d]
            # the subface fluxes on the cells' faces, tested against the nodal basis
            f = subface[d].index_select(ax, torch.arange(0, N * ns + 1, ns, device=DEV))
            split = []
            for a, k in enumerate(self.nc[::-1]):
                split += [N + 1, 1] if a == ax else [k, ns]
            f = f.reshape(split + [f.shape[-1]]).permute([2 * k for k in range(D)] + [2 * k + 1 for k in range(D)] + [2 * D])
            for a in range(D):
                if a != ax:
                    f = along((self.P1 / (self.ns * self.w)).T.contiguous(), f, D + a)
            shape = [self.n if a == nax else 1 for a in range(2 * D + 1)]
            for side in (1, -1):
                m = ~bad & self.shifted(bad, d, side, False)
                fixed = fixed | m
                if side > 0:
                    corr = -dt / self.h[d] * (self.e1 / self.w).view(shape) * (cut(f, ax, 1, N + 1) - flux[d][0].unsqueeze(nax))
                else:
                    corr = dt / self.h[d] * (self.e0 / self.w).view(shape) * (cut(f, ax, 0, N) - flux[d][1].unsqueeze(nax))
                new = pick(m, new + corr, new)
        rep = pick(bad, U, pick(fixed, self.project(new, self.P1), cand))
        return pick(bad, self.project(U, self.R1), new), rep


def exact_steps(case, seed):
    u, mat = initial_state(case, seed)
    S = Scheme(case, mat)
    rep, t = None, 0.0
    if case.get("limiter"):
        sub, flags = subcells(case, seed)
        cut_cells = flags.bool().reshape(S.nc[::-1] + [1] * (S.D + 1))
        rep = torch.where(cut_cells, sub, S.project(u, S.P1))
        u = torch.where(cut_cells, S.project(sub, S.R1), u)
        del sub
    for _ in range(case["steps"]):
        dt = elastic_dt(case) if case["kind"] == "ensemble" else S.cfl(u)
        if rep is None:
            u = S.step(u, dt, t)
        else:
            u, rep = S.step(u, dt, t, rep)
        t += dt
    return u.reshape(-1)


def exact_gradient(case, seed):
    u, mat = initial_state(case, seed)
    mat.requires_grad_(True)
    M = _t(source_of(case, *grid_of(case)[::2])[1]).requires_grad_(True)
    dt = elastic_dt(case)
    pts = receiver_points(grid_of(case)[2])
    g = torch.Generator(device=DEV).manual_seed(seed)
    obs = 1e-3 * torch.randn(case["steps"], len(pts), 3, dtype=F64, device=DEV, generator=g)

    def one(u, mat, M, t):
        return Scheme(case, mat, M).step(u, dt, t)
    S = Scheme(case)
    where = [S.locate(p) for p in pts]
    J, u = 0.0, u.requires_grad_(True)
    for k in range(case["steps"]):
        u = torch.utils.checkpoint.checkpoint(one, u, mat, M, k * dt, use_reentrant=False)
        v = torch.stack([(u[cell][..., :3] * S.basis(xi)[..., None]).sum((0, 1, 2)) for cell, xi in where])
        J = J + 0.5 * dt * ((v - obs[k]) ** 2).sum()
    gm, gM = torch.autograd.grad(J, [mat, M])
    return {"J": float(J.detach()), "grad_mat": gm.reshape(-1), "grad_M": gM}


def exact(case, seed):
    if case["kind"] == "gradient":
        return exact_gradient(case, seed)
    with torch.no_grad():
        if case["kind"] == "ensemble":
            return [exact_steps(dict(m, kind="ensemble"), 100 * seed + i) for i, m in enumerate(members(case))]
        return exact_steps(case, seed)
