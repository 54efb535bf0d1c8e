"""What the framework is timed on.

The cases are the work a user has it do, through its public Python entry
points: uniform 2D ADER-DG steps from the smallest mesh to the largest of the
degree sweep, in FP64 and in mixed precision, with and without the total
variation indicator; steps of an adaptive tree; the gradient of a rollout; a
batch of independent instances; the finite-volume scheme; the 3D scheme.
The meshes are those of the repository's configurations and benchmark, drawn
cases spread over the ranges around them.

`exact` is a plain torch statement of the same discrete equations in 64 bits.
"""
import math

import numpy as np
import torch
from torch.utils.checkpoint import checkpoint

from paper_1905_05524_gb300 import _lib as L
from paper_1905_05524_gb300 import solver as S
from paper_1905_05524_gb300.adjoint import objective_from_theta

PREC = {"fp64": L.ADG_PREC_FP64, "mixed": L.ADG_PREC_MIXED}
T_R, T_C = 2.5, -0.5                       # refinement thresholds of the two-bubble run
F64 = torch.float64


# ------------------------------------------------------------------ the cases
def listed():
    return [
        # Manufactured flow on 9x9 cells, degree 3: the smallest run, one
        # latency-bound step of two launches.
        dict(name="steady_n3_9x9_fp64", kind="steady", degree=3, nx=9, ny=9, prec="fp64", tv=False, steps=1),
        # The rising warm bubble with the indicator of every step: the flagship
        # run, in mixed precision and in FP64.
        dict(name="bubble_n5_81x81_mixed_tv", kind="bubble", degree=5, nx=81, ny=81, prec="mixed", tv=True, steps=1),
        dict(name="bubble_n5_81x81_fp64_tv", kind="bubble", degree=5, nx=81, ny=81, prec="fp64", tv=True, steps=1),
        # Ten steps on an adaptive tree of three cell sizes and the indicator
        # that decides the next regrid.
        dict(name="amr_n5_27x27_mixed", kind="amr", degree=5, nx=27, ny=27, prec="mixed", steps=10),
        # Gradient of a probe misfit with respect to the initial field:
        # checkpointed forward and backward through 40 steps.
        dict(name="adjoint_n3_27x27_fp64", kind="adjoint", degree=3, nx=27, ny=27, prec="fp64", steps=40, every=20),
        # The degree sweep on 243x243 cells: a low degree, the highest, and an
        # odd number of nodes in FP64.
        dict(name="sweep_n2_243x243_mixed", kind="steady", degree=2, nx=243, ny=243, prec="mixed", tv=False, steps=1),
        dict(name="sweep_n7_243x243_mixed", kind="steady", degree=7, nx=243, ny=243, prec="mixed", tv=False, steps=1),
        dict(name="sweep_n4_243x243_fp64", kind="steady", degree=4, nx=243, ny=243, prec="fp64", tv=False, steps=1),
        # 64 independent bubbles of uneven sizes advanced together.
        dict(name="batch_64_bubbles_n5_mixed", kind="batch", degree=5, count=64, lo=9, hi=81, prec="mixed", steps=4),
        # Finite volumes: the colliding bubbles on 630x630 cells.
        dict(name="fv_630x630_mixed", kind="fv", nx=630, ny=630, prec="mixed", steps=10),
        # The 3D bubble, 25^3 cells of degree 2, in both precisions.
        dict(name="bubble3d_n2_25_mixed", kind="bubble3d", degree=2, nx=25, ny=25, nz=25, prec="mixed", steps=4),
        dict(name="bubble3d_n2_25_fp64", kind="bubble3d", degree=2, nx=25, ny=25, nz=25, prec="fp64", steps=2),
    ]


def _log_int(rng, lo, hi):
    return min(hi, max(lo, int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))))


def draw(rng):
    """One more case of the listed ranges: degrees 1..7 (3D 1..4), sides 5..243
    (finite volumes 30..900, 3D 5..32), both precisions."""
    kind = rng.choice(["steady", "steady", "bubble", "bubble", "amr", "adjoint", "batch", "fv", "bubble3d"])
    prec = rng.choice(["fp64", "mixed"])
    if kind in ("steady", "bubble"):
        degree = rng.randint(1, 7)
        nx, ny = _log_int(rng, 5, 243), _log_int(rng, 5, 243)
        while nx * ny * (degree + 1) ** 4 * (20 if prec == "fp64" else 1) > 243 * 243 * 8 ** 4:
            nx, ny = max(5, nx * 2 // 3), max(5, ny * 2 // 3)
        return dict(kind=kind, degree=degree, nx=nx, ny=ny, prec=prec, tv=rng.random() < 0.5, steps=1)
    if kind == "amr":
        return dict(kind=kind, degree=rng.randint(2, 5), nx=_log_int(rng, 9, 40), ny=_log_int(rng, 9, 40), prec=prec,
                    steps=rng.randint(1, 6))
    if kind == "adjoint":
        return dict(kind=kind, degree=rng.randint(1, 4), nx=_log_int(rng, 7, 33), ny=_log_int(rng, 7, 33),
                    prec="fp64", steps=rng.randint(6, 20), every=rng.randint(3, 8))
    if kind == "batch":
        return dict(kind=kind, degree=rng.randint(2, 5), count=_log_int(rng, 2, 32), lo=9, hi=rng.randint(18, 54),
                    prec=prec, steps=rng.randint(1, 4))
    if kind == "fv":
        return dict(kind=kind, nx=_log_int(rng, 30, 900), ny=_log_int(rng, 30, 900), prec=prec, steps=rng.randint(1, 10))
    n = [_log_int(rng, 5, 32) for _ in range(3)]
    return dict(kind=kind, degree=rng.randint(1, 3), nx=n[0], ny=n[1], nz=n[2], prec=prec, steps=rng.randint(1, 3))


# ------------------------------------------------------- inputs (plain torch)
class _Grid:
    """Leaves of one mesh: lower corners and sizes [C, d], nodes per direction n."""

    def __init__(self, cfg, d, corners, sizes, dev):
        self.cfg, self.d, self.n, self.dev = cfg, d, cfg.degree + 1, dev
        self.org = torch.as_tensor(corners, dtype=F64, device=dev)
        self.h = torch.as_tensor(sizes, dtype=F64, device=dev)
        x, w = np.polynomial.legendre.leggauss(self.n)
        self.xi = torch.tensor((x + 1) / 2, dtype=F64, device=dev)
        self.w = torch.tensor(w / 2, dtype=F64, device=dev)

    def coords(self):
        """Node coordinates, one [C, 1.., n, ..1] tensor per direction (x last)."""
        out = []
        for a in range(self.d):
            c = self.org[:, a, None] + self.xi * self.h[:, a, None]
            shape = [c.shape[0]] + [1] * self.d
            shape[-1 - a] = self.n
            out.append(c.reshape(shape))
        return out


def _uniform(cfg, d, dev):
    cnt = [cfg.nx, cfg.ny] + ([cfg.nz] if d == 3 else [])
    org = [cfg.x0, cfg.y0] + ([cfg.z0] if d == 3 else [])
    h = [cfg.Lx / cfg.nx, cfg.Ly / cfg.ny] + ([cfg.Lz / cfg.nz] if d == 3 else [])
    idx = np.stack(np.meshgrid(*[np.arange(c) for c in reversed(cnt)], indexing="ij"), -1).reshape(-1, d)[:, ::-1]
    corners = np.array(org) + idx * np.array(h)
    return _Grid(cfg, d, corners, np.broadcast_to(np.array(h), corners.shape).copy(), dev), idx


def _refined(nx, ny):
    """Leaves (level, ix, iy) of the fixed tree: base cells near a point split
    once, the innermost of their children once more."""
    def near(lv, ix, iy, r):
        h = 3 ** lv
        return math.hypot((ix + 0.5) / (nx * h) - 0.5, (iy + 0.5) / (ny * h) - 0.3) < r
    out = []
    for iy in range(ny):
        for ix in range(nx):
            if not near(0, ix, iy, 0.16):
                out.append((0, ix, iy))
                continue
            for b in range(3):
                for a in range(3):
                    jx, jy = 3 * ix + a, 3 * iy + b
                    if not near(1, jx, jy, 0.04):
                        out.append((1, jx, jy))
                        continue
                    out += [(2, 3 * jx + p, 3 * jy + q) for q in range(3) for p in range(3)]
    return sorted(out, key=lambda c: (c[0], c[2], c[1]))


def _background(z, cfg):
    ex = 1.0 - cfg.g * z / (cfg.gamma * cfg.R / (cfg.gamma - 1.0) * cfg.theta0)
    p = cfg.p0 * ex ** (cfg.gamma / (cfg.gamma - 1.0))
    return p, p / (cfg.R * cfg.theta0 * ex), ex


def _bubble_theta(X, case, seed, k=0):
    """Cosine bubble (two in an adaptive run) whose place, size and strength come from the seed."""
    r = np.random.default_rng([int(seed), k])
    lo, hi = (100.0, 300.0) if case["kind"] == "batch" else (220.0, 270.0)
    out = 0.0
    for A, a, c in [(r.uniform(0.4, 0.6), r.uniform(lo, hi), (r.uniform(480, 520), r.uniform(320, 380)))] + (
            [(r.uniform(-0.2, -0.1), r.uniform(60, 90), (r.uniform(540, 580), r.uniform(600, 660)))]
            if case["kind"] in ("amr", "fv") else []):
        ctr = [c[0]] * (len(X) - 1) + [c[1]]
        rad = torch.sqrt(sum((x - o) ** 2 for x, o in zip(X, ctr)))
        out = out + torch.where(rad <= a, 0.5 * A * (1.0 + torch.cos(math.pi * rad / a)), torch.zeros_like(rad))
    return out


def _bubble_state(theta, z, cfg, d):
    p, _, ex = _background(z, cfg)
    rho = p / (cfg.R * (cfg.theta0 + theta) * ex)
    zero = torch.zeros_like(rho)
    return [rho] + [zero] * d + [p / (cfg.gamma - 1.0) + rho * cfg.g * z]


def _steady_state(X, cfg, seed):
    """The manufactured field under a smooth perturbation."""
    r = np.random.default_rng(int(seed))
    k = 2 * math.pi / cfg.src_L
    x, y = X
    a, f, b, c = r.uniform(0.08, 0.12), r.uniform(-0.3, 0.3), r.uniform(0.02, 0.05), r.uniform(0, 6)
    rho = 1.0 + a * torch.sin(k * (x + y) + f)
    u = cfg.src_U + b * torch.sin(k * x + c) * torch.cos(k * y)
    v = cfg.src_U - b * torch.cos(k * x + c) * torch.sin(k * y)
    p = cfg.src_p + 0.2 * b * torch.cos(k * (x - y) + c)
    return [rho, rho * u, rho * v, p / (cfg.gamma - 1.0) + 0.5 * rho * (u * u + v * v)]


def _config(case, k=0, seed=0):
    prec, kind = PREC[case["prec"]], case["kind"]
    if kind == "steady":
        return S.steady_manufactured_config(case["degree"], case["nx"], case["ny"], prec)
    if kind == "fv":
        cfg = S.fv_bubble_config(case["nx"], case["ny"])
    elif kind == "bubble3d":
        cfg = S.bubble3d_config(case["degree"])
        cfg.nx, cfg.ny, cfg.nz = case["nx"], case["ny"], case["nz"]
    elif kind == "batch":   # sizes belong to the case, the fields in them to the seed
        n = int(np.random.default_rng(3).integers(case["lo"], case["hi"] + 1, size=case["count"])[k])
        cfg = S.atmosphere_config(case["degree"], n, n)
    else:
        cfg = S.atmosphere_config(case["degree"], case["nx"], case["ny"], mu=0.001 if kind == "amr" else 0.01)
        cfg.max_levels = 2 if kind == "amr" else 0
    cfg.precision = prec
    return cfg


def _problem(case, seed, dev, k=0):
    """(config, grid, cell indices or leaves, theta' or None, state, dt) of one mesh."""
    cfg = _config(case, k, seed)
    d = 3 if case["kind"] == "bubble3d" else 2
    if case["kind"] == "amr":
        idx = _refined(cfg.nx, cfg.ny)
        lv = np.array([c[0] for c in idx])
        h = np.stack([cfg.Lx / cfg.nx / 3.0 ** lv, cfg.Ly / cfg.ny / 3.0 ** lv], -1)
        grid = _Grid(cfg, 2, np.array([c[1:] for c in idx]) * h, h, dev)
    else:
        grid, idx = _uniform(cfg, d, dev)
    X = grid.coords()
    th = None if case["kind"] == "steady" else _bubble_theta(X, case, seed, k)
    q = _steady_state(X, cfg, seed) if th is None else _bubble_state(th, X[-1], cfg, d)
    full = [grid.org.shape[0]] + [grid.n] * d
    u = torch.stack([c.expand(full) for c in q], 1).contiguous()
    eq = _Equations(cfg, d)
    lam = (eq.speed(q, X[-1], None) + 2 * _eta(cfg.degree, float(grid.h.min())) * eq.lamv / q[0]).max().item()
    dt = 0.4 * float(grid.h.min()) / (d * (2 * cfg.degree + 1) * lam)
    return cfg, grid, idx, None if th is None else th.expand(full).contiguous(), u, dt


def _fv_problem(case, seed, dev):
    cfg = _config(case)
    x = (torch.arange(cfg.nx, dtype=F64, device=dev) + 0.5) * (cfg.Lx / cfg.nx)
    z = (torch.arange(cfg.ny, dtype=F64, device=dev)[:, None] + 0.5) * (cfg.Ly / cfg.ny)
    U = torch.stack([c.expand(cfg.ny, cfg.nx) for c in _bubble_state(_bubble_theta([x, z], case, seed), z, cfg, 2)])
    return cfg, U.contiguous(), 0.4 / (350.0 * (cfg.nx / cfg.Lx + cfg.ny / cfg.Ly))


def _probes(seed, dev):
    r = np.random.default_rng([int(seed), 77])
    return (torch.tensor(r.uniform(0.0, 1000.0, (64, 2)), device=dev), torch.tensor(r.normal(0.0, 0.1, 64), device=dev))


# ----------------------------------------------------------- prepare and run
def _view(m):
    """The mesh's state without a copy; the mesh owns the memory and lives as long as the view."""
    v = m.state_view()
    v.mesh = m
    return v


def prepare(case, seed):
    dev, kind = torch.device("cuda", 0), case["kind"]
    st = dict(case=case, kind=kind, steps=case["steps"])
    if kind == "fv":
        cfg, U, st["dt"] = _fv_problem(case, seed, dev)
        st["mesh"] = S.FvMesh(cfg)
        st["mesh"].set_state(U)
        return st
    if kind == "batch":
        st["meshes"], st["dts"] = [], []
        for k in range(case["count"]):
            cfg, _, _, _, u, dt = _problem(case, seed, dev, k)
            m = S.Mesh(cfg)
            m.set_state(u)
            st["meshes"].append(m)
            st["dts"].append(dt)
        st["batch"] = S.Batch(st["meshes"])
        st["views"] = [_view(m) for m in st["meshes"]]
        return st
    cfg, _, idx, th, u, st["dt"] = _problem(case, seed, dev)
    m = st["mesh"] = S.Mesh3(cfg) if kind == "bubble3d" else S.Mesh(cfg)
    if kind == "amr":
        for lv in range(2):  # split what the tree has split further
            want = {(c[0] - j, c[1] // 3 ** j, c[2] // 3 ** j) for c in idx for j in range(1, c[0] + 1)}
            m.adapt(torch.tensor([1 if tuple(c) in want else 0 for c in m.leaf_info()], dtype=torch.int8, device=dev))
    if kind == "adjoint":
        st["theta"] = th
        st["xy"], st["target"] = _probes(seed, dev)
        return st
    m.set_state(u)
    if kind != "bubble3d":
        st["view"] = _view(m)
    st["var"] = L.ADG_TV_RHO if kind == "steady" else L.ADG_TV_THETA
    return st


def run(st):
    kind = st["kind"]
    if kind in ("fv", "bubble3d"):
        st["mesh"].step(st["dt"], st["steps"])
        return {"u": st["mesh"].get_state()}
    if kind == "batch":
        st["batch"].step(st["dts"], st["steps"])
        return {"u": st["views"]}
    m = st["mesh"]
    if kind == "adjoint":
        x = st["theta"].detach().requires_grad_(True)
        J = objective_from_theta(x, m, st["dt"], st["steps"], st["case"]["every"], st["xy"], st["target"])
        (g,) = torch.autograd.grad(J, x)
        return {"J": J.detach(), "grad": g}
    if kind == "amr":
        m.step(st["dt"], st["steps"])
        tv, flags, _ = m.tv_indicator(st["var"], T_R, T_C, want_stats=False)
    elif st["case"]["tv"]:
        tv, flags, _ = m.step_tv(st["dt"], st["var"], T_R, T_C, want_stats=False)
    else:
        m.step(st["dt"], st["steps"])
        return {"u": st["view"]}
    return {"u": st["view"], "tv": tv, "flags": flags}


def work(case):
    """State read and written once (per output tensor of the gradient: the
    field read, the gradient written), and the operations of the space-time
    predictor: per evaluation a derivative of every variable and flux along
    every direction and some 55 d operations point by point."""
    if case["kind"] == "fv":
        c = case["nx"] * case["ny"]
        return {"bytes": 64.0 * c, "flops": 500.0 * c * case["steps"]}
    d = 3 if case["kind"] == "bubble3d" else 2
    n = case["degree"] + 1
    if case["kind"] == "batch":
        cells = sum(_config(case, k).cells for k in range(case["count"]))
    elif case["kind"] == "amr":
        cells = len(_refined(case["nx"], case["ny"]))
    else:
        cells = case["nx"] * case["ny"] * case.get("nz", 1)
    V, nodes = d + 2, n ** d
    evals = 1 + (n - 1) * n + n
    step = nodes * (evals * (2.0 * V * d * n * 2 + 2 * V * n + 55.0 * d) + 2 * V * d * n + 4 * d * V * n)
    per = 16.0 * V * nodes
    if case["kind"] == "adjoint":  # forward, recomputed states and about three forward steps of reverse
        return {"bytes": 16.0 * nodes * cells, "flops": step * cells * case["steps"] * 5}
    return {"bytes": per * cells + (9.0 * cells if case.get("tv") or case["kind"] == "amr" else 0.0),
            "flops": step * cells * case["steps"]}


# ------------------------------------------------------------------- exact
def _eta(N, h):
    return (2 * N + 1) / (h * math.sqrt(math.pi / 2.0))


class _Equations:
    """Fluxes and wave speeds of the compressible Navier-Stokes equations with
    gravity along the last direction, in d dimensions, point by point."""

    def __init__(self, cfg, d):
        self.c, self.d = cfg, d
        self.gm1 = cfg.gamma - 1.0
        self.kappa = cfg.mu * cfg.gamma * cfg.R / (self.gm1 * cfg.Pr)
        self.lamv = max(4.0 / 3.0, cfg.gamma / cfg.Pr) * cfg.mu
        self.g = cfg.g if cfg.gravity else 0.0

    def pressure(self, q, z):
        m2 = sum(m * m for m in q[1:-1])
        return self.gm1 * (q[-1] - 0.5 * m2 / q[0] - q[0] * self.g * z)

    def base(self, z):
        return _background(z, self.c)[:2] if self.c.gravity else (torch.zeros_like(z), torch.zeros_like(z))

    def flux(self, q, grads, z, a, heat=None):
        """Flux along direction a; grads[b]: derivatives of q along b."""
        c, d = self.c, self.d
        rho, E = q[0], q[-1]
        v = [m / rho for m in q[1:-1]]
        p = self.pressure(q, z)
        dv = [[(grads[b][1 + i] - v[i] * grads[b][0]) / rho for b in range(d)] for i in range(d)]
        div = sum(dv[i][i] for i in range(d))
        sig = [c.mu * ((2.0 / 3.0 * div if i == a else 0.0) - dv[i][a] - dv[a][i]) for i in range(d)]
        if heat is None:
            # c_v rho dT = dE - (E/rho) drho - rho v.dv - rho g dz
            de = grads[a][-1] - E / rho * grads[a][0] - rho * sum(v[i] * dv[i][a] for i in range(d))
            if a == d - 1:
                de = de - rho * self.g
            heat = de * self.gm1 / (c.R * rho)
        f = [q[1 + a]]
        for i in range(d):
            f.append(q[1 + i] * v[a] + sig[i] + (p - self.base(z)[0] if i == a else 0.0))
        f.append(v[a] * (E + p) + sum(v[i] * sig[i] for i in range(d)) - self.kappa * heat)
        return f

    def source(self, q, z):
        s = [torch.zeros_like(q[0]) for _ in q]
        s[-2] = -self.g * (q[0] - self.base(z)[1])
        return s

    def speed(self, q, z, a):
        c = torch.sqrt(self.c.gamma * self.pressure(q, z) / q[0])
        if a is None:
            return c + torch.sqrt(sum(m * m for m in q[1:-1])) / q[0]
        return c + (q[1 + a] / q[0]).abs()


class _Dg:
    """One ADER-DG step on a list of cells (uniform or a balanced 3:1 tree)."""

    def __init__(self, cfg, grid, idx, adaptive):
        self.cfg, self.g, self.d, self.n = cfg, grid, grid.d, grid.n
        self.eq = _Equations(cfg, grid.d)
        xi, w, n = grid.xi, grid.w, grid.n
        lam = torch.stack([torch.prod(torch.stack([1.0 / (xi[j] - xi[m]) for m in range(n) if m != j])) for j in range(n)])
        D = torch.zeros(n, n, dtype=F64, device=grid.dev)
        for i in range(n):
            for j in range(n):
                if i != j:
                    D[i, j] = lam[j] / lam[i] / (xi[i] - xi[j])
            D[i, i] = -D[i].sum()
        self.D = D
        self.phi = [self._lagrange(torch.zeros(1, dtype=F64, device=grid.dev))[0],
                    self._lagrange(torch.ones(1, dtype=F64, device=grid.dev))[0]]
        K1 = torch.outer(self.phi[1], self.phi[1]) - (w[:, None] * D).T
        self.Kw = torch.linalg.inv(K1) * w
        self.V = (w[:, None] * D / w).T                      # weak volume operator
        self.third = [self._lagrange((s + xi) / 3.0) for s in range(3)]
        self.z = grid.coords()[-1]
        self.faces(idx, adaptive)
        self.Sman = None
        if cfg.source == L.ADG_SRC_STEADY:
            x, y = grid.coords()
            k, a, U, p = 2 * math.pi / cfg.src_L, cfg.src_a, cfg.src_U, cfg.src_p
            s, c = torch.sin(k * (x + y)), torch.cos(k * (x + y))
            rho, r1 = 1.0 + a * s, a * k * c
            lap = 2.0 * p / cfg.R * (2.0 * r1 * r1 / rho ** 3 + a * k * k * s / rho ** 2)
            c = 2.0 * U * r1
            self.Sman = torch.stack([c, c * U, c * U, c * U * U - self.eq.kappa * lap], 1)

    def _lagrange(self, x):
        xi, n = self.g.xi, self.n
        return torch.stack([torch.prod(torch.stack([(x - xi[m]) / (xi[j] - xi[m]) for m in range(n) if m != j]), 0)
                            for j in range(n)], -1)

    def faces(self, idx, adaptive):
        """Per direction: pairs (left cell, right cell, left third, right third) and wall faces (cell, side)."""
        dev, cfg, d = self.g.dev, self.cfg, self.d
        per = [b == L.ADG_BC_PERIODIC for b in ([cfg.bc_x, cfg.bc_y] + ([cfg.bc_z] if d == 3 else []))]
        self.pairs, self.walls = [], []
        if not adaptive:
            cnt = [cfg.nx, cfg.ny] + ([cfg.nz] if d == 3 else [])
            ids = torch.arange(len(idx), device=dev).reshape(cnt[::-1])
            for a in range(d):
                left = ids.movedim(-1 - a, 0)
                right = left.roll(-1, 0)
                if not per[a]:
                    self.walls.append([(left[-1].reshape(-1), 1), (left[0].reshape(-1), 0)])
                    left, right = left[:-1], right[:-1]
                else:
                    self.walls.append([])
                self.pairs.append([(left.reshape(-1), right.reshape(-1), None, None)])
            return
        pos = {tuple(c): k for k, c in enumerate(idx)}
        for a in range(2):
            got, wall = {}, [[], []]
            for k, (lv, ix, iy) in enumerate(idx):
                c = [ix, iy]
                top = (cfg.nx, cfg.ny)[a] * 3 ** lv
                if c[a] == 0:
                    wall[0].append(k)
                if c[a] == top - 1:
                    wall[1].append(k)
                    continue
                c[a] += 1
                if (lv, *c) in pos:
                    got.setdefault((None, None), []).append((k, pos[(lv, *c)]))
                elif lv and (lv - 1, c[0] // 3, c[1] // 3) in pos:
                    got.setdefault((None, c[1 - a] % 3), []).append((k, pos[(lv - 1, c[0] // 3, c[1] // 3)]))
                else:
                    for s in range(3):
                        f = [3 * c[0], 3 * c[1]]
                        f[1 - a] += s
                        got.setdefault((s, None), []).append((k, pos[(lv + 1, *f)]))
            self.pairs.append([(torch.tensor([p[0] for p in v], device=dev), torch.tensor([p[1] for p in v], device=dev), *s)
                               for s, v in got.items()])
            self.walls.append([(torch.tensor(wall[1], device=dev), 1), (torch.tensor(wall[0], device=dev), 0)])

    def along(self, M, q, a):
        return torch.movedim(torch.movedim(q, -1 - a, -1) @ M.T, -1, -1 - a)

    def evaluate(self, q, z, h, sman):
        """Fluxes, source and gradients of q[c, (k,) v, nodes]; the variable axis is -1-d."""
        at = q.dim() - 1 - self.d
        shape = [-1] + [1] * (q.dim() - 1)
        zz = z if at == 1 else z[:, None]
        gr = [self.along(self.D, q, a) / h[:, a].reshape(shape) for a in range(self.d)]
        ql, gl = q.unbind(at), [g.unbind(at) for g in gr]
        F = [torch.stack(self.eq.flux(ql, gl, zz, a), at) for a in range(self.d)]
        src = torch.stack(self.eq.source(ql, zz), at)
        if sman is not None:
            src = src + (sman if at == 1 else sman[:, None])
        return F, src, gr

    def predict(self, u, z, h, sman, dt):
        n = self.n
        q = u[:, None].expand(-1, n, *[-1] * (u.dim() - 1))
        shape = [-1] + [1] * u.dim()
        for _ in range(n):
            F, R, _ = self.evaluate(q, z, h, sman)
            for a in range(self.d):
                R = R - self.along(self.D, F[a], a) / h[:, a].reshape(shape)
            q = u[:, None] + dt * torch.tensordot(R, self.Kw, dims=([1], [1])).movedim(-1, 1)
        F, R, G = self.evaluate(q, z, h, sman)
        mean = lambda t: torch.tensordot(t, self.g.w, dims=([1], [0]))  # noqa: E731
        return [mean(q)] + [mean(f) for f in F] + [mean(R)] + [mean(g) for g in G]

    def step(self, u, dt):
        d, g, h = self.d, self.g, self.g.h
        part = max(1, 12_000_000 // (u[0].numel() * self.n))
        outs = [self.predict(u[i:i + part], self.z[i:i + part], h[i:i + part],
                             None if self.Sman is None else self.Sman[i:i + part], dt) for i in range(0, len(u), part)]
        avg = [torch.cat(t) if len(outs) > 1 else t[0] for t in zip(*outs)]
        del outs
        qb, Fb, Sb, Gb = avg[0], avg[1:1 + d], avg[1 + d], avg[2 + d:]
        shape = [-1] + [1] * (d + 1)
        new = Sb
        for a in range(d):
            new = new + self.along(self.V, Fb[a], a) / h[:, a].reshape(shape)
        for a in range(d):
            ext = [[torch.tensordot(t, self.phi[s], dims=([t.dim() - 1 - a], [0])) for t in (qb, Fb[a])] for s in (0, 1)]
            star = [torch.zeros_like(ext[0][0]), torch.zeros_like(ext[0][0])]
            zn = self.z.expand(-1, *[self.n] * d)
            zf = [(zn.select(zn.dim() - 1 - a, 0) if a < d - 1 else
                   (g.org[:, a] + s * h[:, a]).reshape([-1] + [1] * (d - 1)).expand(-1, *[self.n] * (d - 1)))
                  for s in (0, 1)]
            for lc, rc, ls, rs in self.pairs[a]:
                (ql, fl), (qr, fr), z = [t[lc] for t in ext[1]], [t[rc] for t in ext[0]], zf[1][lc]
                if ls is not None:     # the left cell is the coarse one: its trace on a third of the face
                    ql, fl, z = ql @ self.third[ls].T, fl @ self.third[ls].T, zf[0][rc]
                if rs is not None:
                    qr, fr = qr @ self.third[rs].T, fr @ self.third[rs].T
                hh = torch.minimum(h[lc, a], h[rc, a])
                f = self.riemann(ql, fl, qr, fr, z, a, hh)
                back = lambda s: f if s is None else (f * g.w) @ self.third[s] / (3.0 * g.w)  # noqa: E731
                star[1] = star[1].index_add(0, lc, back(ls))
                star[0] = star[0].index_add(0, rc, back(rs))
            for c, s in self.walls[a]:
                q, f, z = ext[s][0][c], ext[s][1][c], zf[s][c]
                gr = [torch.tensordot(t[c], self.phi[s], dims=([t.dim() - 1 - a], [0])).unbind(1) for t in Gb]
                gq = list(q.unbind(1))
                gq[1 + a] = -gq[1 + a]
                if self.cfg.gravity:
                    p, rho = self.eq.base(z)
                    gq[0], gq[-1] = rho + 0.0 * gq[0], p / self.eq.gm1 + rho * self.eq.g * z
                cp = self.cfg.gamma * self.cfg.R / self.eq.gm1
                heat = torch.full_like(z, -self.eq.g / cp if a == d - 1 else 0.0)
                gf = torch.stack(self.eq.flux(gq, gr, z, a, heat), 1)
                gq = torch.stack(gq, 1)
                f = self.riemann(q, f, gq, gf, z, a, h[c, a]) if s else self.riemann(gq, gf, q, f, z, a, h[c, a])
                star[s] = star[s].index_add(0, c, f)
            for s, sign in ((1, -1.0), (0, 1.0)):
                sh = [1] * (d + 2)
                sh[d + 1 - a] = self.n
                lift = (self.phi[s] / g.w).reshape(sh) / h[:, a].reshape(shape)
                new = new + sign * lift * star[s].unsqueeze(d + 1 - a)
        return u + dt * new

    def riemann(self, ql, fl, qr, fr, z, a, h):
        eta = _eta(self.n - 1, 1.0) / h.reshape([-1] + [1] * (self.d - 1))
        s = torch.maximum(*[self.eq.speed(q.unbind(1), z, a) + 2.0 * eta * self.eq.lamv / q[:, 0] for q in (ql, qr)])
        return 0.5 * (fl + fr) - 0.5 * s[:, None] * (qr - ql)

    def theta(self, u, z):
        p = self.eq.pressure(u.unbind(1), z)
        c = self.cfg
        return p / (u[:, 0] * c.R) * (c.p0 / p) ** ((c.gamma - 1.0) / c.gamma)

    def variation(self, u, var):
        f = self.theta(u, self.z) if var == L.ADG_TV_THETA else u[:, 0]
        w, h = self.g.w, self.g.h
        s = sum((self.along(self.D, f, a) / h[:, a, None, None]).abs() for a in range(2))
        return torch.einsum("cji,j,i->c", s, w, w)


def _fv_step(U, dt, cfg):
    """MUSCL-Hancock with van Albada slopes of the perturbation; slip walls on every side."""
    eq = _Equations(cfg, 2)
    hs = (cfg.Lx / cfg.nx, cfg.Ly / cfg.ny)
    zc = ((torch.arange(cfg.ny, dtype=F64, device=U.device) + 0.5) * hs[1])[:, None].expand(cfg.ny, cfg.nx)

    def rest(z):
        p, rho = eq.base(z)
        return torch.stack([rho, 0 * rho, 0 * rho, p / eq.gm1 + rho * eq.g * z])

    def flux(q, z, a):
        none = torch.zeros_like(z)
        return torch.stack(eq.flux(q.unbind(0), [[none] * 4] * 2, z, a, none))

    up = U - rest(zc)
    zf = [(zc, zc), (zc - 0.5 * hs[1], zc + 0.5 * hs[1])]
    face = []
    for a in range(2):
        ax = 2 - a
        lo, hi = up - up.roll(1, ax), up.roll(-1, ax) - up
        den = lo * lo + hi * hi
        s = torch.where(lo * hi > 0, lo * hi * (lo + hi) / torch.where(den > 0, den, torch.ones_like(den)), torch.zeros_like(up))
        s.index_fill_(ax, torch.tensor([0, s.shape[ax] - 1], device=U.device), 0.0)
        face.append([rest(z) + up + 0.5 * o * s for z, o in zip(zf[a], (-1.0, 1.0))])
    src = torch.stack(eq.source(U.unbind(0), zc))
    half = 0.5 * dt * src
    for a in range(2):
        half = half - 0.5 * dt / hs[a] * (flux(face[a][1], zf[a][1], a) - flux(face[a][0], zf[a][0], a))
    out = U + dt * torch.stack(eq.source((U + half).unbind(0), zc))
    for a in range(2):
        ax = 2 - a
        lo, hi = face[a][0] + half, face[a][1] + half
        zl, zh = zf[a]

        def wall(q, z):
            g = q.clone()
            g[1 + a] = -q[1 + a]
            b = rest(z)
            g[0], g[3] = b[0], b[3]
            return g

        # faces 0..n along the axis: left states (wall, hi...), right states (lo..., wall)
        left = torch.cat([wall(lo.narrow(ax, 0, 1), zl.narrow(ax - 1, 0, 1)), hi], ax)
        right = torch.cat([lo, wall(hi.narrow(ax, -1, 1), zh.narrow(ax - 1, -1, 1))], ax)
        z = torch.cat([zl, zh.narrow(ax - 1, -1, 1)], ax - 1)
        s = torch.maximum(eq.speed(left.unbind(0), z, a), eq.speed(right.unbind(0), z, a))
        f = 0.5 * (flux(left, z, a) + flux(right, z, a)) - 0.5 * s * (right - left)
        n = U.shape[ax]
        out = out - dt / hs[a] * (f.narrow(ax, 1, n) - f.narrow(ax, 0, n))
    return out


def _exact_gradient(dg, th, dt, steps, xy, target):
    cfg, g, d = dg.cfg, dg.g, 2
    x = th.clone().requires_grad_(True)
    u = torch.stack(_bubble_state(x, dg.z.expand_as(x), cfg, d), 1)
    for _ in range(steps):
        u = checkpoint(lambda t: dg.step(t, dt), u, use_reentrant=False)
    r = dg.theta(u, dg.z) - cfg.theta0
    cell = [(xy[:, a] / h).long().clamp(0, m - 1) for a, (h, m) in
            enumerate([(cfg.Lx / cfg.nx, cfg.nx), (cfg.Ly / cfg.ny, cfg.ny)])]
    c = cell[1] * cfg.nx + cell[0]
    loc = (xy - g.org[c]) / g.h[c]
    val = torch.einsum("pj,pi,pji->p", dg._lagrange(loc[:, 1]), dg._lagrange(loc[:, 0]), r[c])
    J = ((val - target) ** 2).sum()
    return J.detach(), torch.autograd.grad(J, x)[0]


def exact(case, seed):
    dev, kind = torch.device("cuda", 0), case["kind"]
    if kind == "fv":
        cfg, U, dt = _fv_problem(case, seed, dev)
        for _ in range(case["steps"]):
            U = _fv_step(U, dt, cfg)
        return {"u": U}
    done = []
    for k in range(case.get("count", 1)):
        cfg, grid, idx, th, u, dt = _problem(case, seed, dev, k)
        dg = _Dg(cfg, grid, idx, kind == "amr")
        if kind == "adjoint":
            J, g = _exact_gradient(dg, th, dt, case["steps"], *_probes(seed, dev))
            return {"J": J, "grad": g}
        for _ in range(case["steps"]):
            u = dg.step(u, dt)
        done.append(u)
    if kind == "batch":
        return {"u": done}
    if kind == "amr" or case.get("tv"):
        return {"u": u, "tv": dg.variation(u, L.ADG_TV_RHO if kind == "steady" else L.ADG_TV_THETA), "flags": None}
    return {"u": u}
