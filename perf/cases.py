"""Performance cases: the work that users of this package have it do.

Each case is one call (or the few calls that belong together) of the public
binding ``paper_2608_24348_gb300.sem`` on inputs that live on the GPU:

  ax         the element operator sem_ax alone
  assembled  sem_ax followed by sem_dssum, the operator of a user's own iteration
  poisson    a singular pressure-Poisson solve by Jacobi-PCG, FP64 or FP32 inner
  velocity   the three Helmholtz solves of a time step in one batched call
  batch      independent Poisson problems of several orders and sizes in one launch
  gmres      the pressure solve by flexible GMRES + hybrid Schwarz multigrid
  tgv        whole Taylor-Green time steps

``listed()`` names fixed sizes, ``draw(rng)`` draws more of the same ranges,
``prepare``/``run`` make the inputs and do one pass, ``work`` counts the bytes
and operations a pass cannot do without, and ``exact`` restates the result in
plain FP64 torch from the textbook formulas.
"""
from __future__ import annotations

import math
import random

import numpy as np
import torch

TWO_PI = 2.0 * math.pi
NU = 1.0 / 1600.0  # Re = 1600
ORDERS = (3, 4, 5, 6, 7, 8, 9)
BATCH_ORDERS = (5, 7, 9)


# ---------------------------------------------------------------------------
# The cases
# ---------------------------------------------------------------------------

def _ax(N, nel, dtype, h1=0.01, h2=1000.0):
    return {"kind": "ax", "N": N, "nelx": nel[0], "nely": nel[1], "nelz": nel[2], "dtype": dtype,
            "h1": h1, "h2": h2}


def _assembled(N, nel, dtype, h1=1.0, h2=0.0):
    return dict(_ax(N, nel, dtype, h1, h2), kind="assembled")


def _poisson(N, nel, inner, periodic=True):
    return {"kind": "poisson", "N": N, "nelx": nel[0], "nely": nel[1], "nelz": nel[2],
            "inner": inner, "periodic": periodic}


def _velocity(N, nel, dt):
    return {"kind": "velocity", "N": N, "nelx": nel[0], "nely": nel[1], "nelz": nel[2], "dt": dt}


def _batch(nprob, pick, most):
    return {"kind": "batch", "nprob": nprob, "pick": pick, "most": most}


def _gmres(N, nel):
    return {"kind": "gmres", "N": N, "nelx": nel[0], "nely": nel[1], "nelz": nel[2]}


def _tgv(N, nel, pressure, projection, dt, steps):
    return {"kind": "tgv", "N": N, "nelx": nel[0], "nely": nel[1], "nelz": nel[2],
            "pressure": pressure, "projection": projection, "dt": dt, "steps": steps}


def listed():
    return [
        # the headline operator: 32^3 elements of order 7 on a deformed mesh, the
        # Helmholtz coefficients of a step of 1e-3
        dict(_ax(7, (32, 32, 32), "f64"), name="ax_f64_32"),
        # the same in FP32, the operator of a mixed-precision user's inner iteration
        dict(_ax(7, (32, 32, 32), "f32"), name="ax_f32_32"),
        # the paper's other order (P = 8) on a box with three different edges
        dict(_ax(8, (18, 21, 17), "f64"), name="ax_f64_p8"),
        # a small assembled operator: launches and latency
        dict(_assembled(7, (6, 5, 7), "f64"), name="assembled_small"),
        # the plain Poisson problem, 4^3 elements of order 5: the smallest solve
        dict(_poisson(5, (4, 4, 4), "f64"), name="poisson_4"),
        # the pressure Poisson problem in FP64 at a middle size
        dict(_poisson(7, (16, 16, 16), "f64"), name="poisson_f64"),
        # the mixed-precision pressure solve (FP32 inner, FP64 refinement), large
        dict(_poisson(7, (24, 24, 24), "f32"), name="poisson_mixed"),
        # the velocity solves of a P = 8 step on a ragged box: few iterations
        dict(_velocity(8, (15, 13, 14), 2e-3), name="velocity_p8"),
        # uneven problems of orders 5, 7 and 9 in one persistent launch
        dict(_batch(12, 4, 12), name="batch_uneven"),
        # the paper's pressure solver
        dict(_gmres(7, (16, 16, 16)), name="gmres_hsmg"),
        # whole steps of the flagship run: FP64, Jacobi-PCG pressure solve
        dict(_tgv(7, (32, 32, 32), "pcg", 0, 1e-3, 2), name="tgv_32"),
        # whole steps with the paper's solver settings (GMRES + HSMG, projection
        # space of 20) at P = 8
        dict(_tgv(8, (12, 14, 13), "gmres_hsmg", 20, 2e-3, 2), name="tgv_p8_gmres"),
    ]


def _log_uniform(rng, lo, hi):
    return math.exp(rng.uniform(math.log(lo), math.log(hi)))


def _edges(rng, N, nodes, least=2, most=40):
    """Three edges of about nodes / (N+1)^3 elements, up to a factor 1.4 apart."""
    e = (nodes / (N + 1) ** 3) ** (1.0 / 3.0)
    return tuple(min(most, max(least, round(e * rng.uniform(0.85, 1.2)))) for _ in range(3))


def draw(rng):
    kind = rng.choice(("ax", "ax", "assembled", "poisson", "poisson", "velocity", "batch", "gmres", "tgv"))
    N = rng.choice(ORDERS)
    if kind == "ax":
        h1, h2 = rng.choice(((1.0, 0.0), (0.01, 1000.0), (NU, 1.0 / 1e-3)))
        return _ax(N, _edges(rng, N, _log_uniform(rng, 5e4, 1.2e7)), rng.choice(("f64", "f32")), h1, h2)
    if kind == "assembled":
        return _assembled(N, _edges(rng, N, _log_uniform(rng, 2e4, 6e6)), rng.choice(("f64", "f32")))
    if kind == "poisson":
        return _poisson(N, _edges(rng, N, _log_uniform(rng, 1e4, 1.5e6)), rng.choice(("f64", "f32")),
                        rng.random() < 0.7)
    if kind == "velocity":
        return _velocity(N, _edges(rng, N, _log_uniform(rng, 5e4, 3e6)), rng.choice((1e-3, 2e-3, 4e-3)))
    if kind == "batch":
        return _batch(rng.randint(4, 12), rng.randint(0, 10 ** 6), rng.choice((8, 10, 12)))
    if kind == "gmres":
        N = rng.choice((5, 6, 7, 8))
        return _gmres(N, _edges(rng, N, _log_uniform(rng, 5e4, 1.5e6), 3))
    N = rng.choice((5, 6, 7, 8))
    pressure = rng.choice(("pcg", "gmres_hsmg"))
    return _tgv(N, _edges(rng, N, _log_uniform(rng, 1e5, 1.5e6), 3), pressure,
                20 if pressure == "gmres_hsmg" else rng.choice((0, 20)), rng.choice((1e-3, 2e-3)), 2)


def _nel(case):
    return case["nelx"], case["nely"], case["nelz"]


def _batch_sizes(case):
    """(N, edge) of every problem of a batch, from the case's own number."""
    rng = random.Random(case["pick"])
    return [(rng.choice(BATCH_ORDERS), rng.randint(4, case["most"])) for _ in range(case["nprob"])]


# ---------------------------------------------------------------------------
# Inputs (from the seed alone; used by prepare and by exact)
# ---------------------------------------------------------------------------

def _vertices(nel, deform, seed):
    """Vertex grid [(nelz+1), (nely+1), (nelx+1), 3] of [0, 2 pi]^3; with deform
    every interior vertex moves by up to 10 % of the element size."""
    nx, ny, nz = nel
    v = np.empty((nz + 1, ny + 1, nx + 1, 3))
    v[..., 0] = np.linspace(0.0, TWO_PI, nx + 1)[None, None, :]
    v[..., 1] = np.linspace(0.0, TWO_PI, ny + 1)[None, :, None]
    v[..., 2] = np.linspace(0.0, TWO_PI, nz + 1)[:, None, None]
    if deform and min(nel) > 1:
        h = TWO_PI / np.array([nx, ny, nz])
        d = np.random.default_rng([seed, 1]).uniform(-0.1, 0.1, (nz - 1, ny - 1, nx - 1, 3))
        v[1:nz, 1:ny, 1:nx] += d * h
    return v


def _unique_index(N, nel, periodic, dev):
    """Unique grid index of every local node, [E * (N+1)^3], and their number."""
    ax = []
    for d in range(3):
        ng = nel[d] * N + (0 if periodic else 1)
        e = torch.arange(nel[d], device=dev)[:, None]
        i = torch.arange(N + 1, device=dev)[None, :]
        ax.append(((e * N + i) % ng, ng))
    (gx, nx), (gy, ny), (gz, nz) = ax
    g = gx[None, None, :, None, None, :] + nx * (gy[None, :, None, None, :, None] +
                                                 ny * gz[:, None, None, :, None, None])
    return g.reshape(-1), nx * ny * nz


def _random_field(N, nel, periodic, seed, dev):
    """A continuous field, uniform in [-1, 1] per unique node."""
    idx, ng = _unique_index(N, nel, periodic, dev)
    gen = torch.Generator(device=dev).manual_seed(seed * 7919 + 2)
    return (torch.rand(ng, generator=gen, device=dev, dtype=torch.float64) * 2.0 - 1.0)[idx]


def _modes(seed, count, kmax):
    rng = np.random.default_rng([seed, 3])
    k = rng.integers(-kmax, kmax + 1, (count, 3))
    k[~k.any(axis=1)] = (1, 0, 0)
    return k, rng.standard_normal((count, 3)), rng.uniform(0.0, TWO_PI, count)


def _source(seed, x, y, z):
    """A smooth mean-free right-hand side: cosines with |k|^-2 amplitudes."""
    k, a, phase = _modes(seed, 12, 5)
    f = torch.zeros_like(x)
    for m in range(len(k)):
        k0, k1, k2 = (float(t) for t in k[m])
        f += float(a[m, 0] / (k[m] ** 2).sum()) * torch.cos(k0 * x + k1 * y + k2 * z + float(phase[m]))
    return f


def _flow(seed, x, y, z):
    """The Taylor-Green vortex and its pressure, shifted and scaled by the seed."""
    rng = np.random.default_rng([seed, 5])
    v0, (a, b, c) = float(rng.uniform(0.8, 1.2)), (float(t) for t in rng.uniform(0.0, TWO_PI, 3))
    x, y, z = x + a, y + b, z + c
    u = [v0 * torch.sin(x) * torch.cos(y) * torch.cos(z), -v0 * torch.cos(x) * torch.sin(y) * torch.cos(z),
         torch.zeros_like(x)]
    p = v0 ** 2 * (torch.cos(2 * x) + torch.cos(2 * y)) * (torch.cos(2 * z) + 2.0) / 16.0
    return u, p


# ---------------------------------------------------------------------------
# One pass through the package
# ---------------------------------------------------------------------------

def _context(sem, N, nel, deform, seed, periodic=True):
    return sem.Ctx(N, nel, (TWO_PI,) * 3, (int(periodic),) * 3, vertices=_vertices(nel, deform, seed))


def _coords(ctx):
    xyz = torch.empty(3 * ctx.nL, dtype=torch.float64, device="cuda")
    ctx.coords(xyz)
    return xyz.view(3, -1)


def _assembled_source(ctx, seed):
    """dssum(B f) of the smooth source f."""
    b = torch.empty(ctx.nL, dtype=torch.float64, device="cuda")
    ctx.ax(_source(seed, *_coords(ctx)), b, 0.0, 1.0, "f64_native")
    return ctx.dssum(b, "f64")


def prepare(case, seed):
    from paper_2608_24348_gb300 import sem
    sem.load()
    dev = torch.device("cuda")
    kind = case["kind"]
    s = {"kind": kind, "sem": sem, "case": case}
    if kind == "batch":
        sizes = _batch_sizes(case)
        s["ctx"] = [_context(sem, N, (e, e, e), True, seed + p) for p, (N, e) in enumerate(sizes)]
        s["b"] = [_assembled_source(c, seed + p) for p, c in enumerate(s["ctx"])]
        s["x"] = [torch.empty_like(b) for b in s["b"]]
        return s
    N, nel = case["N"], _nel(case)
    if kind in ("ax", "assembled"):
        ctx = _context(sem, N, nel, True, seed)
        t = torch.float32 if case["dtype"] == "f32" else torch.float64
        s["u"] = _random_field(N, nel, True, seed, dev).to(t)
        s["w"] = torch.empty_like(s["u"])
    elif kind == "poisson":
        ctx = _context(sem, N, nel, True, seed, case["periodic"])
        s["b"] = _assembled_source(ctx, seed)
        s["x"] = torch.empty_like(s["b"])
    elif kind == "velocity":
        ctx = _context(sem, N, nel, True, seed)
        x, y, z = _coords(ctx)
        s["guess"] = [t.contiguous() for t in _flow(seed, x, y, z)[0]]
        s["b"] = []
        for c in range(3):
            b = torch.empty_like(s["guess"][c])
            ctx.ax(s["guess"][c] * 1.01 + 0.02 * _source(seed + c, x, y, z), b, NU, 11.0 / 6.0 / case["dt"],
                   "f64_native")
            s["b"].append(ctx.dssum(b, "f64"))
        s["x"] = [torch.empty_like(b) for b in s["b"]]
    elif kind == "gmres":
        ctx = _context(sem, N, nel, True, seed)
        s["b"] = _assembled_source(ctx, seed)
        s["x"] = torch.empty_like(s["b"])
        s["hsmg"] = sem.HSMG(ctx, (N, 3, 1))
    else:
        ctx = _context(sem, N, nel, False, seed)
        # a stream of one's own, as a program has whose steps are to be captured
        s["stream"] = torch.cuda.Stream()
        T = sem.TGV(ctx, NU, case["dt"])
        if case["projection"]:
            T.set_projection(case["projection"])
        if case["pressure"] != "pcg":
            T.set_pressure_solver(case["pressure"])
        u, p = _flow(seed, *_coords(ctx))
        u = [t.contiguous() for t in u]
        for level in (2, 1, 0):  # third-order steps from the first one on
            T.set(*u, p if level == 0 else None, level=level, step=3)
        s["tgv"] = T
        s["out"] = [torch.empty_like(p) for _ in range(4)]
        torch.cuda.synchronize()
    s["ctx"] = ctx
    return s


def run(s):
    sem, case, kind = s["sem"], s["case"], s["kind"]
    if kind == "ax":
        return s["ctx"].ax(s["u"], s["w"], case["h1"], case["h2"], case["dtype"])
    if kind == "assembled":
        s["ctx"].ax(s["u"], s["w"], case["h1"], case["h2"], case["dtype"])
        return s["ctx"].dssum(s["w"], case["dtype"])
    if kind == "poisson":
        s["x"].zero_()
        info = s["ctx"].pcg_solve(s["b"], s["x"], 1.0, 0.0, inner=case["inner"])
        return {"x": s["x"], "status": info["status"]}
    if kind == "velocity":
        for x, g in zip(s["x"], s["guess"]):
            x.copy_(g)
        h2 = 11.0 / 6.0 / case["dt"]
        infos = sem.pcg_solve_batched([s["ctx"]] * 3, s["b"], s["x"], [NU] * 3, [h2] * 3, tol=1e-6,
                                      abs_tol=True)
        return {"x": s["x"], "status": [i["status"] for i in infos]}
    if kind == "batch":
        for x in s["x"]:
            x.zero_()
        n = len(s["x"])
        infos = sem.pcg_solve_batched(s["ctx"], s["b"], s["x"], [1.0] * n, [0.0] * n, inner="f32")
        return {"x": s["x"], "status": [i["status"] for i in infos]}
    if kind == "gmres":
        s["x"].zero_()
        info = s["hsmg"].gmres(s["b"], s["x"])
        return {"x": s["x"], "status": info["status"]}
    d = s["tgv"].step(case["steps"], stream=s["stream"])
    u, v, w, p = s["out"]
    s["tgv"].get(u, v, w, p, stream=s["stream"])
    return {"u": u, "v": v, "w": w, "p": p, "ke": [r["ke"] for r in d],
            "enstrophy": [r["enstrophy"] for r in d], "status": [r["status"] for r in d]}


# ---------------------------------------------------------------------------
# What a pass cannot do without
# ---------------------------------------------------------------------------

def _nodes(N, nel):
    return nel[0] * nel[1] * nel[2] * (N + 1) ** 3


def _op_flops(N):
    return 12 * (N + 1) + 20  # six contractions, the factors and the mass term per node


def _cg_iterations(N, nel):
    """Jacobi-PCG iterations of a periodic Poisson problem to 1e-10, measured trend."""
    return 6.5 * N * max(nel)


def work(case):
    kind = case["kind"]
    if kind == "batch":
        total = {"bytes": 0.0, "flops": 0.0}
        for N, e in _batch_sizes(case):
            w = work(_poisson(N, (e, e, e), "f32"))
            total = {k: total[k] + w[k] for k in total}
        return total
    N, nel = case["N"], _nel(case)
    n = _nodes(N, nel)
    if kind in ("ax", "assembled"):
        word = 4 if case["dtype"] == "f32" else 8
        return {"bytes": 9.0 * word * n, "flops": float(_op_flops(N)) * n}  # u, w, seven factors
    # one CG iteration: seven factors, w written and read, x and r read and written,
    # p read and written, the preconditioner read
    iteration = 7 + 2 + 2 + 2 + 2 + 1
    if kind == "poisson":
        word, it = (4, 1.15) if case["inner"] == "f32" else (8, 1.0)
        its = it * _cg_iterations(N, nel)
        return {"bytes": its * iteration * word * n, "flops": its * (_op_flops(N) + 12.0) * n}
    if kind == "velocity":
        return {"bytes": 3 * 3.0 * iteration * 8 * n, "flops": 3 * 3.0 * (_op_flops(N) + 12.0) * n}
    # one V-cycle in FP32 (smoother, residual operator, transfers) and one FP64 operator
    vcycle = {"bytes": (9 * 8 + 14 * 4.0) * n, "flops": (2 * _op_flops(N) + 12.0 * (N + 1)) * n}
    if kind == "gmres":
        return {k: 24.0 * v + (24 * 24 * 8.0 * n if k == "bytes" else 0.0) for k, v in vcycle.items()}
    # a step: 18 history fields read, 6 written, J^-1 and the factors twice; the
    # dealiased convection's 15 interpolations; the solves
    M = (3 * (N + 1) + 1) // 2
    interp = 2.0 * (M * (N + 1) ** 3 + M * M * (N + 1) ** 2 + M ** 3 * (N + 1)) / (N + 1) ** 3
    step = {"bytes": (18 + 6 + 2 * 16) * 8.0 * n, "flops": (15 * interp + 30.0 * (N + 1)) * n}
    solves = work(_velocity(N, nel, case["dt"]))
    pressure_its = 30.0 if case["pressure"] == "pcg" else 0.0
    for k in step:
        step[k] += solves[k] + pressure_its * solves[k] / 9.0
        if case["pressure"] != "pcg":
            step[k] += vcycle[k]
        step[k] *= case["steps"]
    return step


# ---------------------------------------------------------------------------
# The same results in plain FP64 torch
# ---------------------------------------------------------------------------

def _gll(N):
    """GLL nodes and weights: the roots of (1 - x^2) P_N'."""
    P = np.polynomial.legendre.Legendre.basis(N)
    dP, d2P = P.deriv(), P.deriv(2)
    r = np.sort(dP.roots().real)
    for _ in range(3):
        r = r - dP(r) / d2P(r)
    x = np.concatenate([[-1.0], 0.5 * (r - r[::-1]), [1.0]])
    return x, 2.0 / (N * (N + 1) * P(x) ** 2)


def _lagrange(x, at):
    """[q, j]: the Lagrange basis polynomial of node j at the point q."""
    out = np.ones((len(at), len(x)))
    for j in range(len(x)):
        for k in range(len(x)):
            if k != j:
                out[:, j] *= (at - x[k]) / (x[j] - x[k])
    return out


def _derivative(x):
    n = len(x)
    c = np.array([np.prod([x[j] - x[k] for k in range(n) if k != j]) for j in range(n)])
    D = np.zeros((n, n))
    for i in range(n):
        for j in range(n):
            if i != j:
                D[i, j] = c[i] / c[j] / (x[i] - x[j])
        D[i, i] = -D[i].sum()
    return D


class _Mesh:
    """Geometry, operator, gather-scatter and PCG of one mesh, FP64."""

    def __init__(self, N, nel, vertices, periodic, dev):
        self.N, self.n, self.nel, self.dev = N, N + 1, nel, dev
        self.E = nel[0] * nel[1] * nel[2]
        self.xi, self.w = _gll(N)
        t = lambda a: torch.tensor(a, dtype=torch.float64, device=dev)  # noqa: E731
        self.t = t
        self.D = t(_derivative(self.xi))
        v = t(vertices)
        nx, ny, nz = nel
        corners = [v[a:nz + a, b:ny + b, c:nx + c].reshape(self.E, 3)
                   for a in (0, 1) for b in (0, 1) for c in (0, 1)]
        self.corners = torch.stack(corners, 1)  # [E][t, s, r][3]
        w3 = self.w[:, None, None] * self.w[None, :, None] * self.w[None, None, :]
        self.xyz, jac = self.mapping(self.xi)
        det = torch.linalg.det(jac)
        self.jinv = torch.linalg.inv(jac)  # [..., a, c] = dr_a / dx_c
        del jac
        self.B = det * t(w3)
        G = self.B[..., None, None] * (self.jinv @ self.jinv.transpose(-1, -2))
        self.G = [[G[..., a, b].contiguous() if b >= a else None for b in range(3)] for a in range(3)]
        for a in range(3):
            for b in range(a):
                self.G[a][b] = self.G[b][a]
        del G
        self.idx, self.ng = _unique_index(N, nel, periodic, dev)
        self.mult = self.dssum(torch.ones_like(self.B))
        self.volume = self.B.sum()

    def mapping(self, pts):
        """Coordinates [E, k, j, i, 3] and Jacobian [E, k, j, i, c, a] at the tensor grid of pts."""
        p = self.t(pts)
        l, d = torch.stack([(1 - p) / 2, (1 + p) / 2]), torch.tensor([-0.5, 0.5], dtype=p.dtype, device=p.device)
        one = torch.ones_like(p)
        dl = torch.stack([d[0] * one, d[1] * one])
        C = self.corners.reshape(self.E, 2, 2, 2, 3)
        ev = lambda a, b, c: torch.einsum("etsrc,tk,sj,ri->ekjic", C, a, b, c)  # noqa: E731
        return ev(l, l, l), torch.stack([ev(l, l, dl), ev(l, dl, l), ev(dl, l, l)], -1)

    def shape(self, u):
        return u.reshape(self.E, self.n, self.n, self.n)

    def grad(self, u):
        n, E = self.n, u.shape[0]
        return (u @ self.D.T, self.D @ u, (self.D @ u.reshape(E, n, n * n)).reshape(u.shape))

    def grad_t(self, r, s, t):
        n, E = self.n, r.shape[0]
        return r @ self.D + self.D.T @ s + (self.D.T @ t.reshape(E, n, n * n)).reshape(r.shape)

    def ax(self, u, h1, h2):
        g = self.grad(u)
        f = [h1 * (self.G[a][0] * g[0] + self.G[a][1] * g[1] + self.G[a][2] * g[2]) for a in range(3)]
        return self.grad_t(*f) + h2 * self.B * u

    def dssum(self, u):
        s = torch.zeros(self.ng, dtype=u.dtype, device=u.device).index_add_(0, self.idx, u.reshape(-1))
        return s[self.idx].reshape(u.shape)

    def dot(self, a, b):
        return float((a * b / self.mult).sum())

    def diagonal(self, h1, h2):
        D2 = self.D ** 2
        n, G = self.n, self.G
        d = G[0][0] @ D2 + D2.T @ G[1][1] + (D2.T @ G[2][2].reshape(self.E, n, n * n)).reshape(self.B.shape)
        g = torch.diagonal(self.D)
        i, j, k = g[None, None, None, :], g[None, None, :, None], g[None, :, None, None]
        d = d + 2.0 * (i * j * G[0][1] + i * k * G[0][2] + j * k * G[1][2])
        return self.dssum(h1 * d + h2 * self.B)

    def pcg(self, b, x, h1, h2, tol, absolute=False, maxit=20000):
        singular = h2 == 0.0
        if singular:
            b = b - self.dot(b, torch.ones_like(b)) / self.ng
        m = 1.0 / self.diagonal(h1, h2)
        r = b - self.dssum(self.ax(x, h1, h2))
        target = tol if absolute else tol * math.sqrt(self.dot(b, b))
        p, rz, best, stale = None, 0.0, math.inf, 0
        for _ in range(maxit):
            norm = math.sqrt(self.dot(r, r))
            stale = 0 if norm < 0.999 * best else stale + 1
            best = min(best, norm)
            if norm <= target or stale > 400:
                break
            z = m * r
            old, rz = rz, self.dot(r, z)
            p = z if p is None else z + (rz / old) * p
            q = self.dssum(self.ax(p, h1, h2))
            alpha = rz / self.dot(p, q)
            x = x + alpha * p
            r = r - alpha * q
        if singular:
            x = x - (self.B * x).sum() / self.volume
        return x


def _interp(mesh, J, u):
    """(J x J x J) u on a chunk of elements."""
    E, n, M = u.shape[0], J.shape[1], J.shape[0]
    u = J @ (u @ J.T)
    return (J @ u.reshape(E, n, M * M)).reshape(E, M, M, M)


def _interp_t(mesh, J, f):
    E, M, n = f.shape[0], J.shape[0], J.shape[1]
    f = J.T @ (f @ J)
    return (J.T @ f.reshape(E, M, n * n)).reshape(E, n, n, n)


def _convect(mesh, u):
    """Weak dealiased (u . grad) u_c on ceil(3(N+1)/2) Gauss points, chunk by chunk."""
    M = (3 * mesh.n + 1) // 2
    eta, wq = np.polynomial.legendre.leggauss(M)
    J = mesh.t(_lagrange(mesh.xi, eta))
    w3 = mesh.t(wq[:, None, None] * wq[None, :, None] * wq[None, None, :])
    out = [torch.empty_like(c) for c in u]
    whole = mesh.corners, mesh.E
    for e0 in range(0, whole[1], 2048):
        e = slice(e0, min(whole[1], e0 + 2048))
        mesh.corners, mesh.E = whole[0][e], e.stop - e.start
        wd = torch.linalg.det(mesh.mapping(eta)[1]) * w3
        mesh.corners, mesh.E = whole
        fu = [_interp(mesh, J, c[e]) * wd for c in u]
        for c in range(3):
            g = mesh.grad(u[c][e])
            f = 0.0
            for d in range(3):
                f = f + fu[d] * _interp(mesh, J, sum(mesh.jinv[e][..., a, d] * g[a] for a in range(3)))
            out[c][e] = _interp_t(mesh, J, f)
    return out


def _exact_tgv(case, seed, dev):
    N, nel, dt = case["N"], _nel(case), case["dt"]
    m = _Mesh(N, nel, _vertices(nel, False, seed), True, dev)
    u, p = _flow(seed, *(m.xyz[..., d].contiguous() for d in range(3)))
    hist, C = [u, u, u], [_convect(m, u)] * 2
    tol_p = 1e-4 if case["pressure"] == "pcg" and not case["projection"] else 1e-9
    a, bk, b0 = (3.0, -3.0, 1.0), (3.0, -1.5, 1.0 / 3.0), 11.0 / 6.0
    Bs = m.dssum(m.B)
    ke, en = [], []
    for _ in range(case["steps"]):
        C = [_convect(m, hist[0])] + C[:2]
        F = [-(a[0] * C[0][c] + a[1] * C[1][c] + a[2] * C[2][c]) for c in range(3)]
        back = [(bk[0] * hist[0][c] + bk[1] * hist[1][c] + bk[2] * hist[2][c]) / dt for c in range(3)]
        g = [m.dssum(F[c]) / Bs + back[c] for c in range(3)]
        flux = [m.B * sum(m.jinv[..., r, c] * g[c] for c in range(3)) for r in range(3)]
        p = m.pcg(m.dssum(m.grad_t(*flux)), p, 1.0, 0.0, tol_p, absolute=True)
        gp = m.grad(p)
        new = []
        for c in range(3):
            dp = sum(m.jinv[..., r, c] * gp[r] for r in range(3))
            rhs = m.dssum(F[c] + m.B * (back[c] - dp))
            guess = a[0] * hist[0][c] + a[1] * hist[1][c] + a[2] * hist[2][c]
            new.append(m.pcg(rhs, guess, NU, b0 / dt, 1e-6, absolute=True))
        hist = [new] + hist[:2]
        g = [m.grad(c) for c in new]
        du = [[sum(m.jinv[..., r, d] * g[c][r] for r in range(3)) for d in range(3)] for c in range(3)]
        curl = (du[2][1] - du[1][2], du[0][2] - du[2][0], du[1][0] - du[0][1])
        ke.append(float((m.B * sum(c * c for c in new)).sum() / (2 * m.volume)))
        en.append(float((m.B * sum(c * c for c in curl)).sum() / (2 * m.volume)))
        del g, du, curl, flux
    flat = [t.reshape(-1) for t in hist[0] + [p]]
    return {"u": flat[0], "v": flat[1], "w": flat[2], "p": flat[3], "ke": ke, "enstrophy": en,
            "status": [None] * case["steps"]}


def _exact_poisson(N, nel, periodic, seed, dev):
    m = _Mesh(N, nel, _vertices(nel, True, seed), periodic, dev)
    b = m.dssum(m.B * _source(seed, *(m.xyz[..., d] for d in range(3))))
    return m.pcg(b, torch.zeros_like(b), 1.0, 0.0, 1e-13).reshape(-1)


def exact(case, seed):
    dev = torch.device("cuda" if torch.cuda.is_available() else "cpu")
    kind = case["kind"]
    if kind == "batch":
        x = [_exact_poisson(N, (e, e, e), True, seed + p, dev) for p, (N, e) in enumerate(_batch_sizes(case))]
        return {"x": x, "status": [None] * len(x)}
    N, nel = case["N"], _nel(case)
    if kind in ("ax", "assembled"):
        m = _Mesh(N, nel, _vertices(nel, True, seed), True, dev)
        u = _random_field(N, nel, True, seed, dev)
        if case["dtype"] == "f32":
            u = u.float().double()
        w = m.ax(m.shape(u), case["h1"], case["h2"])
        return (m.dssum(w) if kind == "assembled" else w).reshape(-1)
    if kind in ("poisson", "gmres"):
        return {"x": _exact_poisson(N, nel, case.get("periodic", True), seed, dev), "status": None}
    if kind == "velocity":
        m = _Mesh(N, nel, _vertices(nel, True, seed), True, dev)
        x, y, z = (m.xyz[..., d].contiguous() for d in range(3))
        h2 = 11.0 / 6.0 / case["dt"]
        out = []
        for c, g in enumerate(_flow(seed, x, y, z)[0]):
            b = m.dssum(m.ax(g * 1.01 + 0.02 * _source(seed + c, x, y, z), NU, h2))
            out.append(m.pcg(b, g, NU, h2, 1e-6, absolute=True).reshape(-1))
        return {"x": out, "status": [None] * 3}
    return _exact_tgv(case, seed, dev)
