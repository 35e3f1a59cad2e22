"""Performance cases of the library: what a user's program asks of it, through its public entry points.

A case is one simulation from its initial condition (`Solver.set_state`, SSP-RK3 steps, `Solver.moments`),
a batch of such simulations (`Batch`), or one call of the allocation-free equilibrium entry point. The
sizes are those of the repository's workloads (workloads.py) and tests, or lie between them. `exact` is
the same arithmetic in plain FP64 torch (flux reconstruction with upwind fluxes, trapezoid moments, the
conservative Maxwellian by Newton's method, SSP-RK3), written independently of the library.
"""
from __future__ import annotations

import functools
import math

import numpy as np
import torch

from paper_2308_06196_gb300 import bgk
from paper_2308_06196_gb300 import workloads as W

PERIODIC, DIRICHLET, WALL = 0, 1, 2
TWO_PI = 2.0 * math.pi
CFL = 0.1
MAX_WORK = 7.3e9  # degrees of freedom times steps of the largest listed case


def listed():
    return [
        # a single shock tube run to a checkpoint: the smallest problems, where launches and latency
        # count; returns f as a restart file would hold it
        dict(name="tube", kind="tube", ex=24, p=2, n=12, steps=20),
        # a parameter study: 256 independent shock tubes of mixed sizes stepped as one batch
        dict(name="tube_batch", kind="batch", members=256, mesh_seed=0, steps=4),
        # a transverse shear wave on a long line, planar velocity space
        dict(name="shear_line", kind="shear", ex=65536, p=3, n=32, steps=4),
        # planar Taylor-Green flow on quadrilaterals, planar velocity space
        dict(name="vortex_quads", kind="vortex2", ex=128, ey=128, p=3, n=32, steps=4),
        # the headline workload: Taylor-Green flow on hexahedra
        dict(name="vortex", kind="vortex3", ex=16, ey=16, ez=16, p=3, n=24, steps=2),
        # body-force-driven rarefied flow between diffuse walls
        dict(name="channel", kind="channel", ex=32, ey=16, ez=4, p=2, n=32, steps=2),
        # Mach-5 normal shock in a duct with the positivity limiter
        dict(name="shock_duct", kind="shock", ex=128, ey=2, ez=2, p=2, n=48, steps=3),
        # a gas with a viscosity law (variable collision time) and the limiter; odd sizes throughout
        dict(name="viscous_gas", kind="gas", ex=7, ey=9, ez=5, p=3, n=21, limiter=True, steps=2),
        # Taylor-Green flow on a curved structured mesh
        dict(name="vortex_curved", kind="curved", ex=16, ey=16, ez=16, p=3, n=24, steps=2),
        # the same flow on an unstructured curved mesh in a random element order
        dict(name="vortex_unstructured", kind="unstructured", ex=8, ey=8, ez=8, p=3, n=24, steps=2),
        # an accuracy check of a user's setting: the all-FP64 form on a reduced mesh
        dict(name="vortex_fp64", kind="fp64", ex=6, ey=6, ez=6, p=3, n=16, steps=2),
        # moments and conservative Maxwellians of distributions that another program holds
        dict(name="equilibria", kind="equilibria", points=32768, n=24),
    ]


def draw(rng):
    def log_int(lo, hi):
        return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))

    kind = rng.choice(["tube", "batch", "shear", "vortex2", "vortex3", "vortex3", "channel", "shock", "gas", "curved",
                       "unstructured", "fp64", "equilibria"])
    while True:
        if kind == "tube":
            c = dict(kind=kind, ex=log_int(16, 512), p=rng.randint(1, 4), n=rng.randint(12, 24),
                     steps=rng.randint(5, 20))
        elif kind == "batch":
            c = dict(kind=kind, members=log_int(8, 256), mesh_seed=rng.randint(1, 10**6), steps=rng.randint(2, 6))
        elif kind == "shear":
            c = dict(kind=kind, ex=log_int(512, 65536), p=rng.randint(1, 4), n=rng.randint(16, 40),
                     steps=rng.randint(2, 6))
        elif kind == "vortex2":
            c = dict(kind=kind, ex=log_int(16, 128), ey=log_int(16, 128), p=rng.randint(1, 3), n=rng.randint(16, 40),
                     steps=rng.randint(2, 5))
        elif kind in ("vortex3", "curved", "gas"):
            c = dict(kind=kind, ex=log_int(4, 20), ey=log_int(4, 20), ez=log_int(4, 20), p=rng.randint(1, 3),
                     n=rng.randint(12, 28), steps=rng.randint(1, 3))
            if kind == "gas":
                c["limiter"] = rng.random() < 0.5
        elif kind == "channel":
            c = dict(kind=kind, ex=log_int(4, 32), ey=log_int(6, 24), ez=log_int(2, 8), p=rng.randint(1, 3),
                     n=rng.randint(14, 32), steps=rng.randint(1, 3))
        elif kind == "shock":
            c = dict(kind=kind, ex=2 * log_int(16, 64), ey=log_int(1, 4), ez=log_int(1, 4), p=2, n=rng.randint(40, 50),
                     steps=rng.randint(1, 4))
        elif kind == "unstructured":
            c = dict(kind=kind, ex=log_int(4, 9), ey=log_int(4, 9), ez=log_int(4, 9), p=rng.randint(1, 3),
                     n=rng.randint(12, 26), steps=rng.randint(1, 3))
        elif kind == "fp64":
            c = dict(kind=kind, ex=log_int(2, 7), ey=log_int(2, 7), ez=log_int(2, 7), p=rng.randint(1, 3),
                     n=rng.randint(10, 18), steps=rng.randint(1, 2))
        else:
            c = dict(kind=kind, points=log_int(256, 32768), n=rng.randint(12, 28))
        if _size(c) * c.get("steps", 1) <= MAX_WORK:
            return c


# ------------------------------------------------------------------------------------------------
# problem definitions: meshes, velocity grids, collision times and boundary states by kind of case
# ------------------------------------------------------------------------------------------------
def _rankine_hugoniot(mach, gamma=5.0 / 3.0):
    u1 = mach * math.sqrt(gamma)
    r2 = (gamma + 1.0) * mach**2 / ((gamma - 1.0) * mach**2 + 2.0)
    p2 = 1.0 + 2.0 * gamma * (mach**2 - 1.0) / (gamma + 1.0)
    return (1.0, u1, 0.0, 0.0, 1.0), (r2, u1 / r2, 0.0, 0.0, p2 / r2)


def _problem(c, seed):
    """Mesh, velocity grid, collision time and options of a case (the shock tube's end states are the
    seed's)."""
    k, n, p = c["kind"], c["n"], c["p"]
    q = dict(p=p, nv=(n, n, n), tau=1e-3, bc=[[PERIODIC] * 2 for _ in range(3)],
             bc_state=np.zeros((3, 2, 5)), opts={})
    if k == "tube":
        rng = _rng(seed, 1)
        ends = [(r, 0.0, 0.0, 0.0, t) for r, t in zip(rng.uniform(0.125, 1.0, 2), rng.uniform(0.8, 1.25, 2))]
        q.update(dim=1, ne=(c["ex"],), lo=(0.0,), hi=(1.0,), vmax=8.0, tau=c.get("tau", 1e-2))
        q["bc"][0] = [DIRICHLET] * 2
        q["bc_state"][0] = ends
    elif k == "shear":
        q.update(dim=1, ne=(c["ex"],), lo=(0.0,), hi=(1.0,), vmax=7.0, nv=(n, n, 1))
    elif k == "vortex2":
        q.update(dim=2, ne=(c["ex"], c["ey"]), lo=(0.0,) * 2, hi=(TWO_PI,) * 2, vmax=7.0, nv=(n, n, 1))
    else:
        q.update(dim=3, ne=(c["ex"], c["ey"], c["ez"]), lo=(0.0,) * 3, hi=(TWO_PI,) * 3, vmax=5.0)
    if k == "channel":
        q.update(hi=(2.0, 1.0, 0.25), vmax=6.0, tau=0.1 / math.sqrt(math.pi / 2.0))
        q["bc"][1] = [WALL] * 2
        q["bc_state"][1][:, 4] = 1.0
        q["opts"]["body_force"] = (0.01, 0.0, 0.0)
    elif k == "shock":
        q.update(hi=(c["ex"] / 8.0, c["ey"] / 8.0, c["ez"] / 8.0), vmax=14.0, tau=5e-4)
        q["bc"][0] = [DIRICHLET] * 2
        q["bc_state"][0] = _rankine_hugoniot(5.0)
        q["opts"]["limiter"] = True
    elif k == "gas":
        q["opts"].update(mu_ref=2e-3, mu_omega=0.81, limiter=bool(c["limiter"]))
    elif k == "fp64":
        q["opts"]["precision"] = bgk.FP64
    return q


@functools.lru_cache(maxsize=8)
def _members(members, mesh_seed):
    """The tubes of a batch: 16 to 128 elements, p = 2 or 3, 12^3 to 32^3 velocities, tau 1e-4 to 1e-1."""
    rng = np.random.default_rng(mesh_seed)
    return tuple(dict(kind="tube", ex=int(rng.integers(16, 129)), p=int(rng.integers(2, 4)),
                      n=int(rng.choice([12, 16, 24, 32])), tau=float(10.0 ** rng.uniform(-4.0, -1.0)))
                 for _ in range(members))


def _npts(c):
    d = 3 if "ez" in c else (2 if "ey" in c else 1)
    return c["ex"] * c.get("ey", 1) * c.get("ez", 1) * (c["p"] + 1) ** d


def _size(c):
    """Degrees of freedom: points times velocities."""
    if c["kind"] == "batch":
        return sum(_size(m) for m in _members(c["members"], c["mesh_seed"]))
    if c["kind"] == "equilibria":
        return c["points"] * c["n"] ** 3
    return _npts(c) * c["n"] ** (2 if c["kind"] in ("shear", "vortex2") else 3)


def work(c):
    """Bytes: the state sampled once, then per step the three stages' reads of their source and of f^n and
    the writes of their output (8 + 12 + 12 bytes per degree of freedom in FP32, twice that in FP64).
    Operations per degree of freedom and stage: the line sums and traces of every direction, the relaxation
    and the five moments."""
    dof = _size(c)
    if c["kind"] == "equilibria":
        return dict(bytes=4.0 * dof + 80.0 * c["points"], flops=10.0 * dof)
    parts = _members(c["members"], c["mesh_seed"]) if c["kind"] == "batch" else [c]
    size = 8 if c["kind"] == "fp64" else 4
    flops = 0.0
    for m in parts:
        dim = 3 if "ez" in m else (2 if "ey" in m else 1)
        metric = 5 * dim if m["kind"] in ("curved", "unstructured") else 0
        flops += _size(m) * (dim * (2 * (m["p"] + 1) + 6) + metric + 16 + 10)
    return dict(bytes=float(dof) * size * (1 + 8 * c["steps"]), flops=3.0 * c["steps"] * flops)


# ------------------------------------------------------------------------------------------------
# inputs
# ------------------------------------------------------------------------------------------------
def _rng(*parts):
    """A generator seeded by all parts (numbers, or tuples of numbers)."""
    flat = []
    for t in parts:
        flat += list(t) if isinstance(t, tuple) else [t]
    return np.random.default_rng([int(t) % (1 << 63) for t in flat])


def _operators(p):
    """Gauss-Legendre nodes, half weights, derivative matrix, end interpolants and the Radau corrections'
    derivatives on the reference element [-1, 1]."""
    x, w = np.polynomial.legendre.leggauss(p + 1)
    lam = np.array([1.0 / np.prod(x[j] - np.delete(x, j)) for j in range(p + 1)])
    D = np.zeros((p + 1, p + 1))
    for i in range(p + 1):
        for j in range(p + 1):
            if i != j:
                D[i, j] = lam[j] / lam[i] / (x[i] - x[j])
        D[i, i] = -D[i].sum()

    def ends(y):
        t = lam / (y - x)
        return t / t.sum()

    lm, lp = ends(-1.0), ends(1.0)
    return dict(x=x, wq=0.5 * w, D=D, lm=lm, lp=lp, gl=-lm / w, gr=lp / w)


def _points(q):
    """Node coordinates [n_x, 3], element-major with x fastest among elements and among nodes."""
    xg = _operators(q["p"])["x"]
    ax = []
    for d in range(3):
        if d < q["dim"]:
            h = (q["hi"][d] - q["lo"][d]) / q["ne"][d]
            ax.append(q["lo"][d] + h * (np.arange(q["ne"][d])[:, None] + 0.5 * (xg[None, :] + 1.0)))
        else:
            ax.append(np.zeros((1, 1)))
    shape = tuple(a.shape[0] for a in ax[::-1]) + tuple(a.shape[1] for a in ax[::-1])
    X = np.empty(shape + (3,))
    for d in range(3):
        s = [1] * 6
        s[2 - d], s[5 - d] = ax[d].shape
        X[..., d] = ax[d].reshape(s)
    return X.reshape(-1, 3)


def _waves(x, q, rng):
    """A seeded smooth field with the periods of the box, |value| <= 1."""
    f = np.zeros(len(x))
    for _ in range(3):
        a = np.zeros(len(x))
        for d in range(q["dim"]):
            a += rng.integers(-2, 3) * TWO_PI / (q["hi"][d] - q["lo"][d]) * x[:, d]
        f += rng.uniform(-1.0, 1.0) * np.cos(a + rng.uniform(0.0, TWO_PI))
    return f / 3.0


def _prim(c, q, x, seed):
    """Primitive state (rho, u, v, w, T) at the nodes: the flow of the case with a seeded disturbance."""
    k = c["kind"]
    P = np.zeros((len(x), 5))
    P[:, 0] = P[:, 4] = 1.0
    X, Y, Z = x[:, 0], x[:, 1], x[:, 2]
    if k == "tube":
        for i, side in enumerate((X < 0.5, X >= 0.5)):
            P[side] = q["bc_state"][0][i]
    elif k == "shock":
        for i, side in enumerate((X < 0.5 * q["hi"][0], X >= 0.5 * q["hi"][0])):
            P[side] = q["bc_state"][0][i]
    elif k == "shear":
        P[:, 2] = 0.1 * np.sin(TWO_PI * X)
    elif k == "vortex2":
        U0 = 0.1 * math.sqrt(2.0)
        P[:, 1] = U0 * np.sin(X) * np.cos(Y)
        P[:, 2] = -U0 * np.cos(X) * np.sin(Y)
        P[:, 4] = 1.0 + U0 * U0 / 4.0 * (np.cos(2 * X) + np.cos(2 * Y))
    elif k != "channel":
        U0 = 0.1 * math.sqrt(5.0 / 3.0)
        P[:, 1] = U0 * np.sin(X) * np.cos(Y) * np.cos(Z)
        P[:, 2] = -U0 * np.cos(X) * np.sin(Y) * np.cos(Z)
        P[:, 4] = 1.0 + U0 * U0 / 16.0 * (np.cos(2 * X) + np.cos(2 * Y)) * (np.cos(2 * Z) + 2.0)
    P[:, 0] *= 1.0 + 0.03 * _waves(x, q, _rng(seed, 2))
    P[:, 4] *= 1.0 + 0.03 * _waves(x, q, _rng(seed, 3))
    for d in range(2 if q["nv"][2] == 1 else 3):
        P[:, 1 + d] += 0.03 * _waves(x, q, _rng(seed, 4 + d))
    return P


def _dt(q, P):
    speed = sum(q["vmax"] * q["ne"][d] / (q["hi"][d] - q["lo"][d]) for d in range(q["dim"]))
    tau = q["tau"]
    if "mu_ref" in q["opts"]:
        tau = float(np.min(q["opts"]["mu_ref"] * P[:, 4] ** (q["opts"]["mu_omega"] - 1.0) / P[:, 0]))
    return min(CFL / speed, tau)


def _curved(q, x):
    """Smooth periodic displacement of the nodes by 0.3 of an element's width."""
    h = np.array([(q["hi"][d] - q["lo"][d]) / q["ne"][d] for d in range(3)])
    return x + np.stack([0.3 * h[d] * np.sin(x[:, (d + 1) % 3]) for d in range(3)], 1)


@functools.lru_cache(maxsize=8)
def _relabelled(ne, p):
    return W.unstructured_box(ne, p, seed=11)


def _solver(c, q, **more):
    vm = q["vmax"]
    return bgk.Solver(q["dim"], list(q["ne"]), list(q["lo"]), list(q["hi"]), q["p"], q["nv"], (-vm,) * 3, (vm,) * 3,
                      q["tau"], bc=q["bc"], bc_state=q["bc_state"], **q["opts"], **more)


def _distributions(c, seed):
    """f [points, n^3] FP32: drifting Maxwellians with seeded states and 5 % noise."""
    n, m = c["n"], c["points"]
    dev = "cuda" if torch.cuda.is_available() else "cpu"
    u = torch.from_numpy(_rng(seed, 1).uniform(-0.5, 0.5, (m, 5))).to(dev)
    v = torch.linspace(-6.0, 6.0, n, dtype=torch.float64, device=dev)
    T = 1.0 + 0.4 * u[:, 4:]
    a = [torch.exp(-((v[None] - 0.8 * u[:, 1 + d:2 + d]) ** 2) / (2 * T)) / torch.sqrt(TWO_PI * T) for d in range(3)]
    a[0] = a[0] * (1.0 + 0.4 * u[:, :1])
    noise = 1.0 + 0.05 * torch.cos(torch.arange(n**3, device=dev, dtype=torch.float64) * (1.0 + seed % 17))
    f = torch.empty(m, n**3, dtype=torch.float32, device=dev)
    for i in range(0, m, 2048):
        s = slice(i, min(m, i + 2048))
        t = a[2][s, :, None, None] * a[1][s, None, :, None] * a[0][s, None, None, :]
        f[s] = t.reshape(-1, n**3).mul_(noise).float()
    return f


def prepare(c, seed):
    if c["kind"] == "equilibria":
        f = _distributions(c, seed)
        Q = torch.empty(c["points"], 5, dtype=torch.float64, device="cuda")
        return dict(kind="equilibria", n=c["n"], f=f, Q=Q, prim=torch.empty_like(Q))
    if c["kind"] == "batch":
        mem, prim, dts = [], [], []
        for i, m in enumerate(_members(c["members"], c["mesh_seed"])):
            q = _problem(m, (seed, i))
            P = _prim(m, q, _points(q), (seed, i))
            mem.append(_solver(m, q, chunks=1))
            prim.append(torch.from_numpy(P).cuda())
            dts.append(_dt(q, P))
        Q = torch.empty(sum(len(P) for P in prim), 5, dtype=torch.float64, device="cuda")
        torch.cuda.synchronize()
        return dict(kind="batch", members=mem, batch=bgk.Batch(mem), prim=prim, dt=dts, steps=c["steps"], Q=Q,
                    parts=torch.split(Q, [len(P) for P in prim]))
    q = _problem(c, seed)
    x = _points(q)
    P = _prim(c, q, x, seed)
    s = _solver(c, q)
    dt = _dt(q, P)
    if c["kind"] == "curved":
        s.set_geometry(_curved(q, x))
    elif c["kind"] == "unstructured":
        mesh = _relabelled(q["ne"], q["p"])
        s.set_connectivity(mesh["nbr"], mesh["nface"], mesh["orient"])
        s.set_geometry(_curved(q, x)[mesh["node_map"]])
        P = P[mesh["node_map"]]
    prim = torch.from_numpy(np.ascontiguousarray(P)).cuda()
    out = torch.empty_like(prim)
    torch.cuda.synchronize()
    return dict(kind=c["kind"], solver=s, prim=prim, dt=dt, steps=c["steps"], Q=out)


def run(st):
    if st["kind"] == "equilibria":
        n = st["n"]
        rc = bgk.equilibrium_noalloc(st["f"], (n,) * 3, (-6.0,) * 3, (6.0,) * 3, st["Q"], st["prim"])
        if rc != bgk.BGK_OK:
            raise RuntimeError("equilibrium_noalloc returned %d" % rc)
        return dict(Q=st["Q"], prim=st["prim"])
    if st["kind"] == "batch":
        for m, P in zip(st["members"], st["prim"]):
            m.set_state(P)
        st["batch"].step(st["dt"], st["steps"])
        for m, Q in zip(st["members"], st["parts"]):
            m.moments(Q)
        return dict(Q=st["Q"])
    s = st["solver"]
    s.set_state(st["prim"])
    s.step(st["dt"], st["steps"])
    if st["kind"] == "tube":  # a checkpoint on the host
        return dict(Q=s.moments(), f=s.get_f())
    return dict(Q=s.moments(st["Q"]))


# ------------------------------------------------------------------------------------------------
# the same in FP64 torch
# ------------------------------------------------------------------------------------------------
class _Plain64:
    """One problem in FP64: f as blocks of velocities [b, elements (z, y, x), nodes (z, y, x)]."""

    def __init__(self, q, x=None, dev="cpu"):
        self.q, self.dim, self.dev = q, q["dim"], dev
        self.op = _operators(q["p"])
        n1 = q["p"] + 1
        self.shape = tuple(q["ne"][::-1]) + (n1,) * self.dim
        self.npts = int(np.prod(self.shape))
        self.m = 2 if q["nv"][2] == 1 else 3
        v1, w1 = [], []
        for d in range(3):
            n = q["nv"][d]
            if n == 1:
                v1.append(np.zeros(1))
                w1.append(np.ones(1))
                continue
            v = -q["vmax"] + np.arange(n) * (2.0 * q["vmax"] / (n - 1))
            w = np.full(n, 2.0 * q["vmax"] / (n - 1))
            w[[0, -1]] *= 0.5
            v1.append(v)
            w1.append(w)
        self.v1 = [torch.tensor(a, device=dev) for a in v1]
        self.w1 = [torch.tensor(a, device=dev) for a in w1]
        nx, ny, nz = q["nv"]
        k = torch.arange(nx * ny * nz, device=dev)
        self.k = [k % nx, k // nx % ny, k // (nx * ny)]
        self.v = torch.stack([self.v1[d][self.k[d]] for d in range(3)], 1)
        self.w = self.w1[0][self.k[0]] * self.w1[1][self.k[1]] * self.w1[2][self.k[2]]
        nb = max(1, int(6e7 // self.npts))
        self.blocks = [slice(a, min(len(k), a + nb)) for a in range(0, len(k), nb)]
        self.ghost = {}
        for d in range(self.dim):
            for s in range(2):
                b = q["bc"][d][s]
                if b != PERIODIC:
                    r, *u, T = q["bc_state"][d][s]
                    self.ghost[d, s] = self.maxwellian(r if b == DIRICHLET else 1.0, u, T)
        if x is not None:
            self.metric(x)
        else:
            self.Ja = None

    def maxwellian(self, r, u, T):
        e = sum((self.v[:, d] - u[d]) ** 2 for d in range(self.m))
        return r / (TWO_PI * T) ** (self.m / 2) * torch.exp(-e / (2 * T))

    # --- geometry -----------------------------------------------------------------------------
    def along(self, u, M, axis):
        """M applied along an axis (nodes of one direction)."""
        return torch.movedim(torch.tensordot(u, torch.tensor(M, device=self.dev), dims=([axis], [1])), -1, axis)

    def metric(self, x):
        X = torch.tensor(x, device=self.dev).reshape(self.shape + (3,))
        node = [5, 4, 3]
        dX = [[self.along(X[..., n], self.op["D"], node[j]) for j in range(3)] for n in range(3)]
        self.J = sum(dX[0][a] * (dX[1][b] * dX[2][c] - dX[1][c] * dX[2][b]) for a, b, c in ((0, 1, 2), (1, 2, 0), (2, 0, 1)))
        Ja = torch.empty(self.shape + (3, 3), dtype=torch.float64, device=self.dev)  # [..., i, n]
        for n in range(3):
            m, l = (n + 1) % 3, (n + 2) % 3
            V = [X[..., l] * dX[m][j] for j in range(3)]
            for i in range(3):
                a, b = (i + 1) % 3, (i + 2) % 3
                Ja[..., i, n] = -(self.along(V[b], self.op["D"], node[a]) - self.along(V[a], self.op["D"], node[b]))
        self.Ja = Ja
        self.normal = {}
        for d in range(3):
            ends = [torch.tensordot(Ja[..., d, :], torch.tensor(self.op[l], device=self.dev), dims=([5 - d], [0]))
                    for l in ("lm", "lp")]
            left = 0.5 * (ends[0] + torch.roll(ends[1], 1, 2 - d))
            self.normal[d] = (left, torch.roll(left, -1, 2 - d))

    # --- residual of one block of velocities -----------------------------------------------------
    def traces(self, u):
        lo = sum(float(self.op["lm"][j]) * u[j] for j in range(len(u)))
        hi = sum(float(self.op["lp"][j]) * u[j] for j in range(len(u)))
        return lo, hi

    def outside(self, lo, hi, d, b, rw):
        """The neighbours' traces at the two ends of every element (ghost values at boundary faces)."""
        ax = 1 + (self.dim - 1 - d)
        left, right = torch.roll(hi, 1, ax), torch.roll(lo, -1, ax)
        for s, t in ((0, left), (1, right)):
            if (d, s) in self.ghost:
                g = self.ghost[d, s][b].reshape((-1,) + (1,) * (t.dim() - 2))
                if (d, s) in rw:
                    g = g * rw[d, s][None]
                t.select(ax, 0 if s == 0 else t.shape[ax] - 1).copy_(g.expand_as(t.select(ax, 0)))
        return left, right

    def residual(self, f, b, rw):
        v = self.v[b]
        nb = f.shape[0]
        out = torch.zeros_like(f)
        for d in range(self.dim):
            na = 1 + self.dim + (self.dim - 1 - d)
            o = out.unbind(na)
            u = f.unbind(na)
            lo, hi = self.traces(u)
            left, right = self.outside(lo, hi, d, b, rw)
            if self.Ja is None:
                c = (-v[:, d] * 2.0 * self.q["ne"][d] / (self.q["hi"][d] - self.q["lo"][d])).reshape((nb,) + (1,) * (lo.dim() - 1))
                pos = (v[:, d] >= 0).reshape(c.shape)
                jl = torch.where(pos, left - lo, torch.zeros((), dtype=f.dtype, device=f.device)) * c
                jr = torch.where(pos, torch.zeros((), dtype=f.dtype, device=f.device), right - hi) * c
                F = [t * c for t in u]
            else:
                a = torch.tensordot(v, self.Ja[..., d, :], dims=([1], [self.Ja.dim() - 2]))
                F = (a * f).unbind(na)
                del a
                flo, fhi = self.traces(F)
                nl, nr = (torch.tensordot(v, N, dims=([1], [N.dim() - 1])) for N in self.normal[d])
                jl = nl * torch.where(nl >= 0, left, lo) - flo
                jr = nr * torch.where(nr >= 0, hi, right) - fhi
            for i in range(len(u)):
                o[i].add_(jl, alpha=float(self.op["gl"][i])).add_(jr, alpha=float(self.op["gr"][i]))
                for j in range(len(u)):
                    o[i].add_(F[j], alpha=float(self.op["D"][i, j]))
            del F
        if self.Ja is not None:
            out.div_(-self.J)
        return out

    def wall_density(self, fs):
        """Per face point of a diffuse wall, the density of no net discrete mass flux."""
        rw = {}
        for (d, s), g in self.ghost.items():
            if self.q["bc"][d][s] != WALL:
                continue
            un = self.v[:, d] * (1.0 if s else -1.0)
            num = 0.0
            for f, b in zip(fs, self.blocks):
                e = f.select(1 + self.dim - 1 - d, -1 if s else 0)
                t = self.traces(e.unbind(self.dim + (self.dim - 1 - d)))[s]
                num = num + torch.tensordot(self.w[b] * un[b].clamp(min=0.0), t, dims=([0], [0]))
            rw[d, s] = num / (self.w * (-un).clamp(min=0.0) * g).sum()
        return rw

    # --- moments and the conservative Maxwellian ----------------------------------------------------
    def moments_of(self, fs):
        Q = torch.zeros(self.npts, 5, dtype=torch.float64, device=self.dev)
        for f, b in zip(fs, self.blocks):
            v = self.v[b]
            psi = torch.stack([torch.ones_like(v[:, 0]), v[:, 0], v[:, 1], v[:, 2], 0.5 * (v * v).sum(1)], 1)
            Q += f.reshape(f.shape[0], -1).T @ (psi * self.w[b, None])
        return Q

    def state_of(self, Q):
        U = Q[:, 1:4] / Q[:, :1]
        th = (2.0 / self.m) * (Q[:, 4] / Q[:, 0] - 0.5 * (U * U).sum(1))
        return U, th

    def equilibrium(self, Q):
        """Exponential factors per axis [n_x, n_d] of the Maxwellian whose discrete moments are Q, and its
        perturbed state (rho', U', theta')."""
        m, tabs, prim = self.m, [[], [], []], []
        for a in range(0, self.npts, 1 << 16):
            q = Q[a:a + (1 << 16)]
            U, th = self.state_of(q)
            rho = q[:, 0]
            c = [(self.v1[d][None] - U[:, d:d + 1]) / torch.sqrt(th)[:, None] for d in range(m)]
            al = torch.zeros(len(q), m + 2, dtype=torch.float64, device=self.dev)
            al[:, 0] = torch.log(rho / (TWO_PI * th) ** (m / 2))
            al[:, -1] = -0.5
            target = torch.zeros_like(al)
            target[:, 0], target[:, -1] = rho, m * rho
            for _ in range(9):
                s = []
                for d in range(m):
                    e = torch.exp(al[:, 1 + d:2 + d] * c[d] + al[:, -1:] * c[d] ** 2) * self.w1[d]
                    s.append(torch.stack([(e * c[d] ** j).sum(1) for j in range(5)], 1))

                def mom(*pw):
                    r = torch.exp(al[:, 0])
                    for d in range(m):
                        r = r * s[d][:, pw[d]]
                    return r

                unit = [tuple(int(d == e) for e in range(m)) for d in range(m)]
                sq = [tuple(2 * t for t in u) for u in unit]
                basis = [[(0,) * m]] + [[u] for u in unit] + [sq]
                M = torch.stack([sum(mom(*u) for u in basis[i]) for i in range(m + 2)], 1)
                H = torch.stack([torch.stack([sum(mom(*(x + y for x, y in zip(u, t))) for u in basis[i] for t in basis[j])
                                              for j in range(m + 2)], 1) for i in range(m + 2)], 1)
                al = al + torch.linalg.solve(H, (target - M).unsqueeze(2)).squeeze(2)
            for d in range(m):
                e = torch.exp(al[:, 1 + d:2 + d] * c[d] + al[:, -1:] * c[d] ** 2)
                tabs[d].append(e * torch.exp(al[:, :1]) if d == 0 else e)
            if m == 2:
                tabs[2].append(torch.ones(len(q), 1, dtype=torch.float64, device=self.dev))
            tp = -0.5 * th / al[:, -1]
            Up = [U[:, d] + tp / torch.sqrt(th) * al[:, 1 + d] for d in range(m)]
            lnr = al[:, 0] + sum((Up[d] - U[:, d]) ** 2 for d in range(m)) / (2 * tp) + 0.5 * m * torch.log(TWO_PI * tp)
            prim.append(torch.stack([torch.exp(lnr)] + Up + [torch.zeros_like(tp)] * (3 - m) + [tp], 1))
        return [torch.cat(t) for t in tabs], torch.cat(prim)

    def g(self, tabs, b):
        t = [tabs[d][:, self.k[d][b]] for d in range(3)]
        return (t[0] * t[1] * t[2]).T.reshape((-1,) + self.shape)

    def force_poly(self, tabs, Q, F):
        F = torch.tensor(F, dtype=torch.float64, device=self.dev)
        s = [torch.stack([(tabs[d] * self.w1[d] * self.v1[d] ** j).sum(1) for j in range(5)], 1) for d in range(3)]
        unit = [(1, 0, 0), (0, 1, 0), (0, 0, 1)]
        basis = [[(1.0, (0, 0, 0))]] + [[(1.0, u)] for u in unit] + [[(0.5, tuple(2 * t for t in u)) for u in unit]]
        H = torch.stack([torch.stack([sum(x * y * s[0][:, u[0] + t[0]] * s[1][:, u[1] + t[1]] * s[2][:, u[2] + t[2]]
                                          for x, u in basis[i] for y, t in basis[j]) for j in range(5)], 1)
                         for i in range(5)], 1)
        rhs = torch.zeros_like(Q)
        rhs[:, 1:4] = Q[:, :1] * F
        rhs[:, 4] = Q[:, 1:4] @ F
        return torch.linalg.solve(H, rhs.unsqueeze(2)).squeeze(2)

    # --- time stepping ---------------------------------------------------------------------------
    def limit(self, f):
        wq = torch.tensor(self.op["wq"], device=self.dev)
        ax = tuple(range(1 + self.dim, 1 + 2 * self.dim))
        mean = f
        for _ in range(self.dim):
            mean = mean @ wq
        mean = mean.reshape(mean.shape + (1,) * self.dim)
        mn = f.amin(ax, keepdim=True)
        beta = torch.where(mn < 0, (mean / (mean - mn)).abs().clamp(max=1.0), torch.ones_like(mn))
        return torch.where(mn < 0, mean + beta * (f - mean), f)

    def solve(self, P, dt, steps):
        o = self.q["opts"]
        P = torch.tensor(P, device=self.dev)
        fn = []
        for b in self.blocks:
            e = sum((self.v[b, d, None] - P[None, :, 1 + d]) ** 2 for d in range(self.m))
            fn.append((P[:, 0] / (TWO_PI * P[:, 4]) ** (self.m / 2) * torch.exp(-e / (2 * P[:, 4]))).reshape((-1,) + self.shape))
        Q = self.moments_of(fn)
        for _ in range(steps):
            fs = list(fn)
            for st, (an, bb) in enumerate(((0.0, 1.0), (0.75, 0.25), (1.0 / 3.0, 2.0 / 3.0))):
                tabs, _ = self.equilibrium(Q)
                rw = self.wall_density(fs)
                it = 1.0 / self.q["tau"]
                if "mu_ref" in o:
                    _, th = self.state_of(Q)
                    it = (Q[:, 0] * th ** (1.0 - o["mu_omega"]) / o["mu_ref"]).reshape(self.shape)
                beta = self.force_poly(tabs, Q, o["body_force"]) if "body_force" in o else None
                for i, b in enumerate(self.blocks):
                    r = self.residual(fs[i], b, rw)
                    g = self.g(tabs, b)
                    r += it * (g - fs[i])
                    if beta is not None:
                        v = self.v[b]
                        psi = torch.stack([torch.ones_like(v[:, 0]), v[:, 0], v[:, 1], v[:, 2], 0.5 * (v * v).sum(1)], 1)
                        r += g * (psi @ beta.T).reshape(g.shape)
                    r = bb * (fs[i] + dt * r)
                    if an:
                        r += an * fn[i]
                    if o.get("limiter"):
                        r = self.limit(r)
                    fs[i] = r
                Q = self.moments_of(fs)
            fn = fs
        return Q, fn


def exact(c, seed):
    gpu = torch.cuda.is_available()
    dof = _size(c) * c.get("steps", 1)
    if dof > (MAX_WORK if gpu else 4e6):
        return None
    dev = "cuda" if gpu else "cpu"
    if gpu and torch.cuda.mem_get_info()[0] < 24.0 * _size(c) + 12e9:
        return None
    if c["kind"] == "equilibria":
        n = c["n"]
        f = _distributions(c, seed)
        q = dict(p=0, dim=1, ne=(c["points"],), lo=(0.0,), hi=(1.0,), nv=(n,) * 3, vmax=6.0, bc=[[0, 0]] * 3)
        s = _Plain64(q, dev=dev)
        s.blocks = [slice(a, min(n**3, a + 512)) for a in range(0, n**3, 512)]
        Q = s.moments_of([f[:, b].double().T for b in s.blocks])
        return dict(Q=Q, prim=s.equilibrium(Q)[1])
    if c["kind"] == "batch":
        out = []
        for i, m in enumerate(_members(c["members"], c["mesh_seed"])):
            q = _problem(m, (seed, i))
            P = _prim(m, q, _points(q), (seed, i))
            out.append(_Plain64(q, dev=dev).solve(P, _dt(q, P), c["steps"])[0])
        return dict(Q=torch.cat(out))
    q = _problem(c, seed)
    x = _points(q)
    P = _prim(c, q, x, seed)
    bent = c["kind"] in ("curved", "unstructured")
    s = _Plain64(q, x=_curved(q, x) if bent else None, dev=dev)
    Q, f = s.solve(P, _dt(q, P), c["steps"])
    if c["kind"] == "unstructured":
        Q = Q[torch.from_numpy(_relabelled(q["ne"], q["p"])["node_map"]).to(dev)]
    if c["kind"] == "tube":
        return dict(Q=Q.cpu().numpy(), f=torch.cat([t.reshape(len(t), -1) for t in f]).T.contiguous().cpu().numpy())
    return dict(Q=Q)
