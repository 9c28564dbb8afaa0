"""Workloads whose speed is measured: what a program does with this library.

A pass sets an initial field W (FP64, on the device), advances it by some
steps S(dt) and copies the kinetic state f out (and, for FP64 contexts, W):
the life of one chunk of a simulation, from kin_set_state to kin_get_kinetic.
The contexts, batches and output buffers are made once, in prepare().

The sizes are those of the configurations, tests and benchmark of this
repository (256^2 and 128^3 meshes, degrees 1..3, 8..32-cell subdomains, K = 3
iterations, the 64^2..512^2 batch mix, 32^3 x 6 tetrahedra) and ragged ones
around them.  The initial data are the recipes of workloads/__init__.py
(vortices, density waves, plane waves, sines), sampled on the device.

exact() repeats a pass in FP64 torch operations: the K-th iterate of the
subdomain iteration, Crank-Nicolson extrapolation and over-relaxation.
"""
import functools
import math
import random

import numpy as np
import torch

import paper_2212_11010_gb300 as kin

GLL = {1: ((0.0, 1.0), (0.5, 0.5)),
       2: ((0.0, 0.5, 1.0), (1 / 6, 2 / 3, 1 / 6)),
       3: ((0.0, 0.5 - 0.5 / math.sqrt(5.0), 0.5 + 0.5 / math.sqrt(5.0), 1.0), (1 / 12, 5 / 12, 5 / 12, 1 / 12))}
SYSTEM = {"advection": kin.KIN_ADVECTION, "euler": kin.KIN_EULER, "maxwell": kin.KIN_MAXWELL}
DIAGONALS = ((1, 1, 1), (1, -1, -1), (-1, 1, -1), (-1, -1, 1))   # D3Q4
GAMMA = 1.4
DEV = "cuda"


def grid(name, system, dim, cells, tiles, degree, dtype, steps, velset="axis", iters=3, omega=2.0, sigma=0.0,
         inflow=0, dt_mult=5.0):
    """A problem on a Cartesian box; cells and tiles: extents per axis."""
    c = {"kind": "grid", "system": system, "dim": dim, "degree": degree, "dtype": dtype, "steps": steps,
         "velset": velset, "iters": iters, "omega": omega, "sigma": sigma, "inflow": inflow, "dt_mult": dt_mult}
    for a in range(dim):
        c["n%d" % a] = cells[a]
        c["t%d" % a] = tiles[a]
    return dict(c, name=name) if name else c


def tet(name, system, n, tiles, velset, dtype, steps, iters=3, omega=2.0, sigma=0.0):
    """A problem on a box of n^3 cubes cut into six tetrahedra each."""
    c = {"kind": "tet", "system": system, "n0": n, "t0": tiles, "velset": velset, "dtype": dtype, "steps": steps,
         "iters": iters, "omega": omega, "sigma": sigma, "dt_mult": 5.0}
    return dict(c, name=name) if name else c


def batch(name, count, mix, steps, largest=512):
    """count uneven 2D Euler problems (64^2..largest^2, degrees 1..3) of the mix 'mix', stepped together."""
    c = {"kind": "batch", "count": count, "mix": mix, "steps": steps, "largest": largest}
    return dict(c, name=name) if name else c


def listed():
    return [
        # the smallest problem: a scalar 1D run of 100 steps, where launches and latency count
        grid("advection1d 256 f64", "advection", 1, (256,), (4,), 1, "f64", 100),
        # one ordinary 2D flow problem in single precision, the state within L2
        grid("vortex2d 256 p2", "euler", 2, (256, 256), (8, 8), 2, "f32", 50),
        # a mesh whose subdomains (25 cells) fit no power of two, with free-stream boundaries and damping
        grid("vortex2d 225x175 p2 inflow", "euler", 2, (225, 175), (9, 7), 2, "f32", 25, omega=1.8, inflow=1),
        # the same flow for a user who needs double precision
        grid("vortex2d 256 p2 f64", "euler", 2, (256, 256), (8, 8), 2, "f64", 10),
        # a large 3D flow: 2 GB of state
        grid("densitywave3d 128 p1", "euler", 3, (128,) * 3, (16,) * 3, 1, "f32", 20),
        # 3D flow at the next degree on a mid-size mesh
        grid("densitywave3d 48 p2", "euler", 3, (48,) * 3, (6,) * 3, 2, "f32", 15),
        # large electromagnetic problem with a conducting medium
        grid("maxwell3d 128 p1", "maxwell", 3, (128,) * 3, (16,) * 3, 1, "f32", 20, sigma=1.0),
        # electromagnetics in double precision
        grid("maxwell3d 48 p1 f64", "maxwell", 3, (48,) * 3, (6,) * 3, 1, "f64", 8, sigma=1.0),
        # serving: uneven problems of all degrees advanced together
        batch("batch of 24", 24, 0, 20),
        # the minimal (d + 1) velocity sets, whose sweeps are wavefronts
        grid("vortex2d D2Q3 256 p2", "euler", 2, (256, 256), (8, 8), 2, "f32", 20, velset="simplex"),
        grid("densitywave3d D3Q4 128 p1", "euler", 3, (128,) * 3, (16,) * 3, 1, "f32", 12, velset="simplex"),
        # unstructured cells: a tetrahedral mesh swept in levels
        tet("densitywave tetrahedra 32", "euler", 32, 4, "simplex", "f32", 15),
    ]


def _log(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def _extent(rng, common, lo, hi):
    return common if rng.random() < 0.5 else rng.randint(lo, hi)


def draw(rng):
    family = rng.choice(["adv1d", "flow2d", "flow2d", "flow2d f64", "flow3d", "maxwell3d", "batch", "d2q3", "d3q4",
                         "tet"])
    omega = rng.choice([2.0, 2.0, 1.8])
    iters = rng.choice([3, 3, 2])
    mult = round(rng.uniform(2.0, 8.0), 2)
    degree = rng.randint(1, 3)
    inflow = int(rng.random() < 0.25)
    if family == "adv1d":
        t = rng.choice([1, 2, 4, 8])
        return grid(None, "advection", 1, (t * _log(rng, 16, 1024),), (t,), degree, rng.choice(["f64", "f32"]),
                    rng.randint(20, 100), iters=iters, omega=omega, inflow=inflow, dt_mult=mult)
    if family.startswith("flow2d"):
        dt = "f64" if family.endswith("f64") else "f32"
        most = (512 if dt == "f32" else 256) * 3 // (degree + 1)
        L = [_extent(rng, 32, 7, 40) for _ in range(2)]
        t = [min(_log(rng, 1, 16), max(1, most // x)) for x in L]
        return grid(None, "euler", 2, (L[0] * t[0], L[1] * t[1]), t, degree, dt, rng.randint(*((10, 50) if dt == "f32" else (4, 12))),
                    iters=iters, omega=omega, inflow=inflow, dt_mult=mult)
    if family in ("flow3d", "maxwell3d"):
        dt = rng.choice(["f32", "f32", "f64"])
        p = rng.choice([1, 1, 2, 3])
        most = {1: 112, 2: 56, 3: 40}[p] // (2 if dt == "f64" else 1)
        L = [_extent(rng, 8, 4, 12) for _ in range(3)]
        t = [min(_log(rng, 2, 14), max(1, most // x)) for x in L]
        return grid(None, "euler" if family == "flow3d" else "maxwell", 3, [x * y for x, y in zip(L, t)], t, p, dt,
                    rng.randint(*((5, 20) if dt == "f32" else (3, 8))), iters=iters, omega=omega,
                    sigma=rng.choice([0.0, 1.0]), inflow=inflow, dt_mult=mult)
    if family == "batch":
        return batch(None, rng.randint(3, 24), rng.randint(1, 10 ** 6), rng.randint(8, 20), rng.choice([256, 512]))
    if family == "d2q3":
        L = [_extent(rng, 32, 8, 40) for _ in range(2)]
        t = [_log(rng, 2, 384 // x) for x in L]
        return grid(None, "euler", 2, (L[0] * t[0], L[1] * t[1]), t, degree, "f32", rng.randint(5, 20), velset="simplex",
                    iters=iters, omega=omega, dt_mult=mult)
    if family == "d3q4":
        p = rng.choice([1, 1, 2])
        L = [_extent(rng, 8, 4, 12) for _ in range(3)]
        t = [_log(rng, 2, (96 if p == 1 else 48) // x) for x in L]
        return grid(None, "euler", 3, [x * y for x, y in zip(L, t)], t, p, "f32", rng.randint(4, 12), velset="simplex",
                    iters=iters, omega=omega, dt_mult=mult)
    t = rng.choice([1, 2, 3, 4])
    n = t * rng.randint(3, 32 // t if t > 1 else 16)
    return tet(None, rng.choice(["euler", "euler", "maxwell", "advection"]), n, t, rng.choice(["simplex", "axis"]),
               rng.choice(["f32", "f32", "f64"]), rng.randint(4, 15), iters=iters, omega=omega,
               sigma=rng.choice([0.0, 1.0]))


# ---------------------------------------------------------------------------
# problems
# ---------------------------------------------------------------------------

class Problem:
    """One problem: geometry, model and initial field (m, nodes), sampled on the device from the seed."""

    def __init__(self, case, seed):
        self.case, self.dim, self.degree = case, case.get("dim", 3), case.get("degree", 1)
        self.system, self.iters, self.steps = case["system"], case["iters"], case["steps"]
        self.omega, self.sigma, self.inflow = case["omega"], case.get("sigma", 0.0), case.get("inflow", 0)
        self.simplex = case["velset"] == "simplex"
        self.m = {"advection": 1, "euler": self.dim + 2, "maxwell": 6}[self.system]
        self.nvel = self.dim + 1 if self.simplex else 2 * self.dim
        self.prec = kin.KIN_FP64 if case["dtype"] == "f64" else kin.KIN_FP32
        self.dtype = torch.float64 if case["dtype"] == "f64" else torch.float32
        self.mesh = None
        if case["kind"] == "tet":
            self.mesh = tet_mesh(case["n0"])
            self.n, self.tiles = (case["n0"],) * 3, (case["t0"],) * 3
            x = self.mesh["xyz_dev"]
        else:
            self.n = tuple(case["n%d" % a] for a in range(self.dim))
            self.tiles = tuple(case["t%d" % a] for a in range(self.dim))
        rng = random.Random(seed)
        self.vortex = self.system == "euler" and self.dim == 2 and case.get("flow", "vortex") == "vortex"
        self.side = 10.0 if self.vortex else 1.0
        self.h = [self.side / c for c in self.n]
        if self.mesh is None:
            x = self._coords()
        self.W, amax = self._field(x, rng)
        if self.system == "advection":
            self.lam = 2.0
        elif self.system == "maxwell":
            self.lam = 1.5 if self.simplex else 3.3
        else:
            self.lam = ({2: 2.5, 3: 1.5}[self.dim] if self.simplex else 1.1 * self.dim) * amax
        self.adv = (1.0, 0.5, 0.25) if self.mesh is not None else (1.0, 0.0, 0.0)
        if self.mesh is not None:
            # h_min = volume / surface of the (congruent) tetrahedra
            hmin = self.h[0] / 6.0 / (1.0 + math.sqrt(2.0))
            self.dt = case["dt_mult"] * hmin / (self.lam * (math.sqrt(3.0) if self.simplex else 1.0))
        elif self.system == "advection":
            self.dt = 4.0 * self.h[0] / self.lam
        else:
            self.dt = case["dt_mult"] * min(self.h) / ((2 * self.degree + 1) * self.dim * amax)
        # the state on every domain-boundary face of an inflow problem: the free stream, or no field
        self.Wb = {"advection": [1.0], "maxwell": [0.0] * 6,
                   "euler": [1.0] + [1.0] * self.dim + [1.0 / (GAMMA - 1) + 0.5 * self.dim]}[self.system]

    def _coords(self):
        xi = torch.tensor(GLL[self.degree][0], dtype=torch.float64, device=DEV)
        npn, out = self.degree + 1, []
        shape = tuple(self.n[::-1]) + (npn,) * self.dim
        for a in range(self.dim):
            v = (torch.arange(self.n[a], device=DEV, dtype=torch.float64)[:, None] + xi[None, :]) * self.h[a]
            view = [1] * (2 * self.dim)
            view[self.dim - 1 - a], view[2 * self.dim - 1 - a] = self.n[a], npn
            out.append(v.reshape(view).expand(shape).reshape(-1))
        return out

    def _field(self, x, rng):
        if self.system == "advection":
            A, B = rng.uniform(0.5, 1.5), rng.uniform(0.5, 1.5)
            s = x[0] if self.dim == 1 else x[0] + 2 * x[1] - x[2]
            return (A * torch.sin(2 * math.pi * s + rng.uniform(0, 6.28)) + B)[None].contiguous(), 1.0
        if self.system == "maxwell":
            W = torch.zeros((6, x[0].numel()), dtype=torch.float64, device=DEV)
            for a, e, h in ((0, 1, 2), (1, 2, 0), (2, 0, 1)):
                c = rng.uniform(0.5, 1.5) * torch.cos(2 * math.pi * x[a] + rng.uniform(0, 6.28))
                W[e] += c
                W[3 + h] += c
            return W, 1.0
        if self.vortex:
            eps, b = rng.uniform(3.0, 5.0), self.side
            d = [v - rng.uniform(0.0, b) for v in x]
            d = [v - b * torch.round(v / b) for v in d]
            e = torch.exp(0.5 * (1.0 - d[0] ** 2 - d[1] ** 2))
            vel = [1.0 - eps / (2 * math.pi) * e * d[1], 1.0 + eps / (2 * math.pi) * e * d[0]]
            rho = (1.0 - (GAMMA - 1) * eps * eps / (8 * GAMMA * math.pi ** 2) * e * e) ** (1 / (GAMMA - 1))
            pr = rho ** GAMMA
        else:
            rho = 1.0 + 0.2 * torch.sin(2 * math.pi * sum(x) + rng.uniform(0, 6.28))
            vel = [torch.ones_like(rho) for _ in range(self.dim)]
            pr = torch.ones_like(rho)
        c = torch.sqrt(GAMMA * pr / rho)
        amax = max(float((u.abs() + c).max()) for u in vel)
        E = pr / (GAMMA - 1) + 0.5 * rho * sum(u * u for u in vel)
        return torch.stack([rho] + [rho * u for u in vel] + [E]), amax

    def context(self):
        kw = dict(omega=self.omega, gamma=GAMMA, adv=self.adv, sigma=self.sigma, iters=self.iters, precision=self.prec)
        if self.mesh is not None:
            g = self.mesh
            L = self.n[0] // self.tiles[0]
            q = g["cube"] // L
            sub = (q[:, 2] * self.tiles[0] + q[:, 1]) * self.tiles[0] + q[:, 0]
            return kin.TetContext(g["xyz"], g["vid"], g["nbr"], sub, g["wrap"], SYSTEM[self.system],
                                  kin.KIN_D3Q4 if self.simplex else kin.KIN_D3Q6, self.lam, self.dt, **kw)
        vs = {2: kin.KIN_D2Q3, 3: kin.KIN_D3Q4}[self.dim] if self.simplex else None
        ctx = kin.Context(self.dim, self.n, (0.0,) * self.dim, (self.side,) * self.dim, self.degree,
                          SYSTEM[self.system], self.lam, self.dt, tiles=self.tiles, velset=vs,
                          inflow=(self.inflow,) * self.dim, **kw)
        if self.inflow:
            for a in range(self.dim):
                for side in (0, 1):
                    ctx.set_boundary(a, side, self.Wb)
        return ctx

    @property
    def values(self):
        return self.nvel * self.W.numel()


def members(case):
    """The problems of a batch: meshes, degrees and time steps from the mix number, as plain cases."""
    rng = random.Random(case["mix"])
    sizes = [s for s in (64, 128, 256, 512) if s <= case["largest"]]
    out = []
    for _ in range(case["count"]):
        n, p = rng.choice(sizes), rng.randint(1, 3)
        c = grid(None, "euler", 2, (n, n), (n // 32, n // 32), p, "f32", case["steps"],
                 dt_mult=rng.uniform(2.0, 8.0))
        c["flow"] = rng.choice(["vortex", "wave"])
        out.append(c)
    return out


_KUHN = ((0, 1, 2), (0, 2, 1), (1, 0, 2), (1, 2, 0), (2, 0, 1), (2, 1, 0))


@functools.lru_cache(maxsize=8)
def tet_mesh(n):
    """The periodic unit cube as n^3 cubes of six tetrahedra (the mesh of workloads.tet_box)."""
    k, j, i = np.meshgrid(*(np.arange(n),) * 3, indexing="ij")
    base = np.stack([i, j, k], -1).reshape(-1, 1, 1, 3)
    corner = np.zeros((6, 4, 3), dtype=np.int64)
    for q, perm in enumerate(_KUHN):
        for b, a in enumerate(perm):
            corner[q, b + 1:, a] += 1
    ijk = (base + corner[None]).reshape(-1, 4, 3)
    w = ijk % n
    vid = (w[..., 2] * n + w[..., 1]) * n + w[..., 0]
    cells = vid.shape[0]
    other = np.array([[1, 2, 3], [0, 2, 3], [0, 1, 3], [0, 1, 2]])
    face = np.sort(vid[:, other], axis=2).reshape(-1, 3)
    key = (face[:, 0] * n ** 3 + face[:, 1]) * n ** 3 + face[:, 2]
    o = np.argsort(key, kind="stable")
    nbr = np.empty(4 * cells, dtype=np.int64)
    nbr[o[0::2]], nbr[o[1::2]] = o[1::2] // 4, o[0::2] // 4
    nbr = nbr.reshape(cells, 4)
    # a face wraps when its vertices' lattice points differ between the two cells
    wrap = np.zeros((cells, 4), dtype=np.int32)
    for a in range(4):
        b = other[a][0]
        R = nbr[:, a]
        jj = np.argmax(vid[R] == vid[:, b:b + 1], axis=1)
        wrap[:, a] = (ijk[R, jj] != ijk[:, b]).any(axis=1)
    xyz = ijk / n
    dev = torch.from_numpy(xyz.reshape(-1, 3)).to(DEV)
    return {"xyz": xyz, "vid": vid, "nbr": nbr, "wrap": wrap, "cube": ijk[:, 0, :],
            "xyz_dev": [dev[:, a].contiguous() for a in range(3)]}


class State:
    def __init__(self, problems):
        self.problems = problems
        self.contexts = [p.context() for p in problems]
        self.W = [p.W.reshape(-1) for p in problems]
        self.f = [torch.empty(p.values, dtype=p.dtype, device=DEV) for p in problems]
        self.Wout = [torch.empty_like(w) if p.prec == kin.KIN_FP64 else None for p, w in zip(problems, self.W)]
        self.batch = None

    def outputs(self):
        return {"f": self.f, "W": [w for w in self.Wout if w is not None]}


def prepare(case, seed):
    if case["kind"] != "batch":
        return State([Problem(case, seed)])
    s = State([Problem(c, seed * 64 + i) for i, c in enumerate(members(case))])
    for c, w in zip(s.contexts, s.W):
        c.set_state(w)
    s.batch = kin.Batch(s.contexts)
    return s


def run(s):
    for c, w in zip(s.contexts, s.W):
        c.set_state(w)
    steps = s.problems[0].steps
    if s.batch is not None:
        s.batch.step(steps)
    else:
        s.contexts[0].step(steps)
    for c, f, w in zip(s.contexts, s.f, s.Wout):
        kin.kin_get_kinetic(c.ctx, f)
        if w is not None:
            kin.kin_get_state(c.ctx, w)
    return s.outputs()


def work(case):
    total = {"bytes": 0.0, "flops": 0.0}
    for c in (members(case) if case["kind"] == "batch" else [case]):
        dim, p = c.get("dim", 3), c.get("degree", 1)
        m = {"advection": 1, "euler": dim + 2, "maxwell": 6}[c["system"]]
        nvel = dim + 1 if c["velset"] == "simplex" else 2 * dim
        size = 8 if c["dtype"] == "f64" else 4
        if c["kind"] == "tet":
            nodes, per = 24 * c["n0"] ** 3, c["iters"] * (2 * 4 + 8) + 8
        else:
            nodes = math.prod(c["n%d" % a] * (p + 1) for a in range(dim))
            # a line solve per value, or a full cell solve per iterate, then the relaxation
            per = (2 * (p + 1) + 4 if c["velset"] == "axis" else c["iters"] * (2 * (p + 1) ** dim + 8)) + 8
        f = nvel * m * nodes
        # W in, f read and written once per step, f out
        total["bytes"] += 8.0 * m * nodes + 2.0 * size * f * c["steps"] + size * f + (8.0 * m * nodes if size == 8 else 0)
        total["flops"] += float(per) * f * c["steps"]
    return total


# ---------------------------------------------------------------------------
# the same pass in FP64 torch operations
# ---------------------------------------------------------------------------

def _flux(P, W, a):
    if P.system == "advection":
        return P.adv[a] * W
    if P.system == "maxwell":
        Q, j, k = torch.zeros_like(W), (a + 1) % 3, (a + 2) % 3
        Q[k], Q[j], Q[3 + k], Q[3 + j] = -W[3 + j], W[3 + k], W[j], -W[k]
        return Q
    d = P.dim
    u = W[1 + a] / W[0]
    pr = (GAMMA - 1) * (W[1 + d] - 0.5 * (W[1:1 + d] ** 2).sum(0) / W[0])
    Q = W * u
    Q[1 + a] += pr
    Q[1 + d] += pr * u
    return Q


def _velocities(P):
    if not P.simplex:
        return [[(P.lam if k % 2 == 0 else -P.lam) if a == k // 2 else 0.0 for a in range(P.dim)] for k in range(P.nvel)]
    if P.dim == 2:
        return [[P.lam * math.cos(2 * math.pi * k / 3), P.lam * math.sin(2 * math.pi * k / 3) if k else 0.0] for k in range(3)]
    return [[P.lam * s for s in d] for d in DIAGONALS]


def _maxwellian(P, W):
    """M_k(W) for every velocity: (nvel, m, nodes)."""
    Q = [_flux(P, W, a) for a in range(P.dim)]
    if not P.simplex:
        return torch.stack([W / (2 * P.dim) + (1 if k % 2 == 0 else -1) * Q[k // 2] / (2 * P.lam) for k in range(P.nvel)])
    V = torch.tensor(_velocities(P), dtype=torch.float64)
    inv = torch.linalg.inv(torch.cat([torch.ones(1, P.nvel, dtype=torch.float64), V.T])).tolist()
    return torch.stack([inv[k][0] * W + sum(inv[k][1 + a] * Q[a] for a in range(P.dim)) for k in range(P.nvel)])


def _relax(P, f):
    W = f.sum(0)
    if P.system != "maxwell":
        return P.omega * _maxwellian(P, W) + (1 - P.omega) * f
    mu = (1 - 0.5 * P.sigma * P.dt) / (1 + 0.5 * P.sigma * P.dt)
    Wp = torch.cat([mu * W[:3], W[3:]])
    return _maxwellian(P, Wp) + (1 - P.omega) * (f - _maxwellian(P, W))


def _line(p):
    """Weights and Q = diag(w) D of the one-dimensional rule."""
    xi, w = (np.array(v) for v in GLL[p])
    V = np.vander(xi, increasing=True)
    dV = np.zeros_like(V)
    for e in range(1, p + 1):
        dV[:, e] = e * xi ** (e - 1)
    return w, np.diag(w) @ (dV @ np.linalg.inv(V))


def _transport_axis(P, f):
    w, Q = _line(P.degree)
    npn, e0 = P.degree + 1, np.eye(P.degree + 1)[0]
    n, t = (tuple(v) + (1,) * (3 - P.dim) for v in (P.n, P.tiles))
    nd = [npn if a < P.dim else 1 for a in range(3)]
    Mb = _maxwellian(P, torch.tensor(P.Wb, dtype=torch.float64, device=DEV)[:, None]) if P.inflow else None
    for k in range(P.nvel):
        a, back = k // 2, k % 2
        nu = P.lam * 0.5 * P.dt / P.h[a]
        Ai = np.linalg.inv(np.diag(w) + nu * (Q + np.outer(e0, e0)))
        Pm = torch.tensor(Ai @ np.diag(w), device=DEV)
        g = torch.tensor(nu * Ai @ e0, device=DEV)
        # one row per line: (m, transverse..., cells, nodes), reversed for a negative velocity
        X = f[k].reshape(P.m, n[2], n[1], n[0], nd[2], nd[1], nd[0])
        X = X.movedim((3 - a, 6 - a), (-2, -1))
        if back:
            X = X.flip(-2, -1)
        shape = X.shape
        X = X.reshape(P.m, -1, t[a], n[a] // t[a], npn)
        PU = X @ Pm.T
        out, tin = X[..., -1, -1], None
        for it in range(P.iters):
            s = out.roll(1, -1)
            if P.inflow:
                s[..., 0] = Mb[k]
            tin = []
            for c in range(X.shape[-2]):
                tin.append(s)
                s = PU[..., c, -1] + g[-1] * s
            out = s
        X = 2 * (PU + torch.stack(tin, -1)[..., None] * g) - X
        X = X.reshape(shape)
        if back:
            X = X.flip(-2, -1)
        f[k] = X.movedim((-2, -1), (3 - a, 6 - a)).reshape(f[k].shape)
        del X, PU, tin
    return f


def _transport_simplex(P, f):
    w, Q = _line(P.degree)
    npn, d = P.degree + 1, P.dim
    n, t = (tuple(v) + (1,) * (3 - d) for v in (P.n, P.tiles))
    L = [n[a] // t[a] for a in range(3)]
    nn = npn ** d
    node = np.arange(nn)
    jx = [node // npn ** a % npn for a in range(d)]
    wc = np.prod([w[jx[a]] for a in range(d)], axis=0)
    cell = np.arange(L[0] * L[1] * L[2])
    xyz = [cell % L[0], cell // L[0] % L[1], cell // (L[0] * L[1])]
    step = [1, L[0], L[0] * L[1]]
    for k, V in enumerate(_velocities(P)):
        sg = [int(np.sign(v)) for v in V]
        A, faces = np.diag(wc), []
        for a in range(d):
            if sg[a] == 0:
                continue
            nu = abs(V[a]) * 0.5 * P.dt / P.h[a]
            S = sg[a] * Q
            i0 = 0 if sg[a] > 0 else P.degree
            S[i0, i0] += 1.0
            same = np.all([jx[b][:, None] == jx[b][None, :] for b in range(d) if b != a], axis=0)
            wt = np.prod([w[jx[b]] for b in range(d) if b != a], axis=0)
            A = A + nu * same * wt[:, None] * S[jx[a][:, None], jx[a][None, :]]
            at_in, at_out = node[jx[a] == i0], node[jx[a] == P.degree - i0]
            faces.append((a, at_in, at_out, torch.tensor(nu * wt[at_in], device=DEV)))
        Ai = np.linalg.inv(A)
        PW = torch.tensor(Ai @ np.diag(wc), device=DEV)
        Ai = torch.tensor(Ai, device=DEV)
        flip = [1 + (2 - a) for a in range(d) if sg[a] < 0]          # cell axes of (m, cz, cy, cx, node)
        X = f[k].reshape(P.m, n[2], n[1], n[0], nn)
        X = X.flip(flip) if flip else X
        # (cell of the subdomain, m, subdomains z, y, x, node), cells in downwind coordinates
        X = X.reshape(P.m, t[2], L[2], t[1], L[1], t[0], L[0], nn).permute(2, 4, 6, 0, 1, 3, 5, 7)
        shape = X.shape
        X = X.reshape((L[0] * L[1] * L[2],) + tuple(shape[3:])).contiguous()
        PU = X @ PW.T
        depth = sum(xyz[a] for a, *_ in faces)
        prev = X
        for it in range(P.iters):
            cur = torch.empty_like(X)
            for lev in range(int(depth.max()) + 1):
                idx = cell[depth == lev]
                x = PU[torch.from_numpy(idx).to(DEV)]
                for a, at_in, at_out, nuw in faces:
                    tr = torch.empty(x.shape[:-1] + (len(at_out),), dtype=torch.float64, device=DEV)
                    edge = xyz[a][idx] == 0
                    if edge.any():
                        up = torch.from_numpy(idx[edge] + (L[a] - 1) * step[a]).to(DEV)
                        tr[torch.from_numpy(edge).to(DEV)] = prev[up][..., at_out].roll(1, 2 + (2 - a))
                    if not edge.all():
                        up = torch.from_numpy(idx[~edge] - step[a]).to(DEV)
                        tr[torch.from_numpy(~edge).to(DEV)] = cur[up][..., at_out]
                    x = x + (tr * nuw) @ Ai[:, at_in].T
                cur[torch.from_numpy(idx).to(DEV)] = x
            prev = cur
        X = (2 * prev - X).reshape(shape).permute(3, 4, 0, 5, 1, 6, 2, 7).reshape(P.m, n[2], n[1], n[0], nn)
        f[k] = (X.flip(flip) if flip else X).reshape(f[k].shape)
    return f


def _tet_setup(P):
    """Per velocity: A^{-1} M, A^{-1}, inflow factors and the cells of each level (over all subdomains at once)."""
    g = P.mesh
    xyz, nbr = torch.from_numpy(g["xyz"]).to(DEV), torch.from_numpy(g["nbr"]).to(DEV)
    vid = torch.from_numpy(g["vid"]).to(DEV)
    q = torch.from_numpy(g["cube"] // (P.n[0] // P.tiles[0])).to(DEV)
    sub = (q[:, 2] * P.tiles[0] + q[:, 1]) * P.tiles[0] + q[:, 0]
    iface = (sub[nbr] != sub[:, None]) | (torch.from_numpy(g["wrap"]).to(DEV) != 0)
    B = torch.linalg.inv(torch.cat([xyz, torch.ones_like(xyz[..., :1])], -1))    # columns: barycentric coefficients
    grad = B[:, :3, :].transpose(1, 2)                                           # (cells, vertex, xyz)
    vol = torch.linalg.det(xyz[:, 1:] - xyz[:, :1]).abs() / 6
    glen = grad.norm(dim=-1)
    area = 3 * vol[:, None] * glen
    eye = torch.eye(4, dtype=torch.float64, device=DEV)
    Fm = [(1 + eye) * (1 - eye[a])[:, None] * (1 - eye[a])[None, :] / 12 for a in range(4)]
    M = vol[:, None, None] / 20 * (1 + eye)
    # the neighbour's local index of each of this cell's vertices (of the face)
    match = (vid[nbr][:, :, None, :] == vid[:, None, :, None]).to(torch.int8).argmax(-1)    # (cell, face, vertex)
    out = []
    for V in _velocities(P):
        v = torch.tensor(V, dtype=torch.float64, device=DEV)
        vn = -(grad @ v) / glen
        vn = torch.where(vn.abs() <= 1e-12 * v.norm(), torch.zeros_like(vn), vn)
        A = M - 0.5 * P.dt * ((grad @ v) * (vol / 4)[:, None])[:, :, None]
        for a in range(4):
            A = A + 0.5 * P.dt * (vn[:, a].clamp(min=0) * area[:, a])[:, None, None] * Fm[a]
        Ai = torch.linalg.inv(A)
        cin = 0.5 * P.dt * (-vn).clamp(min=0) * area
        up = (vn < 0) & ~iface
        lev = torch.zeros(len(vid), dtype=torch.int64, device=DEV)
        while True:
            new = torch.where(up, lev[nbr] + 1, torch.zeros_like(nbr)).max(1).values
            if bool((new == lev).all()):
                break
            lev = new
        levels = [torch.nonzero(lev == i)[:, 0] for i in range(int(lev.max()) + 1)]
        out.append((Ai @ M, Ai, cin, levels))
    return out, nbr, iface, match, Fm


def _transport_tet(P, f, setup):
    per, nbr, iface, match, Fm = setup
    for k, (PM, Ai, cin, levels) in enumerate(per):
        X = f[k].reshape(P.m, -1, 4)
        PU = torch.einsum("cij,mcj->mci", PM, X)
        prev = X
        for it in range(P.iters):
            cur = torch.empty_like(X)
            for c in levels:
                rhs = 0
                for a in range(4):
                    at = nbr[c, a][None, :, None]
                    g = torch.where(iface[c, a][None, :, None], prev[:, nbr[c, a]], cur[:, nbr[c, a]])
                    g = torch.gather(g, 2, match[c, a][None].expand(P.m, -1, -1))
                    g = torch.where((cin[c, a] > 0)[None, :, None], g, torch.zeros_like(g))
                    rhs = rhs + cin[c, a][None, :, None] * (g @ Fm[a])
                cur[:, c] = PU[:, c] + torch.einsum("cij,mcj->mci", Ai[c], rhs)
            prev = cur
        f[k] = (2 * prev - X).reshape(f[k].shape)
    return f


def _exact_one(P):
    f = _maxwellian(P, P.W)
    setup = _tet_setup(P) if P.mesh is not None else None
    for _ in range(P.steps):
        if setup is not None:
            f = _transport_tet(P, f, setup)
        elif P.simplex:
            f = _transport_simplex(P, f)
        else:
            f = _transport_axis(P, f)
        f = _relax(P, f)
    return f.reshape(-1), (f.sum(0).reshape(-1) if P.prec == kin.KIN_FP64 else None)


def exact(case, seed):
    if case["kind"] == "batch":
        cases = [(c, seed * 64 + i) for i, c in enumerate(members(case))]
    else:
        cases = [(case, seed)]
    got = [_exact_one(Problem(c, s)) for c, s in cases]
    return {"f": [f for f, _ in got], "W": [w for _, w in got if w is not None]}
