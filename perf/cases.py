"""The workloads this framework is timed on, each through its public entry
points as a caller's program uses them.

A case is a plain dict: what is stepped (`kind`), the mesh, the coefficients,
the arithmetic and how many steps one pass takes.  One pass of a stepping case
puts a start state in place (`fs_set_state`), steps (`fs_step`,
`fs_step_picard` or `fs_step_ipcs`) and reads the state back into a device
tensor (`fs_get_state`): a restart from a checkpoint, with no step history.
The handle (mesh, DOF map, step-invariant blocks, multigrid hierarchies,
Krylov workspace) is what a caller keeps between passes.

`exact` is a plain torch restatement in FP64 (quadrature element matrices,
dense LU, Jacobi-CG), for the sizes where that takes seconds.
"""
from __future__ import annotations

import math
from itertools import permutations
from types import SimpleNamespace

import numpy as np
import torch

from paper_2605_25403_gb300 import fs

SQUARE, CHANNEL, CUBE, POLY3 = (fs.FS_PROBLEM_UNSTEADY_BENCH, fs.FS_PROBLEM_CHANNEL,
                                fs.FS_PROBLEM_CUBE, fs.FS_PROBLEM_POLY3)
PREC = {"fp64": fs.FS_PREC_FP64, "fp32": fs.FS_PREC_FP32_REFINE}
FLOW = {"square": SQUARE, "channel": CHANNEL, "cube": CUBE}


def _case(kind, flow, n, prec="fp32", steps=1, nu=1.0, dt=1e-2, jitter=0.0, det=False,
          name=None):
    nx, ny, nz = (tuple(n) + (1, 1))[:3]
    c = dict(kind=kind, flow=flow, nx=nx, ny=ny, nz=nz, prec=prec, steps=steps, nu=nu, dt=dt,
             jitter=jitter, det=det)
    return dict(c, name=name) if name else c


def listed():
    return [
        # the smallest run a user makes: the 128-triangle unit square in FP64,
        # ten Oseen steps; every kernel is far smaller than the chip
        _case("oseen", "square", (8, 8), "fp64", 10, 1.0, 1e-2, 0.1, name="square_8_fp64"),
        # the 2D production run: channel flow from rest, 445,411 unknowns
        _case("oseen", "channel", (512, 96), "fp32", 3, 1e-3, 1e-3, name="channel_512x96"),
        # the same flow at half the resolution in plain FP64
        _case("oseen", "channel", (256, 48), "fp64", 3, 1e-3, 1e-3, name="channel_256x48_fp64"),
        # a small 3D run of odd size on a jittered mesh
        _case("oseen", "cube", (7, 7, 7), "fp32", 2, 1e-2, 5e-3, 0.05, name="cube_7"),
        # the 3D production run: 2.86 million unknowns
        _case("oseen", "cube", (48, 48, 48), "fp32", 2, 1e-2, 5e-3, 0.05, name="cube_48"),
        # a parameter study: 96 independent squares of uneven size and Reynolds
        # number in one problem
        dict(kind="batch", count=96, nmin=16, nmax=128, draw=0, prec="fp32", steps=2, dt=1e-3,
             name="batch_96"),
        # the nonlinear step: Picard iterates of the convection term
        _case("picard", "square", (32, 32), "fp32", 1, 1e-2, 1e-2, name="picard_32"),
        # pressure-correction stepping (FP64 CG), the paper's second scheme
        _case("ipcs", "square", (256, 256), "fp32", 2, 1e-2, 1e-3, name="ipcs_256"),
        # the same scheme with the P3/P2 pair, at a table size of the paper
        _case("p3", "square", (32, 32), "fp64", 2, 1e-2, 1e-3, name="p3_ipcs_32"),
        # assembly alone, with the monolithic system exported to the caller
        _case("assemble", "cube", (24, 24, 24), "fp64", 1, 1e-2, 5e-3, 0.05,
              name="assemble_cube_24"),
        # the operator alone (a caller's own Krylov method), odd size
        _case("apply", "cube", (33, 33, 33), "fp64", 1, 1e-2, 5e-3, 0.05, name="apply_cube_33"),
        # the request loop: a mixed queue of 2D and 3D runs, set up and stepped
        # side by side
        dict(kind="serve", count=10, n2max=128, n3max=16, draw=0, steps=8, dt=1e-3,
             name="serve_10"),
    ]


def _log(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def draw(rng):
    kind = rng.choice(["oseen2", "oseen2", "channel", "channel", "oseen3", "oseen3", "batch",
                       "picard", "ipcs", "p3", "assemble", "apply", "serve"])
    prec = rng.choice(["fp32", "fp32", "fp64"])
    nu = 10 ** rng.uniform(-3, 0)
    jit = rng.choice([0.0, 0.05, 0.1])
    det = rng.random() < 0.25
    if kind == "oseen2":
        n = _log(rng, 8, 300)
        return _case("oseen", "square", (n, max(4, n + rng.randint(-3, 3))), prec,
                     rng.randint(1, 4), nu, rng.choice([1e-2, 1e-3]), jit, det)
    if kind == "channel":
        ny = _log(rng, 6, 96)
        return _case("oseen", "channel", (int(ny * rng.uniform(4, 5.4)), ny), prec,
                     rng.randint(1, 3), 10 ** rng.uniform(-3, -2), 1e-3, 0.0, det)
    if kind == "oseen3":
        n = _log(rng, 5, 40 if prec == "fp32" else 24)
        return _case("oseen", "cube", (n, n, max(4, n + rng.randint(-2, 2))), prec,
                     rng.randint(1, 2), 10 ** rng.uniform(-2, 0), 5e-3, min(jit, 0.05), det)
    if kind == "batch":
        return dict(kind="batch", count=_log(rng, 3, 96), nmin=10, nmax=_log(rng, 24, 128),
                    draw=rng.randint(1, 10 ** 6), prec=prec, steps=rng.randint(1, 2), dt=1e-3)
    if kind == "picard":
        return _case("picard", "square", (_log(rng, 8, 128),) * 2, "fp32", 1, max(nu, 1e-2),
                     1e-2, jit, det)
    if kind == "ipcs":
        n = _log(rng, 12, 256)
        return _case("ipcs", "square", (n, n + rng.randint(0, 5)), prec, rng.randint(1, 3), 1e-2,
                     1e-3, jit)
    if kind == "p3":
        n = _log(rng, 6, 48)
        return _case("p3", "square", (n, n), "fp64", rng.randint(1, 2), 1e-2, 1e-3)
    if kind in ("assemble", "apply"):
        flow = rng.choice(["square", "channel", "cube"])
        n = _log(rng, 5, 32) if flow == "cube" else _log(rng, 10, 300)
        size = (n, n + 1, n) if flow == "cube" else (n, max(5, n // 3))
        return _case(kind, flow, size, prec, 1, 1e-2, 5e-3, 0.0 if flow == "channel" else jit,
                     det)
    return dict(kind="serve", count=rng.randint(3, 16), n2max=_log(rng, 24, 160),
                n3max=rng.randint(8, 16), draw=rng.randint(1, 10 ** 6), steps=rng.randint(3, 10),
                dt=1e-3)


# ---------------------------------------------------------------------------
# Inputs
# ---------------------------------------------------------------------------
def _rand(seed, salt=0):
    return np.random.RandomState((int(seed) * 7919 + salt) % (2 ** 32))


def _box(c):
    """(dim, n, lo, hi, Dirichlet sides, pin, init): the domains of the flows."""
    if c["flow"] == "cube":
        return 3, (c["nx"], c["ny"], c["nz"]), (0.0,) * 3, (1.0,) * 3, 0x3F, 1, 0
    if c["flow"] == "channel":
        return 2, (c["nx"], c["ny"]), (0.0,) * 2, (2.2, 0.41), 0x0D, 0, 1
    return 2, (c["nx"], c["ny"]), (0.0,) * 2, (1.0,) * 2, 0x0F, 1, 0


def _draws(c, seed):
    """What a seed changes: viscosity, start time, the mesh's jitter."""
    r = _rand(seed)
    t0 = 0.0 if c["flow"] == "channel" else float(r.uniform(0.2, 1.0))
    return float(c["nu"] * r.uniform(0.8, 1.25)), t0, int(r.randint(1, 2 ** 30))


def _study(c):
    """The (size, Reynolds number) pairs of a batch or a request queue, and for
    a queue whether each is 3D: log-uniform draws."""
    r = _rand(c["draw"], 17)
    out = []
    for _ in range(c["count"]):
        three = c["kind"] == "serve" and r.uniform() < 0.5
        lo, hi = (6, c["n3max"]) if three else (c.get("nmin", 16), c.get("nmax", c.get("n2max")))
        n = int(round(math.exp(r.uniform(math.log(lo), math.log(hi)))))
        out.append((three, n, math.exp(r.uniform(0.0, math.log(2000.0)))))
    return out


class _Handle:
    """A mesh and a problem, released together."""

    def __init__(self, mesh, prob):
        self.mesh, self.prob = mesh, prob

    def __del__(self):
        fs.fs_problem_destroy(self.prob)
        fs.fs_mesh_destroy(self.mesh)


class _Server(fs.Server):
    """A request loop, closed when dropped."""

    def __del__(self):
        self.close()


class _Request:
    """A request as fs.Server.submit takes it."""

    def __init__(self, three, n, nu, dt):
        d = 3 if three else 2
        self.dim, self.n, self.lo, self.hi = d, (n,) * d, (0.0,) * d, (1.0,) * d
        self.jitter, self.seed, self.side_mask = 0.0, 0, 0x3F if three else 0x0F
        self.problem, self.nu, self.dt = (3 if three else 0), nu, dt
        self.pin_p0, self.init, self.wconst = True, "exact", None
        self.ndof = d * (2 * n + 1) ** d + (n + 1) ** d


def prepare(case, seed):
    c, kind = case, case["kind"]
    if kind == "serve":
        r = _rand(seed)
        reqs = [_Request(three, n, float(r.uniform(0.8, 1.25)) / re, c["dt"])
                for three, n, re in _study(c)]
        return SimpleNamespace(kind=kind, server=_Server(20 << 30, 8), reqs=reqs,
                               steps=c["steps"])
    if kind == "batch":
        r = _rand(seed)
        t0 = float(r.uniform(0.2, 1.0))
        study = _study(c)
        mesh = fs.fs_mesh_create_batch([(2, (n, n), (0.0, 0.0), (1.0, 1.0), 0.0, 0, 0x0F)
                                        for _, n, _ in study])
        prob = fs.fs_problem_create_batch(mesh, [dict(
            problem=SQUARE, nu=float(r.uniform(0.8, 1.25)) / re, dt=c["dt"], t0=t0,
            precision=PREC[c["prec"]]) for _, _, re in study])
    else:
        nu, t0, mseed = _draws(c, seed)
        dim, n, lo, hi, sides, pin, init = _box(c)
        mesh = fs.fs_mesh_create(dim, n, lo, hi, c["jitter"], mseed, sides)
        if kind == "p3":
            prob = fs.fs_problem_create_p3(mesh, FLOW[c["flow"]], nu, c["dt"], t0, pin, init)
        else:
            prob = fs.fs_problem_create(mesh, FLOW[c["flow"]], nu, c["dt"], t0, PREC[c["prec"]],
                                        pin, init, deterministic=c["det"])
    s = SimpleNamespace(kind=kind, steps=c["steps"], h=_Handle(mesh, prob), prob=prob, t0=t0)
    ndof = fs.fs_problem_sizes(prob)[2]
    s.x0 = torch.empty(ndof, dtype=torch.float64, device="cuda")
    fs.fs_get_state(prob, s.x0)
    s.out = torch.empty_like(s.x0)
    if kind == "assemble":
        s.t1 = t0 + c["dt"]
        s.val = torch.empty(fs.fs_dof_map(mesh, arrays=False)["nnz"], dtype=torch.float64,
                            device="cuda")
    if kind == "apply":
        fs.fs_assemble_step(prob, t0 + c["dt"])
        s.x0 = torch.from_numpy(_rand(seed, 3).standard_normal(ndof)).cuda()
    return s


def run(s):
    if s.kind == "serve":
        ids = [s.server.submit(q, s.steps, 0.0, keep_state=True) for q in s.reqs]
        left = len(ids)
        while left:
            left -= s.server.progress(0.0)
        s.server.completed()
        return [s.server.take_state(i) for i in ids]
    if s.kind == "assemble":
        fs.fs_assemble_step(s.prob, s.t1, s.val, s.out)
        return {"values": s.val, "rhs": s.out}
    if s.kind == "apply":
        fs.fs_apply_operator(s.prob, s.x0, s.out)
        return s.out
    fs.fs_set_state(s.prob, s.x0, s.t0)
    if s.kind == "picard":
        fs.fs_step_picard(s.prob, s.steps)
    elif s.kind in ("ipcs", "p3"):
        fs.fs_step_ipcs(s.prob, s.steps)
    else:
        fs.fs_step(s.prob, s.steps)
    fs.fs_get_state(s.prob, s.out)
    return s.out


# ---------------------------------------------------------------------------
# Work no implementation can do without
# ---------------------------------------------------------------------------
def _sizes(dim, n):
    nv = math.prod(k + 1 for k in n)
    n2 = math.prod(2 * k + 1 for k in n)
    cells = (2 if dim == 2 else 6) * math.prod(n)
    # entries of the scalar P2 block and of the divergence block, from the
    # mean row lengths of structured meshes
    nnza, nnzb = (11.5 if dim == 2 else 28.3) * n2, (19 if dim == 2 else 62) * nv
    return nv, n2, cells, nnza, nnzb


def _step_work(dim, n, steps):
    """One linear step: its sparse blocks and vectors once, the convection
    integrals of every cell, one application of the operator."""
    nv, n2, cells, nnza, nnzb = _sizes(dim, n)
    by = 8 * nnza + 2 * 8 * dim * nnzb + 2 * 8 * (dim * n2 + nv)
    fl = cells * (1100 if dim == 2 else 3440) + 2 * dim * nnza + 4 * dim * nnzb
    return steps * by, steps * fl


def work(case):
    c, kind = case, case["kind"]
    if kind in ("serve", "batch"):
        w = [_step_work(3 if three else 2, (n,) * (3 if three else 2), c["steps"])
             for three, n, _ in _study(c)]
        return {"bytes": sum(x[0] for x in w), "flops": sum(x[1] for x in w)}
    dim, n = _box(c)[:2]
    nv, n2, cells, nnza, nnzb = _sizes(dim, n)
    ndof = dim * n2 + nv
    if kind == "assemble":
        nnz = dim * (nnza + 2 * nnzb)
        return {"bytes": 8 * nnz + 8 * nnza + 2 * 8 * ndof + 4 * cells * (6 if dim == 2 else 10),
                "flops": cells * (1100 if dim == 2 else 3440)}
    if kind == "apply":
        return {"bytes": 8 * nnza + 2 * 8 * dim * nnzb + 2 * 8 * ndof,
                "flops": 2 * dim * (nnza + 2 * nnzb)}
    by, fl = _step_work(dim, n, c["steps"])
    if kind == "p3":  # P3 rows hold about 2.4 times the entries of P2 rows, on 2.25 times the nodes
        by, fl = 5.4 * by, 5.4 * fl
    return {"bytes": by, "flops": fl}


# ---------------------------------------------------------------------------
# 64-bit values by plain torch
# ---------------------------------------------------------------------------
_EDGES = {2: [(1, 2), (2, 0), (0, 1)], 3: [(0, 1), (0, 2), (0, 3), (1, 2), (1, 3), (2, 3)]}


def _uniform64(seed, keys):
    """SplitMix64 of seed xor key, its 53 high bits in [0, 1)."""
    with np.errstate(over="ignore"):
        z = (keys.astype(np.uint64) ^ np.uint64(seed)) + np.uint64(0x9E3779B97F4A7C15)
        z = (z ^ (z >> np.uint64(30))) * np.uint64(0xBF58476D1CE4E5B9)
        z = (z ^ (z >> np.uint64(27))) * np.uint64(0x94D049BB133111EB)
        z = z ^ (z >> np.uint64(31))
    return (z >> np.uint64(11)).astype(np.float64) * 2.0 ** -53


def _p2_mesh(dim, n, lo, hi, jitter, seed):
    idx = np.indices(tuple(k + 1 for k in n[::-1])).reshape(dim, -1)[::-1]  # x fastest
    v = np.arange(idx.shape[1])
    inner = np.all([(idx[a] > 0) & (idx[a] < n[a]) for a in range(dim)], axis=0)
    xyz = np.empty((len(v), dim))
    for a in range(dim):
        h = (hi[a] - lo[a]) / n[a]
        move = jitter * h * (2.0 * _uniform64(seed, 3 * v + a) - 1.0)
        xyz[:, a] = lo[a] + idx[a] * h + np.where(inner, move, 0.0)
    stride = np.cumprod([1] + [k + 1 for k in n[:-1]])
    corner = np.indices(tuple(n[::-1])).reshape(dim, -1)[::-1]
    base = sum(int(stride[a]) * corner[a] for a in range(dim))
    if dim == 2:
        sx, sy = int(stride[0]), int(stride[1])
        cells = [np.stack([base, base + sx, base + sx + sy], 1),
                 np.stack([base, base + sx + sy, base + sy], 1)]
    else:
        cells = []
        for p in permutations(range(3)):
            w = [base]
            for a in p:
                w.append(w[-1] + int(stride[a]))
            cells.append(np.stack(w, 1))
    cells = torch.from_numpy(np.concatenate(cells))
    nv = len(v)
    ends = torch.stack([cells[:, list(e)] for e in _EDGES[dim]], 1)  # cell x edge x 2
    key = ends.min(2).values * nv + ends.max(2).values
    uniq, inv = torch.unique(key, return_inverse=True)
    c2 = torch.cat([cells, nv + inv], 1)
    xyz = torch.from_numpy(xyz)
    a, b = uniq // nv, uniq % nv
    nodes = torch.cat([xyz, 0.5 * (xyz[a] + xyz[b])])
    # side of a node: a vertex's own sides; an edge's are those both ends lie on
    on = torch.from_numpy(np.stack([f for ax in range(dim)
                                    for f in (idx[ax] == 0, idx[ax] == n[ax])], 1))
    sides = torch.cat([on, on[a] & on[b]])
    return xyz, cells, c2, nodes, sides


def _quadrature(dim):
    """Conical-product Gauss rule, exact to degree 5: barycentric points and
    weights that sum to the reference volume."""
    g, w = np.polynomial.legendre.leggauss(4)
    g, w = 0.5 * (g + 1), 0.5 * w
    pts, wts = [], []
    for i in np.ndindex(*(4,) * dim):
        rest, weight, lam = 1.0, 1.0, []
        for a in range(dim):
            lam.append(rest * g[i[a]])
            weight *= w[i[a]] * (1 - g[i[a]]) ** (dim - 1 - a)
            rest *= 1 - g[i[a]]
        pts.append([1 - sum(lam)] + lam)
        wts.append(weight)
    return np.array(pts), np.array(wts)


class _Plain:
    """Element matrices, blocks and steps of the P2/P1 pair, by quadrature."""

    def __init__(self, c, seed):
        self.c = c
        self.nu, self.t, mseed = _draws(c, seed)
        self.dt, self.flow = c["dt"], c["flow"]
        self.dim, n, lo, hi, mask, self.pin, init = _box(c)
        dim = self.dim
        dev = self.dev = "cuda" if torch.cuda.is_available() else "cpu"
        xyz, cells, c2, nodes, sides = _p2_mesh(dim, n, lo, hi, c["jitter"], mseed)
        self.nodes, self.c2, self.cells = nodes.to(dev), c2.to(dev), cells.to(dev)
        self.nv, self.n2 = len(xyz), len(nodes)
        self.ndof = dim * self.n2 + self.nv
        bits = torch.tensor([bool(mask >> s & 1) for s in range(2 * dim)])
        self.fixed = (sides & bits).any(1).to(dev)
        X = xyz.to(dev)[self.cells]
        J = (X[:, 1:] - X[:, :1]).transpose(1, 2)  # columns: edge vectors
        self.det = torch.linalg.det(J).abs()
        gl = torch.linalg.inv(J)  # rows: gradients of lambda_1..d
        self.gl = torch.cat([-gl.sum(1, keepdim=True), gl], 1)  # cell x (d+1) x d
        lam, w = _quadrature(dim)
        nb = dim + 1
        phi = np.concatenate([lam * (2 * lam - 1)] +
                             [4 * lam[:, [a]] * lam[:, [b]] for a, b in _EDGES[dim]], 1)
        dphi = np.zeros(phi.shape + (nb,))  # d phi_j / d lambda_r
        for i in range(nb):
            dphi[:, i, i] = 4 * lam[:, i] - 1
        for k, (a, b) in enumerate(_EDGES[dim]):
            dphi[:, nb + k, a], dphi[:, nb + k, b] = 4 * lam[:, b], 4 * lam[:, a]
        T = lambda v: torch.from_numpy(np.ascontiguousarray(v)).to(dev)  # noqa: E731
        phi, dphi, w, lam = T(phi), T(dphi), T(w), T(lam)
        self.tM = torch.einsum("q,qi,qj->ij", w, phi, phi)
        self.tK = torch.einsum("q,qir,qjs->ijrs", w, dphi, dphi)
        self.tN = torch.einsum("q,qi,qk,qjr->kijr", w, phi, phi, dphi)
        self.tB = torch.einsum("q,qv,qjr->vjr", w, lam, dphi)
        self.x = torch.zeros(self.ndof, dtype=torch.float64, device=dev)
        u, p = self.fields(self.t)
        for k in range(dim):
            self.x[k * self.n2:(k + 1) * self.n2] = torch.where(
                self.fixed, u[:, k], torch.zeros_like(u[:, k])) if init else u[:, k]
        self.x[dim * self.n2:] = p[:self.nv]

    # the manufactured solutions: u, p at the P2 nodes, and the load
    # f = u_t - nu lap u + (u . grad) u + grad p by differentiation
    def _up(self, X, t):
        pi, sin, cos = math.pi, torch.sin, torch.cos
        s = torch.sin(t)
        x, y = X[:, 0], X[:, 1]
        if self.flow == "square":
            u = [2 * pi * s * sin(pi * x) ** 2 * sin(pi * y) * cos(pi * y),
                 -2 * pi * s * sin(pi * x) * cos(pi * x) * sin(pi * y) ** 2]
            return u, 20 * s * (x * x * y - 1 / 6)
        if self.flow == "channel":
            H, U = 0.41, 1.5
            return ([4 * U * y * (H - y) / H ** 2 + 0 * s, 0 * x * s],
                    8 * self.nu * U * (2.2 - x) / H ** 2 + 0 * s)
        z = X[:, 2]
        g = [sin(pi * v) ** 2 for v in (x, y, z)]
        d = [pi * sin(2 * pi * v) for v in (x, y, z)]
        D = [d[0] * g[1] * g[2], g[0] * d[1] * g[2], g[0] * g[1] * d[2]]
        return [s * (D[(i + 1) % 3] - D[(i + 2) % 3]) for i in range(3)], \
            s * (x * x * y * z - 1 / 12)

    def fields(self, t):
        tt = torch.tensor(float(t), dtype=torch.float64, device=self.dev)
        u, p = self._up(self.nodes, tt)
        return torch.stack(u, 1), p

    def load(self, t):
        if self.flow == "channel":
            return torch.zeros(self.n2, 2, dtype=torch.float64, device=self.dev)
        X = self.nodes.clone().requires_grad_(True)
        t = torch.full((self.n2,), float(t), dtype=torch.float64, device=self.dev,
                       requires_grad=True)
        u, p = self._up(X, t)
        grad = lambda f, v: torch.autograd.grad(f.sum(), v, create_graph=True)[0]  # noqa: E731
        gp = grad(p, X)
        out = []
        for k, uk in enumerate(u):
            gu = grad(uk, X)
            lap = sum(grad(gu[:, a], X)[:, a] for a in range(self.dim))
            conv = sum(u[a] * gu[:, a] for a in range(self.dim))
            out.append(grad(uk, t) - self.nu * lap + conv + gp[:, k])
        return torch.stack(out, 1).detach()

    # element matrices
    def _scalar(self, w):
        """(M, K, N(w)) of every cell; w: n2 x dim nodal convecting field."""
        M = self.det[:, None, None] * self.tM
        G = torch.einsum("era,esa->ers", self.gl, self.gl)
        K = torch.einsum("e,ers,ijrs->eij", self.det, G, self.tK)
        cw = torch.einsum("eka,era->ekr", w[self.c2], self.gl)
        return M, K, torch.einsum("e,ekr,kijr->eij", self.det, cw, self.tN)

    def _div(self):
        return torch.einsum("e,era,vjr->eavj", self.det, self.gl, self.tB)

    def _sum(self, E, rows, cols, shape):
        i = rows[:, :, None].expand(E.shape).reshape(-1)
        j = cols[:, None, :].expand(E.shape).reshape(-1)
        return torch.sparse_coo_tensor(torch.stack([i, j]), E.reshape(-1), shape).coalesce()

    def velocity(self):
        return self.x[:self.dim * self.n2].view(self.dim, self.n2).t().contiguous()

    def system(self, t1, w, u_old):
        """The step's monolithic matrix as sorted entries with every position of
        the fixed pattern, and its right-hand side."""
        dim, n2, nv = self.dim, self.n2, self.nv
        M, K, N = self._scalar(w)
        A = M / self.dt + self.nu * K + N
        B = self._div()
        off = dim * n2
        free = (~self.fixed).to(torch.float64)
        A = A * free[self.c2][:, :, None]
        pin = torch.ones(nv, dtype=torch.float64, device=self.dev)
        if self.pin:
            pin[0] = 0.0
        ent = []
        add = lambda r, c, v: ent.append((r.reshape(-1) * self.ndof + c.reshape(-1),  # noqa: E731
                                          v.reshape(-1)))
        for k in range(dim):
            r = (self.c2 + k * n2)[:, :, None]
            cells = self.cells
            add(r.expand(A.shape), (self.c2 + k * n2)[:, None, :].expand(A.shape), A)
            Bk = B[:, k]  # cell x vertex x node
            Bt = Bk.transpose(1, 2)
            add(r.expand(Bt.shape), (cells + off)[:, None, :].expand(Bt.shape),
                -Bt * free[self.c2][:, :, None])
            add((cells + off)[:, :, None].expand(Bk.shape),
                (self.c2 + k * n2)[:, None, :].expand(Bk.shape),
                Bk * pin[cells][:, :, None])
        d = torch.arange(self.ndof, device=self.dev)
        one = torch.cat([self.fixed.to(torch.float64).repeat(dim), 1.0 - pin])
        add(d, d, one)
        key = torch.cat([e[0] for e in ent])
        val = torch.cat([e[1] for e in ent])
        del ent
        uniq, inv = torch.unique(key, return_inverse=True)
        vals = torch.zeros(len(uniq), dtype=torch.float64, device=self.dev)
        vals.index_add_(0, inv, val)
        F = u_old / self.dt + self.load(t1)
        u1, p1 = self.fields(t1)
        Ms = self._sum(M, self.c2, self.c2, (n2, n2))
        b = torch.where(self.fixed[:, None], u1, torch.sparse.mm(Ms, F))
        bp = torch.zeros(nv, dtype=torch.float64, device=self.dev)
        if self.pin:
            bp[0] = p1[0]
        return uniq, vals, torch.cat([b.t().reshape(-1), bp])

    def _solve(self, key, val, b):
        K = torch.zeros(self.ndof, self.ndof, dtype=torch.float64, device=self.dev)
        K.view(-1)[key] = val
        lu, piv = torch.linalg.lu_factor(K)
        x = torch.linalg.lu_solve(lu, piv, b[:, None])
        for _ in range(2):
            x = x + torch.linalg.lu_solve(lu, piv, b[:, None] - K @ x)
        return x[:, 0]

    def oseen_step(self):
        u = self.velocity()
        self.x = self._solve(*self.system(self.t + self.dt, u, u))
        self.t += self.dt

    def picard_step(self, tol=1e-10, most=50):
        u_old = w = self.velocity()
        for _ in range(most):
            self.x = self._solve(*self.system(self.t + self.dt, w, u_old))
            new = self.velocity()
            done = (new - w).norm() <= tol * max(1.0, float(new.norm()))
            w = new
            if done:
                break
        self.t += self.dt

    def _cg(self, A, b, x, hold):
        """Jacobi-CG on the free unknowns (those of `hold` keep x's values), with
        two restarts from the true residual."""
        d = torch.zeros(len(b), dtype=torch.float64, device=self.dev)
        i = A.indices()
        on = i[0] == i[1]
        d[i[0][on]] = A.values()[on]
        A = A.to_sparse_csr()
        free = ~hold
        goal = 1e-15 * float(b[free].norm())
        for _ in range(3):
            r = torch.where(free, b - A @ x, torch.zeros_like(b))
            z = r / d
            p, rz = z.clone(), r @ z
            for k in range(6000):
                if k % 32 == 0 and float(r.norm()) <= goal:
                    break
                q = torch.where(free, A @ p, torch.zeros_like(p))
                a = rz / (p @ q)
                x = x + a * p
                r = r - a * q
                z = r / d
                new = r @ z
                p = z + (new / rz) * p
                rz = new
        return x

    def ipcs_step(self):
        dim, n2, nv, t1 = self.dim, self.n2, self.nv, self.t + self.dt
        u, p = self.velocity(), self.x[dim * n2:]
        M, K, N = self._scalar(u)
        B = self._div()
        size = (n2, n2)
        Ms = self._sum(M, self.c2, self.c2, size)
        A0 = self._sum(M / self.dt + self.nu * K, self.c2, self.c2, size)
        Ns = self._sum(N, self.c2, self.c2, size)
        Bs = [self._sum(B[:, k], self.cells, self.c2, (nv, n2)) for k in range(dim)]
        GG = torch.einsum("era,esa->ers", self.gl, self.gl)
        Kp = self._sum(GG * (self.det / math.factorial(dim))[:, None, None], self.cells,
                       self.cells, (nv, nv))
        u1, p1 = self.fields(t1)
        rhs = torch.sparse.mm(Ms, u / self.dt + self.load(t1)) - torch.sparse.mm(Ns, u)
        fixed = self.fixed
        us = torch.empty_like(u)
        for k in range(dim):
            r = rhs[:, k] + torch.mv(Bs[k].t(), p)
            us[:, k] = self._cg(A0, r, torch.where(fixed, u1[:, k], u[:, k]), fixed)
        r = -sum(torch.mv(Bs[k], us[:, k]) for k in range(dim)) / self.dt
        pinned = torch.zeros(nv, dtype=torch.bool, device=self.dev)
        pinned[0] = True
        dp = torch.zeros(nv, dtype=torch.float64, device=self.dev)
        dp[0] = p1[0] - p[0]
        dp = self._cg(Kp, r, dp, pinned)
        out = torch.empty_like(u)
        for k in range(dim):
            r = torch.mv(Ms, us[:, k]) + self.dt * torch.mv(Bs[k].t(), dp)
            out[:, k] = self._cg(Ms, r, torch.where(fixed, u1[:, k], us[:, k]), fixed)
        self.x = torch.cat([out.t().reshape(-1), p + dp])
        self.t = t1


def exact(case, seed):
    c, kind = case, case["kind"]
    if kind in ("serve", "batch", "p3"):
        return None
    dim, n = _box(c)[:2]
    nv, n2, cells, _, _ = _sizes(dim, n)
    ndof = dim * n2 + nv
    if kind in ("oseen", "picard") and ndof * max(1, c["steps"] if kind == "oseen" else 4) > 45000:
        return None  # dense solves would take too long
    if kind in ("assemble", "apply") and cells > 250000:
        return None
    P = _Plain(c, seed)
    if kind in ("assemble", "apply"):
        u = P.velocity()
        key, val, b = P.system(P.t + P.dt, u, u)
        if kind == "assemble":
            return {"values": val, "rhs": b}
        x = torch.from_numpy(_rand(seed, 3).standard_normal(ndof)).to(P.dev)
        y = torch.zeros_like(x)
        y.index_add_(0, key // P.ndof, val * x[key % P.ndof])
        return y
    for _ in range(c["steps"]):
        {"oseen": P.oseen_step, "picard": P.picard_step, "ipcs": P.ipcs_step}[kind]()
    return P.x
