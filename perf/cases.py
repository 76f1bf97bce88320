"""The work that a user of this framework has it do, as cases to be timed.

A case is one call (or one solve) through the package's public entry points on
a block-structured mesh: rectangles or boxes of square / cubic coarse cells,
each split into 2 macro-triangles or 6 Kuhn macro-tets, interior coarse
vertices jittered, refined to a level L (n = 2^L micro-edges per macro-edge).

The inputs and the 64-bit results are formed without the package, on the
refined mesh seen as one global lattice: with these coarse meshes the refined
vertices are the points of a (kx n + 1) x (ky n + 1) [x (kz n + 1)] grid, the
micro-edges its 0/1 vectors, and the stiffness matrix a weight per micro-edge.
"""
from __future__ import annotations

import itertools
import math

import numpy as np
import torch

import paper_2305_15116_gb300 as H

DEV = "cuda"
F8 = torch.float64


def listed():
    return [
        # the smallest product in use: two macro-triangles, 16.6k DoFs, where
        # launches and latency count
        {"name": "apply2d_small", "op": "apply", "dtype": "f64", "kx": 1, "ky": 1, "kz": 0, "level": 7},
        # the throughput workload: 32 macro-triangles at level 11, 67M DoFs
        {"name": "apply2d_f64", "op": "apply", "dtype": "f64", "kx": 4, "ky": 4, "kz": 0, "level": 11},
        # the same product on float32 vectors
        {"name": "apply2d_f32", "op": "apply", "dtype": "f32", "kx": 4, "ky": 4, "kz": 0, "level": 11},
        # native float64 arithmetic on a middle-sized mesh with an uneven
        # number of macros
        {"name": "apply2d_ieee", "op": "apply", "dtype": "ieee", "kx": 3, "ky": 5, "kz": 0, "level": 9},
        # a small 3D product: 36 macro-tets at level 4
        {"name": "apply3d_small", "op": "apply", "dtype": "f64", "kx": 1, "ky": 2, "kz": 3, "level": 4},
        # the 3D throughput workload: 384 macro-tets at level 6, 17M DoFs
        {"name": "apply3d_f64", "op": "apply", "dtype": "f64", "kx": 4, "ky": 4, "kz": 4, "level": 6},
        # a 3D product on float32 vectors at a level above the slab kernel's
        {"name": "apply3d_f32", "op": "apply", "dtype": "f32", "kx": 2, "ky": 2, "kz": 3, "level": 7},
        # the vertex + edge (P2) operator: 67M DoFs
        {"name": "p2_f64", "op": "p2", "dtype": "f64", "kx": 4, "ky": 4, "kz": 0, "level": 10},
        # many small independent products in one call
        {"name": "batch2d", "op": "batch", "dtype": "f64", "kx": 3, "ky": 4, "kz": 0, "level": 7, "count": 48},
        # one multigrid V-cycle from zero, as a preconditioner runs it
        {"name": "vcycle2d", "op": "vcycle", "dtype": "f32", "kx": 4, "ky": 4, "kz": 0, "level": 10},
        # whole mixed-precision solves of the size the solve server meets
        {"name": "solve2d", "op": "solve", "dtype": "f64", "kx": 3, "ky": 4, "kz": 0, "level": 8},
        {"name": "solve3d", "op": "solve", "dtype": "f64", "kx": 2, "ky": 2, "kz": 3, "level": 5},
    ]


def _cells(c):
    return 2 * c["kx"] * c["ky"] if c["kz"] == 0 else 6 * c["kx"] * c["ky"] * c["kz"]


def _per_macro(c):
    n = 2 ** c["level"]
    if c["op"] == "p2":
        return (n + 1) * (2 * n + 1)
    return (n + 1) * (n + 2) // 2 if c["kz"] == 0 else (n + 1) * (n + 2) * (n + 3) // 6


def _batch_cases(c):
    """The products of a batch: meshes of 1 x 1 up to kx x ky cells on three levels."""
    return [dict(c, op="apply", kx=1 + i % c["kx"], ky=1 + (i // 2) % c["ky"], level=c["level"] - i % 3)
            for i in range(c["count"])]


def work(case):
    """Inputs read once, outputs written once; multiply-adds of one operator
    product (a cycle or solve: of its products on the finest level)."""
    if case["op"] == "batch":
        w = [work(c) for c in _batch_cases(case)]
        return {k: sum(v[k] for v in w) for k in ("bytes", "flops")}
    slots = _cells(case) * _per_macro(case)
    elem = 4 if case["dtype"] == "f32" else 8
    per = 17 if case["op"] == "p2" else 14 if case["kz"] == 0 else 30
    products = {"vcycle": 6, "solve": 60}.get(case["op"], 1)
    return {"bytes": 2 * elem * slots, "flops": per * slots * products}


def draw(rng):
    """One more case: any operation, 1..5 coarse cells per side (3D 1..4), the
    size spread over the logarithm of what the operation is used for."""
    op = rng.choice(["apply2", "apply2", "apply3", "apply3", "p2", "batch", "vcycle", "solve2", "solve3"])
    d3 = op.endswith("3")
    top = 4 if d3 else 5
    c = {"op": op.rstrip("23") if op != "p2" else "p2", "dtype": "f64",
         "kx": rng.randint(1, top), "ky": rng.randint(1, top), "kz": rng.randint(1, top) if d3 else 0, "level": 0}
    if c["op"] in ("apply", "p2"):
        c["dtype"] = rng.choice(["f64", "f64", "f32", "f32", "ieee"])
    if c["op"] == "vcycle":
        c["dtype"] = "f32"
    if c["op"] == "batch":
        c.update(level=rng.randint(5, 7), count=rng.randint(5, 64))
        return c
    lo, hi = {"apply2": (500, 67e6), "apply3": (500, 25e6), "p2": (500, 67e6), "vcycle": (2e3, 16.8e6),
              "solve2": (2e3, 8e5), "solve3": (2e3, 4.2e5)}[op]
    want = math.exp(rng.uniform(math.log(lo), math.log(hi)))
    best = None
    for level in range(3 if not d3 else 2, 12):  # the level whose size is nearest to the wanted one
        s = _cells(c) * _per_macro(dict(c, level=level))
        if s <= hi * 1.01 and (best is None or abs(math.log(s / want)) < best[0]):
            best = (abs(math.log(s / want)), level)
    c["level"] = best[1] if best else (3 if not d3 else 2)
    return c


# ---- meshes and the global lattice ---------------------------------------------

def _k(c):
    return (c["kx"], c["ky"], c["kz"]) if c["kz"] else (c["kx"], c["ky"])


def _coarse(c, seed):
    """Coordinates [.., dim] on the coarse grid (index order: axis 0 first) and
    the cells as grid points [cells, dim+1, dim]."""
    k = _k(c)
    d = len(k)
    grid = np.stack(np.meshgrid(*[np.arange(m + 1) for m in k], indexing="ij"), axis=-1)
    xy = grid / max(k)
    inner = np.all((grid > 0) & (grid < np.array(k)), axis=-1)
    a = (0.15 if d == 2 else 0.1) / max(k)
    g = np.random.Generator(np.random.PCG64(seed))
    xy = xy + np.where(inner[..., None], g.uniform(-a, a, xy.shape), 0.0)
    cells = []
    for p in itertools.product(*[range(m) for m in reversed(k)]):
        b = np.array(p[::-1])
        if d == 2:  # the right angle first
            e = [b, b + [1, 0], b + [0, 1], b + [1, 1]]
            cells += [[e[1], e[3], e[0]], [e[2], e[0], e[3]]]
        else:  # the path along the axes of a permutation
            for s in itertools.permutations(range(3)):
                t = np.eye(3, dtype=int)[list(s)]
                cells.append([b, b + t[0], b + t[0] + t[1], b + 1])
    return xy, np.array(cells)


def _mesh(c, seed):
    xy, cells = _coarse(c, seed)
    d = xy.shape[-1]
    ids = np.ravel_multi_index(tuple(np.moveaxis(cells, -1, 0)), xy.shape[:-1])
    return H.Mesh(xy.reshape(-1, d), ids)


def _simplex(n, d):
    """Local coordinates of the points of a refined macro in slot order."""
    r = torch.arange(n + 1, device=DEV)
    if d == 2:
        y = torch.repeat_interleave(r, n + 1 - r)
        x = torch.arange(y.numel(), device=DEV) - (y * (n + 1) - y * (y - 1) // 2)
        return [x, y]
    xs, ys, zs = [], [], []
    for z in range(n + 1):
        x, y = _simplex(n - z, 2)
        xs.append(x), ys.append(y), zs.append(torch.full_like(x, z))
    return [torch.cat(xs), torch.cat(ys), torch.cat(zs)]


def _slots(c):
    """Lattice index of every slot, and the lattice's shape; P2: the lattice of
    half micro-edges, whose even points are the vertices."""
    n = 2 ** c["level"]
    k = _k(c)
    d = len(k)
    f = 2 if c["op"] == "p2" else 1
    shape = [f * m * n + 1 for m in k]
    q = _simplex(n, d)
    if f == 2:
        ex, ey = _simplex(n - 1, 2)
        q = [torch.cat([2 * q[0], 2 * ex + 1, 2 * ex, 2 * ex + 1]), torch.cat([2 * q[1], 2 * ey, 2 * ey + 1, 2 * ey + 1])]
    out = []
    for v in _coarse(c, 0)[1]:
        i = 0
        for a in range(d):
            p = int(v[0, a]) * n * f + sum(int(v[j + 1, a] - v[0, a]) * q[j] for j in range(d))
            i = i * shape[a] + p
        out.append(i)
    return torch.cat(out), shape


def _random(shape, seed):
    g = torch.Generator(device=DEV)
    g.manual_seed(seed)
    return torch.rand(math.prod(shape), generator=g, device=DEV, dtype=F8) * 2 - 1


def _rhs(c, seed):
    """Lumped mass times a smooth function plus noise, zero on the boundary, on the lattice."""
    lat = _Lattice(c, seed, c["level"])
    f = torch.ones(lat.shape, device=DEV, dtype=F8)
    for a, m in enumerate(lat.shape):
        s = torch.sin(math.pi * torch.linspace(0, 1, m, device=DEV, dtype=F8))
        f = f * s.reshape([-1 if b == a else 1 for b in range(len(lat.shape))])
    g = torch.Generator(device=DEV)
    g.manual_seed(seed)
    f = f + 0.1 * torch.randn(lat.shape, generator=g, device=DEV, dtype=F8)
    return lat.mass() * f * lat.inner


# ---- the cases ------------------------------------------------------------------

def _input(c, seed):
    """The input vector on the lattice, in the type that the call takes."""
    if c["op"] in ("solve", "vcycle"):
        v = _rhs(c, seed).reshape(-1)
    else:
        shape = [(2 if c["op"] == "p2" else 1) * m * 2 ** c["level"] + 1 for m in _k(c)]
        v = _random(shape, seed)
    return v.float() if c["dtype"] == "f32" else v


def prepare(case, seed):
    if case["op"] == "batch":
        parts = [prepare(c, seed + 1000 * i) for i, c in enumerate(_batch_cases(case))]
        return {"case": case, "mesh": [p["mesh"] for p in parts], "x": [p["x"] for p in parts],
                "y": [p["y"] for p in parts], "level": [p["case"]["level"] for p in parts]}
    mesh = _mesh(case, seed).refine(case["level"])
    if case["op"] in ("solve", "vcycle"):
        mesh.solver_setup(case["level"])
    x = _input(case, seed)[_slots(case)[0]]
    return {"case": case, "mesh": mesh, "x": x, "y": torch.empty_like(x)}


def run(state):
    c, m, x = state["case"], state["mesh"], state["x"]
    if c["op"] == "apply":
        return m.apply(c["level"], x, state["y"], ieee=c["dtype"] == "ieee")
    if c["op"] == "p2":
        return m.p2_apply(c["level"], x, state["y"], ieee=c["dtype"] == "ieee")
    if c["op"] == "batch":
        return H.apply_batch(m, state["level"], x, state["y"])
    u = state["y"].zero_()
    if c["op"] == "vcycle":
        return m.vcycle(c["level"], x, u)
    # the solution; the count of iterations and the last residual, which the
    # rounding of the float32 cycles decides, steer nothing here
    m.solve(c["level"], x, u, rtol=1e-10)
    return u


# ---- 64-bit results ---------------------------------------------------------------

class _Lattice:
    """The P1 stiffness matrix of the refined mesh: a weight per micro-edge."""

    def __init__(self, c, seed, level):
        self.c, k, n = c, _k(c), 2 ** level
        self.d, self.n, self.k = len(k), n, k
        self.shape = [m * n + 1 for m in k]
        self.dirs = [v for v in itertools.product((0, 1), repeat=self.d) if any(v)]
        self.paths = list(itertools.permutations(range(self.d)))
        self.inner = torch.zeros(self.shape, device=DEV, dtype=F8)
        self.inner[tuple(slice(1, -1) for _ in k)] = 1
        xy, cells = _coarse(c, seed)
        # per macro (coarse cell, path): the images of one micro-step along each axis
        self.step = np.empty((*k, len(self.paths), self.d, self.d))
        for b in itertools.product(*[range(m) for m in k]):
            for s, path in enumerate(self.paths):
                p = np.array(b)
                for a in path:
                    q = p + np.eye(self.d, dtype=int)[a]
                    self.step[(*b, s, a)] = (xy[tuple(q)] - xy[tuple(p)]) / n
                    p = q
        self.vol = np.abs(np.linalg.det(self.step)) / math.factorial(self.d)

    def macro(self, path):
        """The flat index (coarse cell, path) of the macro that holds the
        micro-simplex `path` of every lattice cell."""
        r = [torch.arange(m * self.n, device=DEV).reshape([-1 if b == a else 1 for b in range(self.d)])
             for a, m in enumerate(self.k)]
        cell = 0
        for a in range(self.d):
            cell = cell * self.k[a] + r[a] // self.n
        pos = [(r[a] % self.n) * 4 + (3 - path.index(a)) for a in range(self.d)]  # its centroid, scaled
        s = 0
        for i, q in enumerate(self.paths):  # the macro whose path orders the coordinates descending
            inside = True
            for a, b in zip(q, q[1:]):
                inside = (pos[a] > pos[b]) & inside
            s = s + i * inside.long()
        return cell * len(self.paths) + s

    def at(self, start, step=1):
        """The slice of the lattice points at `start` in every cell (`step`: points per cell and axis)."""
        return tuple(slice(int(s), int(s) + step * (m * self.n - 1) + 1, step) for s, m in zip(start, self.k))

    def table(self, t):
        return torch.from_numpy(np.ascontiguousarray(t).reshape(-1)).to(DEV)

    def mass(self):
        out = torch.zeros(self.shape, device=DEV, dtype=F8)
        part = self.table(self.vol / (self.d + 1))
        for path in self.paths:
            w = part[self.macro(path)]
            p = np.zeros(self.d, dtype=int)
            for a in (None, *path):
                if a is not None:
                    p[a] += 1
                out[self.at(p)] += w
        return out

    def grads(self, path):
        """Gradients of the barycentric coordinates of the micro-simplex `path` in every macro."""
        e = self.step[..., list(path), :]  # edges between consecutive vertices
        edges = np.cumsum(e, axis=-2)  # from the first vertex
        g = np.moveaxis(np.linalg.inv(edges), -1, -2)
        return np.concatenate([-g.sum(axis=-2, keepdims=True), g], axis=-2)

    def assemble(self):
        self.w = {v: torch.zeros(self.shape, device=DEV, dtype=F8) for v in self.dirs}
        for path in self.paths:
            g, m = self.grads(path), self.macro(path)
            for i in range(self.d + 1):
                for j in range(i + 1, self.d + 1):
                    v, p = [0] * self.d, [0] * self.d
                    for a in path[:i]:
                        p[a] = 1
                    for a in path[i:j]:
                        v[a] = 1
                    w = -self.vol * (g[..., i, :] * g[..., j, :]).sum(-1)
                    self.w[tuple(v)][self.at(p)] += self.table(w)[m]
        self.diag = torch.zeros(self.shape, device=DEV, dtype=F8)
        for v in self.dirs:
            lo, hi = self.ends(v)
            self.diag[lo] += self.w[v][lo]
            self.diag[hi] += self.w[v][lo]
        self.diag = torch.where(self.inner > 0, self.diag, 1.0)
        return self

    def ends(self, v):
        lo = tuple(slice(0, m - a) for m, a in zip(self.shape, v))
        hi = tuple(slice(a, m) for m, a in zip(self.shape, v))
        return lo, hi

    def apply(self, u):
        y = torch.zeros_like(u)
        for v in self.dirs:
            lo, hi = self.ends(v)
            t = self.w[v][lo] * (u[lo] - u[hi])
            y[lo] += t
            y[hi] -= t
        return torch.where(self.inner > 0, y, u)

    def apply_p2(self, u):
        """On the lattice of half micro-edges, from the quadratic element matrices."""
        nodes = list(itertools.combinations_with_replacement(range(3), 2))
        mid = [(0.5, 0.5, 0.0), (0.0, 0.5, 0.5), (0.5, 0.0, 0.5)]
        y = torch.zeros_like(u)
        for path in self.paths:
            g, m = self.grads(path), self.macro(path)
            vert = [(0, 0), tuple(int(a == path[0]) for a in range(2)), (1, 1)]
            at = [self.at([vert[i][a] + vert[j][a] for a in range(2)], step=2) for i, j in nodes]
            dphi = [[((4 * q[i] - 1) * g[..., i, :] if i == j else 4 * (q[i] * g[..., j, :] + q[j] * g[..., i, :]))
                     for i, j in nodes] for q in mid]
            for a in range(6):
                for b in range(6):
                    kab = sum((dphi[q][a] * dphi[q][b]).sum(-1) for q in range(3)) * self.vol / 3
                    y[at[a]] += self.table(kab)[m] * u[at[b]]
        out = u.clone()
        out[1:-1, 1:-1] = y[1:-1, 1:-1]
        return out


class _Multigrid:
    """V(3,3) with weighted Jacobi, linear prolongation and its transpose, level 0 solved directly."""

    def __init__(self, c, seed):
        self.lv = [_Lattice(c, seed, l).assemble() for l in range(c["level"] + 1)]
        l0 = self.lv[0]
        n0 = math.prod(l0.shape)
        a0 = torch.stack([l0.apply(e.reshape(l0.shape)).reshape(-1) for e in torch.eye(n0, device=DEV, dtype=F8)], 1)
        self.a0 = torch.linalg.inv(a0)

    def sweeps(self, a, u, b):
        for _ in range(3):
            u = u + (2.0 / 3.0) / a.diag * (b - a.apply(u))
        return u

    def cycle(self, l, u, b):
        a = self.lv[l]
        if l == 0:
            return (self.a0 @ b.reshape(-1)).reshape(b.shape)
        ac = self.lv[l - 1]
        u = self.sweeps(a, u, b)
        r = b - a.apply(u)
        two = tuple(slice(0, None, 2) for _ in a.shape)
        rc = r[two].clone()
        for v in a.dirs:
            odd = r[tuple(slice(s, m - s, 2) for s, m in zip(v, a.shape))]
            lo, hi = ac.ends(v)
            rc[lo] += 0.5 * odd
            rc[hi] += 0.5 * odd
        e = self.cycle(l - 1, torch.zeros_like(rc), rc * ac.inner)
        u = u.clone()
        u[two] += e
        for v in a.dirs:
            lo, hi = ac.ends(v)
            u[tuple(slice(s, m - s, 2) for s, m in zip(v, a.shape))] += 0.5 * (e[lo] + e[hi])
        return self.sweeps(a, u, b)


def exact(case, seed):
    if case["op"] == "batch":
        return [exact(c, seed + 1000 * i) for i, c in enumerate(_batch_cases(case))]
    idx, shape = _slots(case)
    x = _input(case, seed).to(F8).reshape(shape)
    if case["op"] == "apply":
        y = _Lattice(case, seed, case["level"]).assemble().apply(x)
    elif case["op"] == "p2":
        y = _Lattice(case, seed, case["level"]).apply_p2(x)
    else:
        mg, l = _Multigrid(case, seed), case["level"]
        y = mg.cycle(l, torch.zeros_like(x), x)
        if case["op"] == "solve":
            low = torch.zeros_like(y)
            for _ in range(30):  # the remainder of every correction is kept
                e = mg.cycle(l, torch.zeros_like(x), x - mg.lv[l].apply(y) - mg.lv[l].apply(low))
                s = y + e
                low, y = low + (e - (s - y)), s
    return y.reshape(-1)[idx]
