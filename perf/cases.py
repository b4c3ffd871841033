"""What a user of the library has it do, as measurable cases.

Every case builds a matrix of a synthetic surface mesh (spheres, ellipsoids,
cubes) and takes one call through the public entry points: a product, a
product from host buffers, a batched product, a Helmholtz product or a GMRES
solve.  Sizes are those of the five workloads of the benchmark and of the
tests: 5,120 to 1,310,720 triangles, interpolation orders 3 and 4 (2 and 5 in
the draws), 1 to 32 right-hand sides, leaves of 16 to 64 triangles.

``exact`` is a second implementation of the whole method in FP64 torch (trees,
bases, coupling, Sauter-Schwab nearfield, the three passes), written from the
method: Börm, "Distributed H²-matrices for boundary element methods",
Section 2, and Sauter & Schwab, "Boundary Element Methods", Section 5.2.
"""
from __future__ import annotations

import functools
import math
import random

import numpy as np
import torch

from paper_2203_05665_gb300 import Batch, H2Matrix, HelmholtzMatrix

ETA = 2.0
QUAD = 3
RTOL = 1e-8


# ------------------------------------------------------------------ the cases
def listed():
    return [
        # the smallest workload: one product of a 5,120-triangle sphere with one vector; launches and latency
        dict(name="sphere4_m3_f64_1rhs", call="product", mesh="ball", level=4, ax=1.0, ay=1.0, az=1.0, order=3,
             leaf=32, prec="f64", nrhs=1),
        # the solve of the same workload: GMRES(30) to 1e-8, 60 to 80 products and their orthogonalisation
        dict(name="solve4_m3_f64_1rhs", call="solve", mesh="ball", level=4, ax=1.0, ay=1.0, az=1.0, order=3, leaf=32,
             prec="f64", nrhs=1),
        # one vector at a time through an accurate matrix (a user's own Krylov method or a field evaluation)
        dict(name="ellipsoid6_m4_f64_1rhs", call="product", mesh="ball", level=6, ax=1.5, ay=1.0, az=0.7, order=4,
             leaf=32, prec="f64", nrhs=1),
        # a mesh whose leaves are ragged (29 and 30 triangles) and an odd block of vectors, default order
        dict(name="cube50_m3_f64_5rhs", call="product", mesh="cube", s=50, order=3, leaf=32, prec="f64", nrhs=5),
        # the solve server's residual products: order 3, 32 slots, FP64 accuracy
        dict(name="sphere6_m3_f64_32rhs", call="product", mesh="ball", level=6, ax=1.0, ay=1.0, az=1.0, order=3,
             leaf=32, prec="f64", nrhs=32),
        # the solve server's inner products: the same in FP32
        dict(name="sphere6_m3_f32_32rhs", call="product", mesh="ball", level=6, ax=1.0, ay=1.0, az=1.0, order=3,
             leaf=32, prec="f32", nrhs=32),
        # the main workload: 327,680 triangles, order 4, a block of 16 vectors, FP64 accuracy
        dict(name="sphere7_m4_f64_16rhs", call="product", mesh="ball", level=7, ax=1.0, ay=1.0, az=1.0, order=4,
             leaf=32, prec="f64", nrhs=16),
        # the same in FP32 (the inner products of mixed-precision solves)
        dict(name="sphere7_m4_f32_16rhs", call="product", mesh="ball", level=7, ax=1.0, ay=1.0, az=1.0, order=4,
             leaf=32, prec="f32", nrhs=16),
        # 1.3 million triangles in 16-bit storage, coupling regenerated in the product
        dict(name="sphere8_m3_bf16_4rhs", call="product", mesh="ball", level=8, ax=1.0, ay=1.0, az=1.0, order=3,
             leaf=32, prec="bf16", nrhs=4),
        # an uneven batch of independent FP32 problems in one call
        dict(name="batch6_f32", call="batch", count=6, mix=1004, prec="f32"),
        # the Helmholtz kernel with a block of complex vectors
        dict(name="helmholtz6_m4_f64_4rhs", call="helmholtz", mesh="ball", level=6, ax=1.0, ay=1.0, az=1.0, order=4,
             leaf=32, prec="f64", nrhs=4, kappa=2.0),
        # a product of pinned host arrays: copy in, product, copy out
        dict(name="host6_m4_f64_16rhs", call="host", mesh="ball", level=6, ax=1.0, ay=1.0, az=1.0, order=4, leaf=32,
             prec="f64", nrhs=16),
    ]


def draw(rng: random.Random):
    """One more case: mostly products, some host calls, batches, Helmholtz products and solves."""
    call = rng.choices(["product", "host", "batch", "helmholtz", "solve"], [12, 1, 1, 2, 1])[0]
    if call == "batch":
        return dict(call="batch", count=rng.randint(2, 6), mix=rng.randrange(1 << 20), prec="f32")
    while True:
        case = dict(call=call)
        axes = [round(rng.uniform(0.5, 2.0), 4) for _ in range(3)]
        if rng.random() < 0.5:
            case.update(mesh="ball", level=rng.choices([4, 5, 6, 7], [2, 3, 3, 1])[0], ax=axes[0], ay=axes[1],
                        az=axes[2])
        else:
            case.update(mesh="cube", s=int(round(math.exp(rng.uniform(math.log(20), math.log(160))))))
        case.update(order=rng.choices([2, 3, 4, 5], [1, 5, 5, 1])[0], leaf=rng.choices([16, 32, 64], [1, 4, 1])[0],
                    prec=rng.choices(["f64", "f32", "bf16", "f16"], [5, 3, 1, 1])[0],
                    nrhs=int(round(math.exp(rng.uniform(0.0, math.log(32))))))
        if call == "helmholtz":
            case.update(kappa=round(rng.uniform(0.5, 2.5), 4), prec=rng.choice(["f64", "f32"]),
                        nrhs=min(case["nrhs"], 16))
        if call == "solve":
            case.update(prec="f64", nrhs=min(case["nrhs"], 4))
        # no larger than the largest listed case, in work and in memory
        n, k = _count(case), case["order"] ** 3
        parts = 2 if call == "helmholtz" else 1
        shape = 2 if case["mesh"] == "cube" else 1    # cubes have more blocks per triangle
        if n * k * k * parts * shape * max(1.0, case["nrhs"] / 16) > 327680 * 4096:
            continue
        if call == "solve" and n > 12000:
            continue
        return case


def _count(case):
    return 20 * 4 ** case["level"] if case["mesh"] == "ball" else 12 * case["s"] ** 2


def _problems(case):
    """The problems of a batch: ellipsoids and cubes of 20k to 130k triangles in turn."""
    rng = random.Random(case["mix"])
    out = []
    for p in range(case["count"]):
        if p % 2 == 0:
            spec = dict(mesh="ball", level=rng.choice([5, 6]), ax=rng.uniform(0.5, 2), ay=rng.uniform(0.5, 2),
                        az=rng.uniform(0.5, 2))
        else:
            spec = dict(mesh="cube", s=rng.randint(41, 104))
        spec.update(order=rng.choice([3, 4]), nrhs=rng.randint(1, 8), leaf=64, prec="f32")
        out.append(spec)
    return out


# ------------------------------------------------------------------ meshes
@functools.lru_cache(maxsize=4)
def _sphere(level):
    """Icosahedron refined `level` times, midpoints moved to the unit sphere."""
    g = (1.0 + 5.0 ** 0.5) / 2.0
    v = np.array([(-1, g, 0), (1, g, 0), (-1, -g, 0), (1, -g, 0), (0, -1, g), (0, 1, g), (0, -1, -g), (0, 1, -g),
                  (g, 0, -1), (g, 0, 1), (-g, 0, -1), (-g, 0, 1)], dtype=np.float64)
    v /= np.linalg.norm(v, axis=1, keepdims=True)
    d = np.linalg.norm(v[:, None] - v[None], axis=2)
    near = (d > 0) & (d < 1.2)
    f = [(a, b, c) for a in range(12) for b in range(a + 1, 12) for c in range(b + 1, 12)
         if near[a, b] and near[b, c] and near[a, c]]
    f = np.array([t if np.linalg.det(v[list(t)]) > 0 else (t[0], t[2], t[1]) for t in f], dtype=np.int64)
    for _ in range(level):
        e = np.concatenate([f[:, [0, 1]], f[:, [1, 2]], f[:, [2, 0]]])
        e.sort(axis=1)
        key, inv = np.unique(e[:, 0] * (1 << 32) + e[:, 1], return_inverse=True)
        mid = v[key >> 32] + v[key & 0xFFFFFFFF]
        mid /= np.sqrt((mid * mid).sum(axis=1, keepdims=True))
        ab, bc, ca = (inv.reshape(3, -1) + len(v))
        a, b, c = f.T
        v = np.concatenate([v, mid])
        f = np.stack([a, ab, ca, b, bc, ab, c, ca, bc, ab, bc, ca], axis=1).reshape(-1, 3)
    return v, f.astype(np.int32)


def _cube(s):
    """The surface of [-1, 1]^3, s x s squares per face, two triangles per square."""
    pts, tri = [], []
    i, j = np.meshgrid(np.arange(s), np.arange(s), indexing="ij")
    i, j = i.ravel(), j.ravel()
    for axis in range(3):
        for side in (0, s):
            corner = []
            for di, dj in ((0, 0), (1, 0), (1, 1), (0, 1)):
                p = np.empty((s * s, 3), dtype=np.int64)
                p[:, axis], p[:, (axis + 1) % 3], p[:, (axis + 2) % 3] = side, i + di, j + dj
                corner.append((p[:, 0] * (s + 1) + p[:, 1]) * (s + 1) + p[:, 2])
            a, b, c, d = corner if side == s else (corner[0], corner[3], corner[2], corner[1])
            tri.append(np.stack([a, b, c, a, c, d], axis=1).reshape(-1, 3))
    key, inv = np.unique(np.concatenate(tri), return_inverse=True)
    pts = np.stack([key // (s + 1) ** 2, key // (s + 1) % (s + 1), key % (s + 1)], axis=1)
    return pts * (2.0 / s) - 1.0, inv.reshape(-1, 3).astype(np.int32)


def _mesh(case):
    if case["mesh"] == "cube":
        return _cube(case["s"])
    v, f = _sphere(case["level"])
    return v * np.array([case["ax"], case["ay"], case["az"]]), f


# ------------------------------------------------------------------ inputs, calls
def _vectors(n, nrhs, seed, complex_=False):
    """(nrhs, n) vectors of doubles, entries uniform in [-1, 1]."""
    rng = np.random.default_rng(seed)
    x = rng.uniform(-1.0, 1.0, (nrhs, n))
    return x + 1j * rng.uniform(-1.0, 1.0, (nrhs, n)) if complex_ else x


def _inputs(case, seed):
    if case["call"] == "batch":
        return [_vectors(_count(p), p["nrhs"], seed * 1000 + i).astype(np.float32)
                for i, p in enumerate(_problems(case))]
    x = _vectors(_count(case), case["nrhs"], seed, case["call"] == "helmholtz")
    if case["call"] in ("product",) and case["prec"] != "f64":
        x = x.astype(np.float32)
    return x


def _matrix(case):
    v, f = _mesh(case)
    if case["call"] == "helmholtz":
        return HelmholtzMatrix(v, f, case["kappa"], leaf_size=case["leaf"], eta=ETA, order=case["order"],
                               prec=case["prec"], quad_order=QUAD)
    return H2Matrix(v, f, leaf_size=case["leaf"], eta=ETA, order=case["order"], prec=case["prec"], quad_order=QUAD)


def prepare(case, seed):
    x = _inputs(case, seed)
    if case["call"] == "batch":
        probs = _problems(case)
        mats = [_matrix(dict(p, call="product")) for p in probs]
        b = Batch(mats, [p["nrhs"] for p in probs])
        xd = torch.from_numpy(np.concatenate([a.ravel() for a in x])).cuda()
        return dict(call="batch", mat=b, x=xd, y=torch.empty_like(xd))
    mat = _matrix(case)
    if case["call"] == "host":
        xh = torch.from_numpy(x).pin_memory()
        return dict(call="host", mat=mat, x=xh.t(), y=torch.empty_like(xh, pin_memory=True).t())
    xd = torch.from_numpy(x).cuda().t()
    return dict(call=case["call"], mat=mat, x=xd, y=torch.empty_like(xd.t()).t())


def run(state):
    m, x, y = state["mat"], state["x"], state["y"]
    if state["call"] == "solve":
        return m.solve(x, rtol=RTOL, restart=30, maxit=2000)[0]
    if state["call"] == "host":
        return m.matvec_host((x, y))
    return m.matvec(x, y)


# ------------------------------------------------------------------ work and tolerance
@functools.lru_cache(maxsize=64)
def _blocks_of(key):
    t = _Tree(*_mesh(dict(key)), dict(key)["leaf"])
    return t.depth, int(len(t.adm[0])), int((t.size_of(t.near[0]) * t.size_of(t.near[1])).sum())


def _structure(case):
    return _blocks_of(tuple(sorted((k, v) for k, v in case.items() if k in ("mesh", "level", "ax", "ay", "az", "s",
                                                                              "leaf"))))


def _product_work(case):
    n, r, k, m = _count(case), case["nrhs"], case["order"] ** 3, case["order"]
    depth, nadm, near = _structure(case)
    clusters = 2 << depth
    half = case["prec"] in ("bf16", "f16")
    e = 8 if case["prec"] == "f64" else 4
    parts = 2 if case["call"] == "helmholtz" else 1
    cols = r * parts
    coupling = 0 if half else e * nadm * k * k
    stored = parts * (coupling + (2 if half else e) * near) + (2 if case["prec"] == "f16" else e) * n * k
    flops = parts * 2 * cols * (nadm * k * k + near) + 2 * cols * 2 * n * k + 2 * cols * 6 * m * k * clusters
    return dict(bytes=stored + 2 * e * n * cols, flops=flops + (12 * nadm * k * k if half else 0))


def work(case):
    if case["call"] == "batch":
        w = [_product_work(dict(p, call="product")) for p in _problems(case)]
        return dict(bytes=sum(a["bytes"] for a in w), flops=sum(a["flops"] for a in w))
    w = _product_work(case)
    if case["call"] == "solve":   # about 75 iterations on these meshes, the basis read twice per iteration
        n, r = _count(case), case["nrhs"]
        return dict(bytes=75 * (w["bytes"] + 16 * 15 * n * r), flops=75 * (w["flops"] + 8 * 15 * n * r))
    return w


def tolerance(case):
    """About four times the error against ``exact`` that was measured over these ranges."""
    if case["call"] == "solve":
        return dict(rel=3e-7)     # a residual of 1e-8 times the condition: 1e-8 to 7e-8 measured
    prec = case["prec"]
    if prec == "f64":
        return dict(rel=6e-13)    # 44 to 48 bits per operation: 1e-14 to 1.6e-13 measured
    if case["call"] == "batch":
        return dict(rel=1.5e-6)   # 3.5e-7 measured: sums of up to 64 x 690 terms on the cubes
    if prec == "f32":
        return dict(rel=1e-6)     # 1.3e-7 to 2.3e-7 measured
    return dict(rel=4e-3)         # 16-bit storage: 7e-4 to 1e-3 measured


# ------------------------------------------------------------------ the method in FP64 torch
def _device():
    return "cuda" if torch.cuda.is_available() else "cpu"


class _Tree:
    """Cluster tree by median bisection of centroids, and the block tree."""

    def __init__(self, vert, tri, leaf):
        dev = _device()
        v = torch.from_numpy(np.ascontiguousarray(vert)).to(dev)
        f = torch.from_numpy(tri.astype(np.int64)).to(dev)
        a, b, c = v[f[:, 0]], v[f[:, 1]], v[f[:, 2]]
        cen = (a + b + c) / torch.full_like(a, 3.0)   # an IEEE division, as the sort keys decide ties
        tlo, thi = torch.minimum(torch.minimum(a, b), c), torch.maximum(torch.maximum(a, b), c)
        n = len(f)
        self.depth = 0
        while -(-n >> self.depth) > leaf:
            self.depth += 1
        order = torch.arange(n, device=dev)
        size = torch.tensor([n], device=dev)
        sizes, los, his = [], [], []
        for level in range(self.depth + 1):
            cid = torch.repeat_interleave(torch.arange(len(size), device=dev), size)

            def bound(x, op, start):
                out = torch.full((len(size), 3), start, dtype=torch.float64, device=dev)
                return out.scatter_reduce(0, cid[:, None].expand(-1, 3), x[order], op)

            sizes.append(size)
            los.append(bound(tlo, "amin", math.inf))
            his.append(bound(thi, "amax", -math.inf))
            if level == self.depth:
                break
            ext = bound(cen, "amax", -math.inf) - bound(cen, "amin", math.inf)
            axis = torch.zeros(len(size), dtype=torch.int64, device=dev)
            best = ext[:, 0].clone()
            for d in (1, 2):    # the longest axis, the lowest on ties
                better = ext[:, d] > best
                axis[better] = d
                best = torch.maximum(best, ext[:, d])
            # triangles by (cluster, coordinate, index): three stable sorts, the last key first
            key = cen[order, axis[cid]] + 0.0
            p = torch.argsort(order, stable=True)
            p = p[torch.argsort(key[p], stable=True)]
            order = order[p[torch.argsort(cid[p], stable=True)]]
            size = torch.stack([size // 2, size - size // 2], dim=1).reshape(-1)
        self.order, self.leaf_id, self.leaf_size = order, cid, size
        self.sizes, self.lo, self.hi = sizes, torch.cat(los), torch.cat(his)
        self._block_tree()

    def size_of(self, c):
        return torch.cat(self.sizes)[c]

    def _block_tree(self):
        lo, hi = self.lo, self.hi
        ext = hi - lo
        diam = torch.sqrt(ext[:, 0] * ext[:, 0] + ext[:, 1] * ext[:, 1] + ext[:, 2] * ext[:, 2])
        t = torch.zeros(1, dtype=torch.int64, device=lo.device)
        s = t.clone()
        adm = []
        for level in range(self.depth + 1):
            gap = torch.clamp(torch.maximum(lo[t] - hi[s], lo[s] - hi[t]), min=0.0)
            dist = torch.sqrt(gap[:, 0] * gap[:, 0] + gap[:, 1] * gap[:, 1] + gap[:, 2] * gap[:, 2])
            far = torch.maximum(diam[t], diam[s]) <= (2.0 * ETA) * dist
            adm.append((t[far], s[far]))
            t, s = t[~far], s[~far]
            if level < self.depth:
                t, s = (torch.cat([2 * t + i for i in (1, 1, 2, 2)]), torch.cat([2 * s + j for j in (1, 2, 1, 2)]))
        self.adm = torch.cat([a for a, _ in adm]), torch.cat([b for _, b in adm])
        self.near = t, s


def _gauss(q, dev):
    x, w = np.polynomial.legendre.leggauss(q)
    return torch.from_numpy(0.5 * (x + 1)).to(dev), torch.from_numpy(0.5 * w).to(dev)


def _collapsed(q, dev):
    """Points (s, t) and weights of the collapsed Gauss rule on 0 <= t <= s <= 1."""
    x, w = _gauss(q, dev)
    s = x[:, None].expand(q, q)
    return s.reshape(-1), (x[:, None] * x[None]).reshape(-1), (w[:, None] * w[None] * s).reshape(-1)


def _lagrange(z, x):
    """Lagrange polynomials of the nodes z (..., m) at x (...): (..., m)."""
    m = z.shape[-1]
    out = []
    for j in range(m):
        v = torch.ones_like(x)
        for i in range(m):
            if i != j:
                v = v * (x - z[..., i]) / (z[..., j] - z[..., i])
        out.append(v)
    return torch.stack(out, dim=-1)


def _singular_regions(kind, dev):
    """The Sauter-Schwab regions of a singular pair: per quadrature point the
    weight and the reference points (x1, x2) and (y1, y2)."""
    g, w = _gauss(QUAD, dev)
    xi, a, b, c = (t.reshape(-1) for t in torch.meshgrid(g, g, g, g, indexing="ij"))
    w = torch.einsum("i,j,k,l->ijkl", w, w, w, w).reshape(-1)
    if kind == 3:     # identical
        W = w * xi ** 3 * a ** 2 * b
        p = [((xi, xi * (1 - a + a * b)), (xi * (1 - a * b * c), xi * (1 - a))),
             ((xi, xi * a * (1 - b + b * c)), (xi * (1 - a * b), xi * a * (1 - b))),
             ((xi * (1 - a * b * c), xi * a * (1 - b * c)), (xi, xi * a * (1 - b)))]
        reg = [(W, x, y) for x, y in p] + [(W, y, x) for x, y in p]
    elif kind == 2:   # common edge
        W1, W2 = w * xi ** 3 * a ** 2, w * xi ** 3 * a ** 2 * b
        reg = [(W1, (xi, xi * a * c), (xi * (1 - a * b), xi * a * (1 - b))),
               (W2, (xi, xi * a), (xi * (1 - a * b * c), xi * a * b * (1 - c))),
               (W2, (xi * (1 - a * b), xi * a * (1 - b)), (xi, xi * a * b * c)),
               (W2, (xi * (1 - a * b * c), xi * a * b * (1 - c)), (xi, xi * a)),
               (W2, (xi * (1 - a * b * c), xi * a * (1 - b * c)), (xi, xi * a * b))]
    else:             # common vertex
        W = w * xi ** 3 * b
        reg = [(W, (xi, xi * a), (xi * b, xi * b * c)), (W, (xi * b, xi * b * c), (xi, xi * a))]
    cat = lambda f: torch.cat([f(r) for r in reg])
    return cat(lambda r: r[0]), cat(lambda r: r[1][0]), cat(lambda r: r[1][1]), cat(lambda r: r[2][0]), \
        cat(lambda r: r[2][1])


class _Exact:
    """The H² matrix of one mesh; `part` is 'laplace', 'cos' or 'sin' (real and imaginary Helmholtz parts)."""

    def __init__(self, case, part="laplace"):
        vert, tri = _mesh(case)
        dev = _device()
        self.dev, self.m, self.part, self.kappa = dev, case["order"], part, case.get("kappa", 0.0)
        self.tree = t = _Tree(vert, tri, case["leaf"])
        self.k = self.m ** 3
        self.v = torch.from_numpy(np.ascontiguousarray(vert)).to(dev)
        self.f = torch.from_numpy(tri.astype(np.int64)).to(dev)
        self.n = len(tri)
        a, b, c = (self.v[self.f[:, i]] for i in range(3))
        self.area = 0.5 * torch.linalg.norm(torch.linalg.cross(b - a, c - a), dim=1)
        ext = t.hi - t.lo
        emax = ext.max(dim=1, keepdim=True).values
        half = torch.where(ext <= 1e-12 * emax, 1e-6 * emax.expand_as(ext), 0.5 * ext)
        nodes = torch.cos((2 * torch.arange(self.m, device=dev, dtype=torch.float64) + 1) * math.pi / (2 * self.m))
        self.cheb = (0.5 * (t.lo + t.hi))[..., None] + half[..., None] * nodes     # (clusters, 3, m)
        self.leaf0 = (1 << t.depth) - 1
        self.lmax = int(t.leaf_size.max())
        first = torch.cumsum(t.leaf_size, 0) - t.leaf_size
        pos = torch.arange(self.lmax, device=dev)
        self.pad = torch.where(pos < t.leaf_size[:, None], first[:, None] + pos, self.n)   # cluster-order index or n
        par = (torch.arange(len(t.lo), device=dev) - 1).clamp(min=0) // 2
        self.E = _lagrange(self.cheb[par][:, :, None, :].expand(-1, -1, self.m, -1), self.cheb)
        self.V = self._leaf_bases()
        self.near = self._nearfield()

    def kernel(self, r2):
        r = torch.sqrt(r2)
        if self.part == "sin":
            return torch.where(r > 0, torch.sin(self.kappa * r) / (4 * math.pi * r.clamp(min=1e-300)),
                               torch.full_like(r, self.kappa / (4 * math.pi)))
        g = 1.0 / (4 * math.pi * r)
        return torch.cos(self.kappa * r) * g if self.part == "cos" else g

    def _points(self, tri, s, t):
        """Points A + s (B - A) + t (C - B) of triangles given by vertex indices (..., 3)."""
        A, B, C = (self.v[tri[..., i]] for i in range(3))
        return A[..., None, :] + s[:, None] * (B - A)[..., None, :] + t[:, None] * (C - B)[..., None, :]

    def _leaf_bases(self):
        s, t, w = _collapsed((3 * (self.m - 1) + 3) // 2 + 1, self.dev)
        out = torch.empty(self.n, self.k, dtype=torch.float64, device=self.dev)
        for i in range(0, self.n, 1 << 15):
            tri = self.tree.order[i:i + (1 << 15)]
            x = self._points(self.f[tri], s, t)
            z = self.cheb[self.leaf0 + self.tree.leaf_id[i:i + (1 << 15)]]
            lx, ly, lz = (_lagrange(z[:, None, d].expand(-1, len(s), -1), x[..., d]) for d in range(3))
            wt = 2 * self.area[tri, None] * w
            zy = (lz * wt[..., None])[..., :, None] * ly[..., None, :]
            out[i:i + (1 << 15)] = torch.einsum("tqzy,tqx->tzyx", zy, lx).reshape(-1, self.k)
        return out

    def _nearfield(self):
        tb, sb = self.tree.near
        tb, sb = tb - self.leaf0, sb - self.leaf0
        s, t, w = _collapsed(QUAD, self.dev)
        X = self._points(self.f, s, t)                     # (n, q, 3)
        wa = 2 * self.area[:, None] * w
        L = self.lmax
        order = torch.cat([self.tree.order, self.tree.order.new_tensor([-1])])
        G = torch.empty(len(tb), L, L, dtype=torch.float64, device=self.dev)
        step = max(1, int(1.2e6) // (L * L))
        for b in range(0, len(tb), step):
            i, j = order[self.pad[tb[b:b + step]]], order[self.pad[sb[b:b + step]]]     # (blocks, L), -1: padding
            xi, xj = X[i], X[j]
            r2 = 0
            for d in range(3):
                diff = xi[:, :, None, :, None, d] - xj[:, None, :, None, :, d]
                r2 = r2 + diff * diff
            g = torch.einsum("btsac,bta,bsc->bts", self.kernel(r2), wa[i], wa[j])
            self._singular(g, i, j)
            g[(i < 0)[:, :, None].expand_as(g) | (j < 0)[:, None, :].expand_as(g)] = 0.0
            G[b:b + step] = g
        return G

    def _singular(self, g, i, j):
        """Overwrite the entries of pairs that share vertices."""
        fi, fj = self.f[i], self.f[j]
        common = torch.zeros(g.shape, dtype=torch.int64, device=self.dev)
        for a in range(3):
            for b in range(3):
                common += fi[:, :, None, a] == fj[:, None, :, b]
        common[(i < 0)[:, :, None].expand_as(g) | (j < 0)[:, None, :].expand_as(g)] = 0
        for kind in (1, 2, 3):
            blk, p, q = torch.nonzero(common == kind, as_tuple=True)
            if not len(blk):
                continue
            a, b = i[blk, p], j[blk, q]
            lo, hi = torch.minimum(a, b), torch.maximum(a, b)
            f, h = self._local(self.f[lo], self.f[hi], kind)
            W, x1, x2, y1, y2 = _singular_regions(kind, self.dev)
            vals = torch.empty(len(a), dtype=torch.float64, device=self.dev)
            for o in range(0, len(a), 1 << 16):
                sl = slice(o, o + (1 << 16))
                d = self._points(f[sl], x1, x2) - self._points(h[sl], y1, y2)
                vals[sl] = self.kernel((d * d).sum(-1)) @ W
            g[blk, p, q] = 4 * self.area[a] * self.area[b] * vals

    @staticmethod
    def _local(f, h, kind):
        """The vertices of both triangles in the order of the singular rules."""
        r = torch.arange(3, device=f.device)
        if kind == 3:
            f = torch.gather(f, 1, (f.argmin(dim=1, keepdim=True) + r) % 3)
            return f, f
        same = f[:, :, None] == h[:, None, :]
        inf, inh = same.any(dim=2), same.any(dim=1)
        if kind == 1:
            return (torch.gather(f, 1, (inf.int().argmax(dim=1, keepdim=True) + r) % 3),
                    torch.gather(h, 1, (inh.int().argmax(dim=1, keepdim=True) + r) % 3))
        big = torch.iinfo(torch.int64).max
        shared = torch.sort(torch.where(inf, f, big), dim=1).values[:, :2]
        of = torch.gather(f, 1, (~inf).int().argmax(dim=1, keepdim=True))
        oh = torch.gather(h, 1, (~inh).int().argmax(dim=1, keepdim=True))
        return torch.cat([shared, of], 1), torch.cat([shared, oh], 1)

    def apply(self, x):
        """G x for x (n, r) in the caller's order."""
        t, m, k, dev = self.tree, self.m, self.k, self.dev
        r = x.shape[1]
        xc = x[t.order]
        xp = torch.cat([xc, xc.new_zeros(1, r)])[self.pad]               # (leaves, L, r)
        Vp = torch.cat([self.V, self.V.new_zeros(1, k)])[self.pad]       # (leaves, L, k)
        xh = torch.zeros(len(t.lo), k, r, dtype=torch.float64, device=dev)
        yh = torch.zeros_like(xh)
        xh[self.leaf0:] = Vp.transpose(1, 2) @ xp
        for level in range(t.depth, 0, -1):
            c = slice((1 << level) - 1, (2 << level) - 1)
            E = self.E[c]
            up = xh[c].view(-1, m, m, m, r)
            up = torch.einsum("cia,czyir->czyar", E[:, 0], up)
            up = torch.einsum("cjb,czjxr->czbxr", E[:, 1], up)
            up = torch.einsum("clg,clyxr->cgyxr", E[:, 2], up)
            xh[(1 << (level - 1)) - 1:(1 << level) - 1] = up.reshape(-1, 2, k, r).sum(1)
        tb, sb = t.adm
        nodes = torch.stack([self.cheb[:, 0].repeat(1, m * m), self.cheb[:, 1].repeat_interleave(m, 1).repeat(1, m),
                             self.cheb[:, 2].repeat_interleave(m * m, 1)], dim=2)       # (clusters, k, 3)
        step = max(1, int(3e7) // (k * k + k * r))
        for b in range(0, len(tb), step):
            a, s = tb[b:b + step], sb[b:b + step]
            r2 = 0
            for d in range(3):
                diff = nodes[a, :, None, d] - nodes[s, None, :, d]
                r2 = r2 + diff * diff
            yh.index_add_(0, a, self.kernel(r2) @ xh[s])
        for level in range(1, t.depth + 1):
            c = slice((1 << level) - 1, (2 << level) - 1)
            E = self.E[c]
            par = yh[(1 << (level - 1)) - 1:(1 << level) - 1].repeat_interleave(2, 0).view(-1, m, m, m, r)
            par = torch.einsum("cia,czyar->czyir", E[:, 0], par)
            par = torch.einsum("cjb,czbxr->czjxr", E[:, 1], par)
            yh[c] += torch.einsum("clg,cgyxr->clyxr", E[:, 2], par).reshape(-1, k, r)
        yp = Vp @ yh[self.leaf0:]
        tb, sb = t.near[0] - self.leaf0, t.near[1] - self.leaf0
        step = max(1, int(1e8) // (self.lmax * max(r, self.lmax)))
        for b in range(0, len(tb), step):
            yp.index_add_(0, tb[b:b + step], self.near[b:b + step] @ xp[sb[b:b + step]])
        y = torch.zeros(self.n + 1, r, dtype=torch.float64, device=dev)
        y[torch.cat([t.order, t.order.new_tensor([self.n])])[self.pad].reshape(-1)] = yp.reshape(-1, r)
        return y[:self.n]

    def dense(self):
        cols = [self.apply(torch.eye(self.n, dtype=torch.float64, device=self.dev)[:, c:c + 512])
                for c in range(0, self.n, 512)]
        return torch.cat(cols, dim=1)


def exact(case, seed):
    x = _inputs(case, seed)
    if case["call"] == "batch":
        out = [_Exact(p).apply(torch.from_numpy(a.astype(np.float64)).to(_device()).t()).t().reshape(-1)
               for p, a in zip(_problems(case), x)]
        return torch.cat(out)
    if case["call"] == "helmholtz":
        xd = torch.from_numpy(x).to(_device()).t()
        n, r = xd.shape
        cols = torch.cat([xd.real, xd.imag], dim=1).contiguous()
        c, s = (_Exact(case, p).apply(cols) for p in ("cos", "sin"))
        return torch.complex(c[:, :r] - s[:, r:], c[:, r:] + s[:, :r])
    mat = _Exact(case)
    xd = torch.from_numpy(x.astype(np.float64)).to(_device()).t()
    if case["call"] == "solve":
        return torch.linalg.solve(mat.dense(), xd) if mat.n <= 12000 else None
    y = mat.apply(xd)
    return y.cpu() if case["call"] == "host" else y
