"""What the performance of this framework is measured on: the calls its users make.

A user has a scatterer (a mesh, or an H-Matrix of their own as explicit blocks),
turns it into an operator once, and then solves, multiplies or forms residuals
for excitations as they come.  The sizes are those of the benchmark, the tests
and the serving catalog, with odd ones between them.

  kind       one pass
  solve      hm_powerseries_solve on device vectors (HMatrix.solve, graph replay)
  host       hm_powerseries_solve_host: right-hand sides and solutions in host memory
  apply      hm_apply with its default FP64-class accumulation (a matvec of an outer solver)
  residual   hm_residual
  build      a new mesh to its solution: hm_build, hm_factor_leaf, excitation, solve
  serve      a burst of requests to the solve server, host vectors in and out

An operator (for `serve`, a server) is what a program keeps between calls, so the
states of one case share it; what the seed makes is the excitation, and for
`build` the mesh as well.
"""

import math

import numpy as np
import torch

from paper_2307_03968_gb300.hm import HMatrix, Server

DEV = "cuda"


# ------------------------------------------------------------------ the cases ----

def listed():
    return [
        # the smallest solve of the benchmark: one excitation of a small sphere, all launches and latency
        dict(name="sphere_1920_1rhs", kind="solve", body="sphere", n=8, size=0.3, leaf=32, arity=8, adm=2.0, tol=1e-4,
             nrhs=1, levels=1, refine=True),
        # the headline workload: one excitation of the two-wavelength sphere, operator streamed from HBM
        dict(name="sphere_30720_1rhs", kind="solve", body="sphere", n=32, size=2.0, leaf=64, arity=8, adm=2.0, tol=1e-4,
             nrhs=1, levels=1, refine=True),
        # the monostatic sweep over 181 angles on the same operator
        dict(name="sphere_30720_181rhs", kind="solve", body="sphere", n=32, size=2.0, leaf=64, arity=8, adm=2.0,
             tol=1e-4, nrhs=181, levels=1, refine=True),
        # every level of the tree, nested, without refinement: the full form of the series
        dict(name="sphere_30720_all_levels", kind="solve", body="sphere", n=32, size=2.0, leaf=64, arity=8, adm=2.0,
             tol=1e-4, nrhs=1, levels=-1, refine=False),
        # the paper's PEC plate at its tree depth: 64 leaves of 1,050 unknowns, its settings, one excitation
        dict(name="plate_67200_1rhs", kind="solve", body="plate", n=150, size=15.0, leaf=1050, arity=2, adm=1.0,
             tol=1e-3, nrhs=1, levels=1, refine=False),
        # inhomogeneous dielectric cube (volume equation), a batch of 16 incidences
        dict(name="cube_12600_16rhs", kind="solve", body="cube", n=10, size=2.0 / 3.0, leaf=64, arity=2, adm=1.0,
             tol=1e-4, nrhs=16, levels=1, refine=True),
        # an operator of the user's own (explicit blocks of odd sizes), a small batch through host memory
        dict(name="import_3001_13rhs_host", kind="host", body="import", n=3001, size=1.0, leaf=48, adm=1.0, nrhs=13,
             levels=1, refine=True),
        # the matvec of an outer iterative solver on such an operator, far blocks on every level
        dict(name="import_7500_apply", kind="apply", body="import", n=7500, size=1.6, leaf=64, adm=1.0, nrhs=1,
             levels=-1),
        # the residual check of a batch of finished solutions
        dict(name="import_7500_residual_50rhs", kind="residual", body="import", n=7500, size=1.6, leaf=64, adm=1.0,
             nrhs=50, levels=1),
        # a new geometry from its mesh to its solution: surface
        dict(name="build_sphere_7680", kind="build", body="sphere", n=16, size=1.0, leaf=64, arity=8, adm=2.0, tol=1e-4,
             nrhs=1, levels=1, refine=True),
        # the same for an inhomogeneous dielectric volume
        dict(name="build_cube_2808", kind="build", body="cube", n=6, size=0.4, leaf=64, arity=2, adm=1.0, tol=1e-4,
             nrhs=1, levels=1, refine=True),
        # the serving stream: twelve requests of 1..32 right-hand sides on three resident operators, queued at once
        dict(name="serve_12_requests", kind="serve", n=12, max_rhs=32),
    ]


def draw(rng):
    def log(lo, hi):
        return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))

    kind = rng.choice(["solve", "solve", "solve", "solve", "host", "apply", "residual", "residual", "build", "serve"])
    if kind == "serve":
        return dict(kind=kind, n=rng.randint(4, 16), max_rhs=log(4, 32))
    if kind == "build":
        if rng.random() < 0.5:
            return dict(kind=kind, body="sphere", n=rng.randint(6, 16), size=round(rng.uniform(0.3, 1.0), 3),
                        leaf=rng.randint(30, 64), arity=rng.choice([2, 8]), adm=rng.choice([1.0, 2.0]), tol=1e-4,
                        nrhs=log(1, 8), levels=1, refine=True)
        return dict(kind=kind, body="cube", n=rng.randint(3, 6), size=round(rng.uniform(0.2, 0.4), 3),
                    leaf=rng.randint(24, 64), arity=2, adm=1.0, tol=1e-4, nrhs=log(1, 8), levels=1, refine=True)
    if kind in ("apply", "residual") or (kind == "host" and rng.random() < 0.5):
        levels = rng.choice([1, -1])
        c = dict(kind=kind, body="import", n=log(300, 7500), size=round(rng.uniform(0.3, 1.6), 3),
                 leaf=rng.randint(24, 64), adm=1.0, nrhs=log(1, 64), levels=levels)
        if kind == "host":
            c.update(levels=1, refine=rng.random() < 0.7)
        return c
    body = rng.choice(["sphere", "sphere", "plate", "cube"])
    if body == "sphere":
        return dict(kind=kind, body=body, n=log(5, 30), size=round(rng.uniform(0.3, 2.0), 3), leaf=rng.randint(30, 64),
                    arity=8, adm=2.0, tol=1e-4, nrhs=log(1, 181), levels=1, refine=rng.random() < 0.7)
    if body == "plate":
        return dict(kind=kind, body=body, n=log(30, 140), size=round(rng.uniform(2.0, 12.0), 3), leaf=log(64, 1050),
                    arity=2, adm=1.0, tol=1e-3, nrhs=log(1, 4), levels=1, refine=False)
    return dict(kind=kind, body=body, n=rng.randint(4, 8), size=round(rng.uniform(0.25, 0.5), 3),
                leaf=rng.randint(32, 64), arity=2, adm=1.0, tol=1e-4, nrhs=log(1, 48), levels=1, refine=True)


# ------------------------------------------------------------------ the bodies ----

def sphere_mesh(f, radius):
    """Geodesic sphere: each icosahedron face cut into f^2 triangles (20 f^2 triangles, 30 f^2 edges)."""
    t = (1.0 + 5.0 ** 0.5) / 2.0
    v = np.array([(-1, t, 0), (1, t, 0), (-1, -t, 0), (1, -t, 0), (0, -1, t), (0, 1, t), (0, -1, -t), (0, 1, -t),
                  (t, 0, -1), (t, 0, 1), (-t, 0, -1), (-t, 0, 1)], dtype=np.float64)
    faces = [(0, 11, 5), (0, 5, 1), (0, 1, 7), (0, 7, 10), (0, 10, 11), (1, 5, 9), (5, 11, 4), (11, 10, 2), (10, 7, 6),
             (7, 1, 8), (3, 9, 4), (3, 4, 2), (3, 2, 6), (3, 6, 8), (3, 8, 9), (4, 9, 5), (2, 4, 11), (6, 2, 10),
             (8, 6, 7), (9, 8, 1)]
    pts, tris = [], []
    for a, b, c in faces:
        at = {}
        for i in range(f + 1):
            for j in range(f + 1 - i):
                at[i, j] = len(pts)
                pts.append((v[a] * (f - i - j) + v[b] * i + v[c] * j) / f)
        for i in range(f):
            for j in range(f - i):
                tris.append((at[i, j], at[i + 1, j], at[i, j + 1]))
                if i + j < f - 1:
                    tris.append((at[i + 1, j], at[i + 1, j + 1], at[i, j + 1]))
    pts = np.array(pts)
    pts /= np.linalg.norm(pts, axis=1, keepdims=True)
    _, first, back = np.unique(np.round(pts * 1e7).astype(np.int64), axis=0, return_index=True, return_inverse=True)
    xyz, tri = pts[first] * radius, back.reshape(-1)[np.array(tris)].astype(np.int32)
    p = xyz[tri]
    inward = np.einsum("ij,ij->i", np.cross(p[:, 1] - p[:, 0], p[:, 2] - p[:, 0]), p.sum(1)) < 0
    tri[inward] = tri[inward][:, [0, 2, 1]]
    return xyz, tri


def plate_mesh(n, side):
    """Square plate of n x n squares, two triangles each."""
    g = np.linspace(-side / 2, side / 2, n + 1)
    X, Y = np.meshgrid(g, g, indexing="ij")
    xyz = np.stack([X.ravel(), Y.ravel(), np.zeros(X.size)], axis=1)
    i, j = (a.ravel() for a in np.meshgrid(np.arange(n), np.arange(n), indexing="ij"))
    a, b, c, d = i * (n + 1) + j, (i + 1) * (n + 1) + j, (i + 1) * (n + 1) + j + 1, i * (n + 1) + j + 1
    return xyz, np.stack([np.stack([a, b, c], 1), np.stack([a, c, d], 1)], 1).reshape(-1, 3).astype(np.int32)


def cube_mesh(n, side):
    """Cube of n^3 voxels, six tetrahedra each around the main diagonal."""
    g = np.linspace(-side / 2, side / 2, n + 1)
    xyz = np.stack([a.ravel() for a in np.meshgrid(g, g, g, indexing="ij")], axis=1)
    step = ((n + 1) ** 2, n + 1, 1)
    v0 = np.stack([a.ravel() for a in np.meshgrid(*[np.arange(n)] * 3, indexing="ij")], 1) @ np.array(step)
    tets = []
    for p in [(0, 1, 2), (0, 2, 1), (1, 0, 2), (1, 2, 0), (2, 0, 1), (2, 1, 0)]:
        corner, path = v0, [v0]
        for ax in p:
            corner = corner + step[ax]
            path.append(corner)
        tets.append(np.stack(path, 1))
    return xyz, np.stack(tets, 1).reshape(-1, 4).astype(np.int32)


def mesh_of(case, stretch=1.0):
    size = case["size"] * stretch
    if case["body"] == "sphere":
        return sphere_mesh(case["n"], size) + (None,)
    if case["body"] == "plate":
        return plate_mesh(case["n"], size) + (None,)
    xyz, tet = cube_mesh(case["n"], size)
    return xyz, tet, np.random.default_rng(4).uniform(2.0, 6.0, len(tet))   # inhomogeneous: eps_r uniform in [2, 6]


def incidences(case, seed):
    """The sweep's angles for many right-hand sides of a surface, else random plane waves."""
    rng = np.random.default_rng(seed)
    n = case["nrhs"]
    if n > 64 and case["body"] == "sphere":
        th, ph = np.linspace(0.0, np.pi, n), rng.uniform(0.0, 2 * np.pi)
        k = -np.stack([np.sin(th) * np.cos(ph), np.sin(th) * np.sin(ph), np.cos(th)], 1)
        return k, np.stack([np.cos(th) * np.cos(ph), np.cos(th) * np.sin(ph), -np.sin(th)], 1)
    k = rng.normal(size=(n, 3))
    k /= np.linalg.norm(k, axis=1, keepdims=True)
    a = rng.normal(size=(n, 3))
    p = a - np.einsum("ij,ij->i", a, k)[:, None] * k
    return k, p / np.linalg.norm(p, axis=1, keepdims=True)


# -------------------------------------------- an operator of the user's own ----

class Blocks:
    """An H-Matrix assembled by the user's program: the scalar kernel exp(-jkr)/(4 pi r)
    between points of a sphere, bisected into leaves; near blocks dense, admissible
    pairs as Q (Q^H B) of a fixed rank per level.  complex128 on the GPU, by groups
    of equal shape, the values rounded to single precision (what the library stores)."""

    def __init__(self, case):
        n, radius, leaf = case["n"], case["size"], case["leaf"]
        i = np.arange(n) + 0.5
        ct, ph = 1 - 2 * i / n, np.pi * (1 + 5 ** 0.5) * i
        st = np.sqrt(1 - ct * ct)
        pts = radius * np.stack([st * np.cos(ph), st * np.sin(ph), ct], 1)
        depths = [[np.arange(n)]]
        while max(len(c) for c in depths[-1]) > leaf:
            nxt = []
            for c in depths[-1]:
                ax = int(np.argmax(np.ptp(pts[c], axis=0)))
                o = c[np.argsort(pts[c, ax], kind="stable")]
                nxt += [o[:len(o) // 2], o[len(o) // 2:]]
            depths.append(nxt)
        self.perm = np.concatenate(depths[-1])
        pts = pts[self.perm]
        spans = []
        for d in depths:
            off = np.concatenate([[0], np.cumsum([len(c) for c in d])])
            spans.append([(int(off[q]), len(c)) for q, c in enumerate(d)])
        self.n, self.leaf_off = n, np.array([o for o, _ in spans[-1]] + [n])
        last = len(spans) - 1
        box = [[(pts[o:o + m].min(0), pts[o:o + m].max(0)) for o, m in s] for s in spans]
        near, far = [], {}

        def visit(d, t, s):
            (al, ah), (bl, bh) = box[d][t], box[d][s]
            gap = np.linalg.norm(np.maximum(0, np.maximum(bl - ah, al - bh)))
            if t != s and gap > 0 and gap >= case["adm"] * min(np.linalg.norm(ah - al), np.linalg.norm(bh - bl)):
                far.setdefault(last - d + 1, []).append((spans[d][t], spans[d][s]))
            elif d == last:
                if t != s:
                    near.append((spans[d][t], spans[d][s]))
            else:
                for ct_ in (2 * t, 2 * t + 1):
                    for cs in (2 * s, 2 * s + 1):
                        if t != s or ct_ <= cs:
                            visit(d + 1, ct_, cs)

        visit(0, 0, 0)
        P = torch.tensor(pts, device=DEV)
        area = 4 * math.pi * radius ** 2 / n
        gen = torch.Generator(device=DEV).manual_seed(7)

        def kernel(r0, m, c0, w):
            d = torch.cdist(P[self.rows(r0, m)], P[self.rows(c0, w)], compute_mode="donot_use_mm_for_euclid_dist")
            d0 = d.clamp_min(1e-9)
            g = torch.polar(area / (4 * math.pi * d0), -2 * math.pi * d0)
            return torch.where(d > 0, g, torch.tensor(1.5 * math.sqrt(area / math.pi), dtype=g.dtype, device=DEV))

        def single(a):
            return a.to(torch.complex64).to(torch.complex128)

        def grouped(pairs):
            shapes = {}
            for (a, m), (b, w) in pairs:
                shapes.setdefault((m, w), []).append((a, b))
            for (m, w), ab in sorted(shapes.items()):
                t = torch.tensor(ab, device=DEV)
                yield t[:, 0], m, t[:, 1], w

        # groups: (level, row starts, column starts, factors); level 0 = self blocks, dense near blocks have level 1
        self.groups = []
        for r0, m, c0, w in grouped([(s, s) for s in spans[-1]]):
            self.groups.append((0, r0, c0, (single(kernel(r0, m, c0, w)),)))
        for r0, m, c0, w in grouped(near):
            self.groups.append((1, r0, c0, (single(kernel(r0, m, c0, w)),)))
        for lev in sorted(far):
            for r0, m, c0, w in grouped(far[lev]):
                k = min(m, w, 7 + 2 * lev)
                B = kernel(r0, m, c0, w)
                om = torch.randn(w, k, dtype=B.dtype, device=DEV, generator=gen)
                Q = torch.linalg.qr(B @ om)[0]
                self.groups.append((lev, r0, c0, (single(Q), single(Q.mH @ B))))
        self.levels = max(far, default=1)

    @staticmethod
    def rows(r0, m):
        return r0[:, None] + torch.arange(m, device=DEV)[None, :]

    def elems(self, levels=-1):
        """Stored complex elements of the self blocks and of the other blocks of levels 1..levels."""
        top = self.levels if levels < 0 else levels
        s = sum(g[3][0].numel() for g in self.groups if g[0] == 0)
        return s, sum(f.numel() for g in self.groups if 0 < g[0] <= top for f in g[3])

    def operator(self):
        """The same blocks handed to the library."""
        blocks = {0: [], 1: [], 2: []}
        for lev, r0, c0, f in self.groups:
            r0, c0, f = r0.tolist(), c0.tolist(), [a.cpu().numpy() for a in f]
            for q in range(len(r0)):
                if lev == 0:
                    blocks[0].append((r0[q], f[0][q]))
                elif len(f) == 1:
                    blocks[1].append((r0[q], c0[q], f[0][q]))
                else:
                    blocks[2].append((lev, r0[q], c0[q], f[0][q], f[1][q]))
        selfs = [b for _, b in sorted(blocks[0], key=lambda e: e[0])]
        A = HMatrix.from_blocks(self.perm, self.leaf_off, selfs, blocks[1], blocks[2])
        A.factor_leaf()
        return A

    # the same quantities in 64 bits; vectors are (N, R) in tree order
    def to_tree(self, v):
        return v.to(torch.complex128).reshape(-1, self.n)[:, torch.as_tensor(self.perm, device=v.device)].T.contiguous()

    def from_tree(self, v, like):
        out = torch.empty_like(v)
        out[torch.as_tensor(self.perm, device=v.device)] = v
        return out.T.reshape(like.shape).contiguous()

    def off_diagonal(self, x, levels):
        z, top = torch.zeros_like(x), self.levels if levels < 0 else levels
        for lev, r0, c0, f in self.groups:
            if not 0 < lev <= top:
                continue
            i, j = self.rows(r0, f[0].shape[1]), self.rows(c0, f[-1].shape[2])
            xi, xj = x[i], x[j]
            for g in f[::-1]:
                xj = g @ xj
            for g in f:
                xi = g.mT @ xi
            z.index_add_(0, i.reshape(-1), xj.reshape(-1, x.shape[1]))
            z.index_add_(0, j.reshape(-1), xi.reshape(-1, x.shape[1]))
        return z

    def diagonal(self, x, solve):
        z = torch.empty_like(x)
        for lev, r0, _, f in self.groups:
            if lev == 0:
                i = self.rows(r0, f[0].shape[1])
                z[i] = torch.linalg.solve(f[0], x[i]) if solve else f[0] @ x[i]
        return z

    def product(self, x, levels):
        return self.diagonal(x, False) + self.off_diagonal(x, levels)

    def series(self, r, terms=2):
        y = x = self.diagonal(r, True)
        for _ in range(terms):
            x = y - self.diagonal(self.off_diagonal(x, 1), True)
        return x


# ------------------------------------------------- what a program keeps, inputs ----

_kept = {}


def keep(key, make):
    """The operators a program has resident: the last few, each made once."""
    if key not in _kept:
        while len(_kept) >= 4:
            _kept.pop(next(iter(_kept)))
        _kept[key] = make()
    _kept[key] = _kept.pop(key)      # the most recent last
    return _kept[key]


def operator(case):
    own = ("body", "n", "size", "leaf", "adm") + (() if case["body"] == "import" else ("arity", "tol"))
    key = tuple(case[k] for k in own)
    if case["body"] == "import":
        return keep(key + ("operator",), lambda: keep(key, lambda: Blocks(case)).operator())

    def make():
        xyz, cells, eps = mesh_of(case)
        A = HMatrix.build(xyz, cells, leaf_size=case["leaf"], arity=case["arity"], adm=case["adm"],
                          aca_tol=case["tol"], levels=-1, eps_r=eps)
        A.factor_leaf()
        return A

    return keep(key, make)


def own_blocks(case):
    return keep(tuple(case[k] for k in ("body", "n", "size", "leaf", "adm")), lambda: Blocks(case))


SERVED = [("sphere", 8, 0.3, 64, 8, 2.0), ("sphere", 16, 1.0, 64, 8, 2.0), ("cube", 4, 0.27, 64, 2, 1.0)]


def server(case):
    def make():
        s = Server(n_slots=4, max_batch_rhs=64)
        ops = []
        for body, n, size, leaf, arity, adm in SERVED:
            xyz, cells, eps = mesh_of(dict(body=body, n=n, size=size))
            ops.append(s.add_mesh(xyz, cells, leaf_size=leaf, arity=arity, adm=adm, levels=1, refine=True, eps_r=eps))
        for op, n in ops:            # resident before the stream starts
            s.wait(s.submit(op, np.zeros((1, n), np.complex64)))
        return s, ops

    return keep(("serve",), make)


def requests(case):
    """(operator, right-hand sides) of the burst: part of the case."""
    rng = np.random.default_rng(1000 * case["n"] + case["max_rhs"])
    return [(int(rng.integers(len(SERVED))), int(rng.integers(1, case["max_rhs"] + 1))) for _ in range(case["n"])]


def random_vectors(rng, *shape):
    return (rng.normal(size=shape) + 1j * rng.normal(size=shape)).astype(np.complex64)


def prepare(case, seed):
    rng = np.random.default_rng(seed)
    if case["kind"] == "serve":
        s, ops = server(case)
        return dict(case=case, server=s, work=[(ops[o][0], random_vectors(rng, r, ops[o][1])) for o, r in requests(case)])
    if case["kind"] == "build":
        xyz, cells, eps = mesh_of(case, stretch=rng.uniform(0.98, 1.02))
        khat, phat = incidences(case, seed)
        return dict(case=case, mesh=(xyz, cells, eps), khat=khat, phat=phat)
    A = operator(case)
    shape = (case["nrhs"], A.n)
    st = dict(case=case, op=A)
    if case["body"] != "import":
        b = torch.empty(shape, dtype=torch.complex64, device=DEV)
        A.rhs_plane_wave(*incidences(case, seed), b)
    else:
        b = torch.from_numpy(random_vectors(rng, *shape)).to(DEV)
    if case["kind"] == "host":       # page-locked, as a program that streams excitations keeps them
        st["b"] = torch.empty(shape, dtype=torch.complex64, pin_memory=True).copy_(b).numpy()
        st["x"] = torch.empty(shape, dtype=torch.complex64, pin_memory=True).numpy()
        return st
    if case["kind"] == "residual":   # solutions good to about 1e-3
        st["x"] = b
        B = own_blocks(case)
        noise = torch.from_numpy(random_vectors(rng, *shape)).to(DEV)
        st["b"] = B.from_tree(B.product(B.to_tree(b + 1e-3 * noise), case["levels"]), b).to(torch.complex64)
    else:
        st["b"] = b
    st["out"] = torch.empty_like(b)
    return st


def run(state):
    case = state["case"]
    kind = case["kind"]
    if kind == "serve":
        s = state["server"]
        queued = [s.submit(op, b) for op, b in state["work"]]
        return [s.wait(q)[0] for q in queued]
    opts = dict(n_terms=2, n_levels=case["levels"], nested=True)
    if kind == "build":
        xyz, cells, eps = state["mesh"]
        A = HMatrix.build(xyz, cells, leaf_size=case["leaf"], arity=case["arity"], adm=case["adm"],
                          aca_tol=case["tol"], levels=1, eps_r=eps)
        A.factor_leaf()
        b = torch.empty((case["nrhs"], A.n), dtype=torch.complex64, device=DEV)
        A.rhs_plane_wave(state["khat"], state["phat"], b)
        x = torch.empty_like(b)
        A.solve(b, x, refine=case["refine"], graph=False, **opts)
        return b, x
    A, b = state["op"], state["b"]
    if kind == "host":
        return A.solve_host(b, refine=case["refine"], out=state["x"], **opts)
    if kind == "apply":
        A.apply(b, state["out"], n_levels=case["levels"])
    elif kind == "residual":
        norms = A.residual(b, state["x"], state["out"], n_levels=case["levels"])
        return state["out"], norms[0], norms[1]
    else:
        A.solve(b, state["out"], refine=case["refine"], **opts)
    return state["out"]


def exact(case, seed):
    """On the user's own blocks; an operator built from a mesh has its own fill and ACA
    behind it, which 64-bit torch or numpy does not redo in seconds."""
    if case.get("body") != "import":
        return None
    st, B = prepare(case, seed), own_blocks(case)
    b = torch.as_tensor(st["b"], device=DEV)
    bt = B.to_tree(b)
    if case["kind"] == "apply":
        return B.from_tree(B.product(bt, case["levels"]), b)
    if case["kind"] == "residual":
        r = bt - B.product(B.to_tree(st["x"]), case["levels"])
        return B.from_tree(r, b), (r.abs() ** 2).sum(0).cpu().numpy(), (bt.abs() ** 2).sum(0).cpu().numpy()
    x = B.series(bt)
    if case["refine"]:
        x = x + B.series(bt - B.product(x, 1))
    return B.from_tree(x, b)


# ------------------------------------------------------------------- the work ----

def solve_work(self_elems, elems, n, case):
    """A solve: every stored element and leaf inverse read once, b read and x written.
    A product applies each stored element to both of its clusters."""
    r, refine = case["nrhs"], case.get("refine", False)
    products = 2 * (2 if refine else 1) + (1 if refine else 0)
    leaves = 3 * (2 if refine else 1) + (1 if refine else 0)
    return {"bytes": 8.0 * (elems + self_elems * (2 if refine else 1)) + 16.0 * n * r,
            "flops": 8.0 * r * (2 * products * elems + leaves * self_elems)}


def work(case):
    kind = case["kind"]
    if kind == "serve":
        total = {"bytes": 0.0, "flops": 0.0}
        for o, r in requests(case):
            n = {"sphere": 30 * SERVED[o][1] ** 2, "cube": 12 * SERVED[o][1] ** 3 + 6 * SERVED[o][1] ** 2}[SERVED[o][0]]
            total["bytes"] += 16.0 * n * r
            total["flops"] += 8.0 * r * 10 * (n * n / 3)    # about a third of the pairs, as elements, in ten half products
        return total
    if kind == "build":
        # the matrix entries of the near half (about a fifth of all pairs) and of the ACA
        # crosses, each a product of quadrature rules over up to four element pairs
        n = 30 * case["n"] ** 2 if case["body"] == "sphere" else 12 * case["n"] ** 3 + 6 * case["n"] ** 2
        return {"bytes": 8.0 * n * n / 5 + 16.0 * n * case["nrhs"],
                "flops": (n * n / 5.0) * (4 * 49 if case["body"] == "sphere" else 4 * 16 + 4 * 28 + 49) * 40.0}
    if case["body"] == "import":
        s, e = own_blocks(case).elems(case["levels"])
        n = case["n"]
    else:
        i = operator(case).info()
        n, s = i.n, i.self_elems
        e = i.near_elems + sum(i.far_elems[:16] if case["levels"] < 0 else i.far_elems[:case["levels"]])
        if case["levels"] < 0:      # nested: three solves of the leaf level and two products of the next
            w = solve_work(s, i.near_elems + i.far_elems[0], n, case)
            return {"bytes": w["bytes"] + 8.0 * sum(i.far_elems[1:16]),
                    "flops": 3 * w["flops"] + 8.0 * case["nrhs"] * 4 * sum(i.far_elems[1:16])}
    if kind in ("apply", "residual"):
        return {"bytes": 8.0 * (s + e) + (16.0 + 8.0 * (kind == "residual")) * n * case["nrhs"],
                "flops": 8.0 * case["nrhs"] * (s + 2 * e)}
    return solve_work(s, e, n, case)
