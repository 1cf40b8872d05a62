"""The work that users of the library have it do, as measurable cases.

Every case goes through the public entry points of paper_1510_07244_gb300 on a
seeded mesh: dense matrices, near-field and coupling blocks (single calls and
plans, piecewise constant and linear, the FP64 form and the float-full form,
fixed and learned orders), the Green matrices of the GCA, the H2 product, and
the exterior problem's solve.  Cluster trees, block lists and pivots are made
here (numpy, from the mesh before its jitter, so that a case's shapes do not
depend on the seed); the seed moves the vertices and fills the vectors.

exact() evaluates the same integrals with the same quadrature rules in 64 bits
with torch alone: tensor Gauss rules after the Duffy map or Radon's 7 points
for disjoint triangles, Sauter-Schwab rules for touching ones.
"""
import functools
import math

import numpy as np
import torch

import paper_1510_07244_gb300 as bem

DEVICE = "cuda:0"
COMPLEX = ("helmholtz_slp", "helmholtz_dlp", "helmholtz_bw")
LEAF, ETA = 32, 2.0


# ---------------------------------------------------------------------------
# Cases
# ---------------------------------------------------------------------------
def _case(work, mesh, kernels, basis="p0", precision="fp64", rule="duffy", q=3, singular=5,
          kappa=0.0, rank=16, points=0, name=None):
    c = {"work": work, "mesh": mesh, "kernels": kernels, "basis": basis, "precision": precision,
         "rule": rule, "q": q, "singular": singular, "kappa": kappa, "rank": rank, "points": points}
    return {"name": name, **c} if name else c


def listed():
    return [
        # the smallest call: a dense single layer with the default descriptors, where a user
        # waits for launches, not for arithmetic
        _case("dense", "ico:2", "laplace_slp", name="dense_small"),
        # the dense matrix of the 1280-triangle sphere in the float-full form, Radon's rule
        _case("dense", "ico:8", "laplace_slp", precision="mixed_full", rule="tri7", singular=4,
              name="dense_mixed"),
        # the operator of the exterior Helmholtz problem (complex, FP64 in every precision)
        _case("dense", "octa:16", "helmholtz_bw", kappa=3.0, name="dense_exterior"),
        # that problem's solve: GMRES on the dense matrix, then the field off the surface
        _case("solve", "octa:16", "helmholtz_bw", kappa=3.0, points=256, name="solve_exterior"),
        # near-field and coupling calls without a plan, Helmholtz on a cube, default precision
        _case("blocks", "cube:21", "helmholtz_slp", kappa=8.0, name="blocks_fp64"),
        # the same calls as one step on a new mesh: upload, blocks, free; double layer in the
        # float-full form with its cancellation guard
        _case("upload", "torus:100x50", "laplace_dlp", precision="mixed_full", name="upload_mixed"),
        # many bodies of mixed shapes and sizes in one plan, both operators, float-full form
        _case("plan", "octa:60+cube:30+torus:110x55+octa:9+cube:12+torus:40x21+octa:25+torus:62x31",
              "laplace_dlp+helmholtz_slp", precision="mixed_full", kappa=5.0, name="plan_bodies"),
        # both Laplace layers over the same blocks, piecewise linear, float-full form
        _case("plan", "ico:32", "laplace_slp+laplace_dlp", basis="p1", precision="mixed_full",
              name="plan_linear"),
        # the same operators in the FP64 form on a small body
        _case("plan", "octa:13", "laplace_slp+laplace_dlp", basis="p1", name="plan_linear_fp64"),
        # quadrature orders chosen per pair by the order model
        _case("learned", "octa:48", "laplace_dlp+helmholtz_slp", precision="mixed_full", kappa=16.0,
              name="plan_learned"),
        # the Green matrices of a whole cluster tree, as the GCA needs them
        _case("green", "ico:32", "laplace_slp", basis="p1", rule="tri7", name="green_tree"),
        # one product with an H2 matrix, the inner step of every iterative solve
        _case("h2", "octa:64", "laplace_slp", rank=32, name="h2_product"),
    ]


def _log(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def _body(rng, lo, hi):
    """A body of about lo .. hi triangles."""
    n = _log(rng, lo, hi)
    kind = rng.choice(("octa", "cube", "torus"))
    if kind == "torus":
        v = max(5, int(math.sqrt(n / 2 / rng.uniform(1.5, 3.0))))
        return "torus:%dx%d" % (max(5, n // (2 * v)), v)
    return "%s:%d" % (kind, max(1, int(math.sqrt(n / (8 if kind == "octa" else 12)))))


def draw(rng):
    work = rng.choice(("dense", "dense", "solve", "blocks", "upload", "plan", "plan", "plan",
                       "learned", "green", "h2"))
    rule, q = rng.choice((("duffy", 2), ("duffy", 3), ("duffy", 3), ("duffy", 4), ("tri7", 3)))
    kappa = round(rng.uniform(1.0, 12.0), 3)
    singular = rng.choice((3, 4, 5, 5, 6))
    rank = rng.randint(6, 20)
    if work == "dense":
        precision = rng.choice(("fp64", "mixed", "mixed_full"))
        kernel = rng.choice(("laplace_slp", "laplace_dlp", "helmholtz_slp"))
        if precision == "fp64":
            kernel = rng.choice((kernel, "helmholtz_dlp", "helmholtz_bw"))
            return _case(work, _body(rng, 80, 900), kernel, rule=rule, q=q, singular=singular,
                         kappa=kappa, basis=rng.choice(("p0", "p0", "p1")))
        return _case(work, _body(rng, 200, 6000), kernel, precision=precision, rule=rule, q=q,
                     singular=singular, kappa=kappa)
    if work == "solve":
        return _case(work, _body(rng, 200, 2000), "helmholtz_bw", kappa=round(rng.uniform(1, 4), 3),
                     points=_log(rng, 20, 400))
    if work == "blocks":
        precision = rng.choice(("fp64", "mixed_full"))
        hi = 2500 if precision == "fp64" else 12000
        return _case(work, _body(rng, 300, hi), rng.choice(("laplace_slp", "laplace_dlp",
                     "helmholtz_slp")), precision=precision, rule=rule, q=q, singular=singular,
                     kappa=kappa, rank=rank)
    if work == "upload":
        return _case(work, _body(rng, 500, 10000), rng.choice(("laplace_dlp", "helmholtz_slp")),
                     precision="mixed_full", rule=rule, q=q, singular=singular, kappa=kappa,
                     rank=rank)
    if work == "plan":
        if rng.random() < 0.4:
            precision = rng.choice(("mixed_full", "fp64"))
            hi = 18000 if precision == "mixed_full" else 1200
            q = min(q, 3)
            return _case(work, _body(rng, 400, hi), "laplace_slp+laplace_dlp", basis="p1",
                         precision=precision, rule=rule, q=q, singular=singular, rank=rank)
        bodies = "+".join(_body(rng, 400, 9000) for _ in range(rng.randint(1, 6)))
        return _case(work, bodies, rng.choice(("laplace_dlp+helmholtz_slp", "laplace_slp",
                     "laplace_dlp")), precision=rng.choice(("mixed", "mixed_full", "mixed_full")),
                     rule=rule, q=min(q, 3), singular=min(singular, 5), kappa=kappa, rank=rank)
    if work == "learned":
        return _case(work, _body(rng, 1000, 16000), "laplace_dlp+helmholtz_slp",
                     precision="mixed_full", kappa=kappa, singular=singular, rank=rank)
    if work == "green":
        basis = rng.choice(("p0", "p1"))
        rule, q = rng.choice((("tri7", 3), ("duffy", 2), ("duffy", 3)))
        return _case(work, _body(rng, 500, 16000), rng.choice(("laplace_slp", "helmholtz_slp")),
                     basis=basis, rule=rule, q=q, kappa=kappa, rank=rank)
    return _case(work, _body(rng, 1000, 30000), "laplace_slp", rank=rng.randint(8, 32))


# ---------------------------------------------------------------------------
# Meshes, cluster trees and block lists (numpy; shared by all seeds of a case)
# ---------------------------------------------------------------------------
def _split_faces(corners, faces, n, sphere):
    """Every triangle (or parallelogram corner a, b, c, d) split regularly, equal points merged."""
    points, tris, base = [], [], 0
    i, j = np.meshgrid(np.arange(n + 1), np.arange(n + 1), indexing="ij")
    for f in faces:
        a, b, c = (corners[k] for k in f[:3])
        if len(f) == 3:
            ii, jj = i[i + j <= n], j[i + j <= n]
            p = (a * (n - ii - jj)[:, None] + b * ii[:, None] + c * jj[:, None]) / n
            at = np.full((n + 2, n + 2), -1)
            at[ii, jj] = np.arange(len(ii))
            up = [(x, y) for x in range(n) for y in range(n - x)]
            x, y = np.array(up).T
            t = [np.stack([at[x, y], at[x + 1, y], at[x, y + 1]], 1)]
            x, y = x[x + y + 1 < n], y[x + y + 1 < n]
            t.append(np.stack([at[x + 1, y], at[x + 1, y + 1], at[x, y + 1]], 1))
        else:
            p = a + (b - a) * (i.reshape(-1, 1) / n) + (corners[f[3]] - a) * (j.reshape(-1, 1) / n)
            at = np.arange((n + 1) ** 2).reshape(n + 1, n + 1)
            q = [at[:-1, :-1].ravel(), at[1:, :-1].ravel(), at[1:, 1:].ravel(), at[:-1, 1:].ravel()]
            t = [np.stack([q[0], q[1], q[2]], 1), np.stack([q[0], q[2], q[3]], 1)]
        points.append(p)
        tris.append(np.concatenate(t) + base)
        base += len(p)
    points = np.concatenate(points)
    _, first, where = np.unique(np.round(points * 2.0 ** 30).astype(np.int64), axis=0,
                                return_index=True, return_inverse=True)
    v = points[first]
    t = where.reshape(-1)[np.concatenate(tris)]
    middle = v.mean(0)
    if sphere:
        v = v / np.linalg.norm(v, axis=1, keepdims=True)
    w = v[t]
    out = np.einsum("ij,ij->i", np.cross(w[:, 1] - w[:, 0], w[:, 2] - w[:, 1]), w.mean(1) - middle)
    t[out < 0] = t[out < 0][:, [0, 2, 1]]
    return v, t.astype(np.int32)


@functools.lru_cache(maxsize=None)
def _surface(spec):
    """(vertices, triangles) of a closed, outward oriented body."""
    kind, size = spec.split(":")
    if kind == "torus":
        nu, nv = (int(x) for x in size.split("x"))
        u, v = np.meshgrid(2 * np.pi * np.arange(nu) / nu, 2 * np.pi * np.arange(nv) / nv,
                           indexing="ij")
        p = np.stack([(1 + 0.3 * np.cos(v)) * np.cos(u), (1 + 0.3 * np.cos(v)) * np.sin(u),
                      0.3 * np.sin(v)], -1).reshape(-1, 3)
        at = np.arange(nu * nv).reshape(nu, nv)
        a, b = at.ravel(), np.roll(at, -1, 0).ravel()
        c, d = np.roll(at, (-1, -1), (0, 1)).ravel(), np.roll(at, -1, 1).ravel()
        return p, np.concatenate([np.stack([a, b, c], 1), np.stack([a, c, d], 1)]).astype(np.int32)
    n = int(size)
    if kind == "octa":
        corners = np.array([(1, 0, 0), (-1, 0, 0), (0, 1, 0), (0, -1, 0), (0, 0, 1), (0, 0, -1)],
                           float)
        return _split_faces(corners, [(a, b, c) for a in (0, 1) for b in (2, 3) for c in (4, 5)],
                            n, True)
    if kind == "cube":
        corners = np.array([(x, y, z) for x in (0, 1) for y in (0, 1) for z in (0, 1)], float)
        faces = [(0, 1, 3, 2), (4, 5, 7, 6), (0, 1, 5, 4), (2, 3, 7, 6), (0, 2, 6, 4), (1, 3, 7, 5)]
        return _split_faces(corners, faces, n, False)
    g = (1 + 5 ** 0.5) / 2
    corners = np.array([p for a in (-1, 1) for b in (-g, g)
                        for p in ((0, a, b), (a, b, 0), (b, 0, a))], float)
    near = np.abs(np.linalg.norm(corners[:, None] - corners[None], axis=2) - 2) < 1e-9
    faces = [(a, b, c) for a in range(12) for b in range(a) for c in range(b)
             if near[a, b] and near[b, c] and near[a, c]]
    return _split_faces(corners / np.linalg.norm(corners[0]), faces, n, True)


def _mesh(spec, seed):
    """The body with every coordinate moved by up to 5% of the mean edge length."""
    v, t = _surface(spec)
    h = np.linalg.norm(v[t[:, 1]] - v[t[:, 0]], axis=1).mean()
    rng = np.random.default_rng([seed, len(t)])
    return v + rng.uniform(-0.05 * h, 0.05 * h, v.shape), t


class _Tree:
    """Cluster tree by geometric bisection and its block partition."""

    def __init__(self, spec, basis):
        v, t = _surface(spec)
        w = v[t]
        lo, hi = w.min(1), w.max(1)
        points = w.mean(1)
        if basis == "p1":
            points = v
            slo, shi = np.full(v.shape, np.inf), np.full(v.shape, -np.inf)
            for k in range(3):
                np.minimum.at(slo, t[:, k], lo)
                np.maximum.at(shi, t[:, k], hi)
            lo, hi = slo, shi
        self.n = len(points)
        self.idx, self.sons, self.depth = [], [], []
        todo = [(np.arange(self.n), -1, 0)]
        while todo:
            idx, parent, depth = todo.pop()
            c = len(self.idx)
            self.idx.append(idx)
            self.sons.append([])
            self.depth.append(depth)
            if parent >= 0:
                self.sons[parent].append(c)
            if len(idx) > LEAF:
                p = points[idx]
                axis = int(np.argmax(p.max(0) - p.min(0)))
                left = p[:, axis] <= 0.5 * (p[:, axis].max() + p[:, axis].min())
                todo += [(idx[~left], c, depth + 1), (idx[left], c, depth + 1)]
        self.nc = len(self.idx)
        self.lo = np.array([lo[i].min(0) for i in self.idx])
        self.hi = np.array([hi[i].max(0) for i in self.idx])
        son = np.array([s if s else [-1, -1] for s in self.sons])
        self.son = son.astype(np.int32)
        diam = np.linalg.norm(self.hi - self.lo, axis=1)
        a, b = np.zeros(1, np.int64), np.zeros(1, np.int64)
        near, far = [], []
        while len(a):
            gap = np.maximum(0, np.maximum(self.lo[a] - self.hi[b], self.lo[b] - self.hi[a]))
            ok = np.maximum(diam[a], diam[b]) <= ETA * np.linalg.norm(gap, axis=1)
            far.append(np.stack([a[ok], b[ok]], 1))
            a, b = a[~ok], b[~ok]
            la, lb = son[a, 0] < 0, son[b, 0] < 0
            near.append(np.stack([a[la & lb], b[la & lb]], 1))
            parts = []
            for i in range(2):
                for j in range(2):
                    m = ~(la & lb) & ~(la & (i == 1)) & ~(lb & (j == 1))
                    parts.append(np.stack([np.where(la, a, son[a, i])[m],
                                           np.where(lb, b, son[b, j])[m]], 1))
            a, b = np.concatenate(parts).T
        self.near = self._sorted(np.concatenate(near))
        self.far = self._sorted(np.concatenate(far))

    @staticmethod
    def _sorted(p):
        return p[np.lexsort((p[:, 1], p[:, 0]))]

    def pivots(self, rank):
        """At most `rank` indices of every cluster, the sons' pivots for inner clusters."""
        rng = np.random.default_rng(7)
        piv = [None] * self.nc
        for c in sorted(range(self.nc), key=lambda c: -self.depth[c]):
            rows = np.concatenate([piv[s] for s in self.sons[c]]) if self.sons[c] else self.idx[c]
            piv[c] = np.sort(rng.permutation(rows)[:rank])
        return piv


@functools.lru_cache(maxsize=None)
def _tree(spec, basis):
    return _Tree(spec, basis)


def _csr(lists):
    ptr = np.zeros(len(lists) + 1, np.int32)
    ptr[1:] = np.cumsum([len(x) for x in lists])
    return ptr, np.concatenate(lists).astype(np.int32)


@functools.lru_cache(maxsize=None)
def _lists(spec, basis, rank):
    """{"near", "far"}: (ptr, idx, blk_row, blk_col, blk_off, entries) over the index sets / pivots."""
    tree = _tree(spec, basis)
    got = {}
    for name, sets, pairs in (("near", tree.idx, tree.near), ("far", tree.pivots(rank), tree.far)):
        ptr, idx = _csr(sets)
        size = np.diff(ptr).astype(np.int64)
        n = size[pairs[:, 0]] * size[pairs[:, 1]]
        off = np.concatenate([[0], np.cumsum(n)])
        got[name] = (ptr, idx, pairs[:, 0].astype(np.int32), pairs[:, 1].astype(np.int32),
                     off[:-1].astype(np.int64), int(off[-1]))
    return got


def _entries(ptr, idx, row, col, off, n):
    """(rows, columns) of every entry of a block list, in the order of its output."""
    size = np.diff(ptr).astype(np.int64)
    nr = size[row]
    blk = np.repeat(np.arange(len(row)), nr * size[col])
    local = np.arange(n) - off[blk]
    return (idx[ptr[row][blk] + local % nr[blk]].astype(np.int64),
            idx[ptr[col][blk] + local // nr[blk]].astype(np.int64))


# ---------------------------------------------------------------------------
# What a user's program has in hand, and one pass
# ---------------------------------------------------------------------------
class _State:
    """A context with its meshes, plans and handles, released together."""

    def __init__(self, case, seed):
        self.case, self.seed = case, seed
        self.ctx = bem.Context(0)
        self.release = []

    def __del__(self):
        for f, *args in self.release:
            f(*args)
        self.ctx.close()


def _dev(a, dtype):
    return torch.as_tensor(np.ascontiguousarray(a)).to(device=DEVICE, dtype=dtype)


def _out(kernel, n):
    return torch.zeros(max(1, n), device=DEVICE, dtype=torch.complex128
                       if kernel in COMPLEX else torch.float64)


def _quad(case):
    s = case["singular"]
    return bem.quad_desc(case["q"], case["rule"], s, s, s, case["precision"],
                         "learned" if case["work"] == "learned" else "fixed")


def _kernel(case, kernel):
    return bem.kernel_desc(kernel, case["kappa"] if kernel.startswith("helm") else 0.0,
                           case["kappa"] if kernel == "helmholtz_bw" else 0.0)


def _jobs(case, mesh_ids):
    """Block jobs {"near", "far"} of all bodies and operators: both operators of a body share the
    lists, all bodies of an operator share one output."""
    bodies, kernels = case["mesh"].split("+"), case["kernels"].split("+")
    jobs, outs = {}, {}
    for part in ("near", "far"):
        lists = [_lists(b, case["basis"], case["rank"])[part] for b in bodies]
        total = sum(x[5] for x in lists)
        out = {k: _out(k, total) for k in kernels}
        at, jobs[part] = 0, []
        for m, (ptr, idx, row, col, off, n) in zip(mesh_ids, lists):
            p, i, r, c = (_dev(x, torch.int32) for x in (ptr, idx, row, col))
            o = _dev(off, torch.int64)
            jobs[part] += [bem.BlockJob(m, p, i, p, i, r, c, o, out[k][at:], _kernel(case, k),
                                        _quad(case)) for k in kernels]
            at += n
        outs.update({part + "_" + k: v for k, v in out.items()})
    return jobs, outs


def _order_model(ctx):
    """A ladder on the closest-vertex distance over the diameter: the further apart, the cheaper;
    about 230 points per disjoint pair on a jittered sphere, as with a trained model."""
    x0 = (3.2, 1.5, 0.3, -0.4, -1.0)   # log2 distances at which the next cheaper rule takes over
    w1, w2, w3 = np.zeros((64, 8)), np.zeros((64, 64)), np.zeros((6, 64))
    w1[0, 1], w1[1, 1] = 1.0, -1.0
    w2[0, 0] = w2[1, 1] = 1.0
    steep, b3 = 8.0, np.zeros(6)
    for c in range(5):
        w3[c, 0], w3[c, 1] = steep * (5 - c), -steep * (5 - c)
        b3[c] = -steep * sum(x0[c:])
    mlp = ctx.bem_mlp_create(0)
    ctx.bem_mlp_set_params(mlp, np.concatenate([w1.ravel(), np.zeros(64), w2.ravel(), np.zeros(64),
                                                w3.ravel(), b3]).astype(np.float32),
                           np.concatenate([np.zeros(8), np.ones(8)]).astype(np.float32))
    return mlp


def _green_inputs(case, seed):
    """Rows, box points, normals and factors of every cluster (4 x 4 Gauss points per face)."""
    tree = _tree(case["mesh"], case["basis"])
    piv = tree.pivots(case["rank"])
    ptr, rows = _csr([np.concatenate([piv[s] for s in tree.sons[c]]) if tree.sons[c]
                      else tree.idx[c] for c in range(tree.nc)])
    h = np.linalg.norm(tree.hi - tree.lo, axis=1) * (1 + 0.01 * np.random.default_rng(seed).random())
    lo, hi = tree.lo - 0.5 * h[:, None], tree.hi + 0.5 * h[:, None]
    g, w = np.polynomial.legendre.leggauss(4)
    z, nz, wt = [], [], []
    for axis in range(3):
        a, b = [d for d in range(3) if d != axis]
        u, t = (x.ravel() for x in np.meshgrid(g, g, indexing="ij"))
        for side in (-1, 1):
            p = np.zeros((tree.nc, 16, 3))
            p[:, :, axis] = (lo if side < 0 else hi)[:, axis, None]
            for d, x in ((a, u), (b, t)):
                p[:, :, d] = 0.5 * (lo + hi)[:, d, None] + 0.5 * (hi - lo)[:, d, None] * x
            n = np.zeros_like(p)
            n[:, :, axis] = side
            z.append(p)
            nz.append(n)
            wt.append(np.outer((hi - lo)[:, a] * (hi - lo)[:, b] / 4, np.outer(w, w).ravel()))
    wt = np.sqrt(np.concatenate(wt, 1))
    return {"row_ptr": ptr, "rows": rows, "pt_ptr": np.arange(tree.nc + 1, dtype=np.int32) * 96,
            "z": np.concatenate(z, 1).reshape(-1, 3), "nz": np.concatenate(nz, 1).reshape(-1, 3),
            "sp": wt.ravel(), "sm": (wt * h[:, None]).ravel(),
            "off": np.concatenate([[0], np.cumsum(192 * np.diff(ptr).astype(np.int64))])}


def _h2_inputs(case, seed):
    """The parts of an H2 matrix: bases with identity rows at the pivots, entries of the size of
    the one-point rule's, a vector."""
    spec, rank = case["mesh"], case["rank"]
    tree, lists = _tree(spec, "p0"), _lists(spec, "p0", rank)
    rng = np.random.default_rng(seed)
    piv = tree.pivots(rank)
    mats = []
    for c in range(tree.nc):
        rows = np.concatenate([piv[s] for s in tree.sons[c]]) if tree.sons[c] else tree.idx[c]
        m = rng.uniform(-0.2, 0.4, (len(rows), len(piv[c])))
        m[np.argsort(rows, kind="stable")[np.searchsorted(np.sort(rows), piv[c])]] = np.eye(len(piv[c]))
        mats.append(m)
    v, t = _mesh(spec, seed)
    mid = _dev(v[t].mean(1), torch.float64)
    size = 4 * math.pi / len(t)
    vals = {}
    for part in ("near", "far"):
        i, j = _h2_index(spec, rank, part)
        r = torch.linalg.vector_norm(mid[i] - mid[j], dim=1).clamp_min_(0.6 * math.sqrt(size))
        vals[part] = size * size / (4 * math.pi) / r
    x = _dev(rng.standard_normal(tree.n), torch.float64)
    return tree, piv, mats, lists, vals, x


@functools.lru_cache(maxsize=2)
def _h2_index(spec, rank, part):
    return tuple(_dev(x, torch.int64) for x in _entries(*_lists(spec, "p0", rank)[part]))


def prepare(case, seed):
    s = _State(case, seed)
    work = case["work"]
    ctx = s.ctx
    if work == "h2":
        tree, piv, mats, lists, s.vals, s.x = _h2_inputs(case, seed)
        pp, pi = _csr(piv)
        cp, ci = _csr(tree.idx)
        s.y = torch.zeros_like(s.x)
        s.h2 = ctx.bem_h2_create(tree.n, cp, ci, tree.son, pp, pi, mats, lists["near"][2:5],
                                 s.vals["near"], lists["far"][2:5], s.vals["far"])
        s.release.append((ctx.bem_h2_destroy, s.h2))
        return s
    meshes = [_mesh(b, seed + 101 * k) for k, b in enumerate(case["mesh"].split("+"))]
    if work == "upload":
        s.mesh = meshes[0]
        s.jobs, s.outs = _jobs(case, [0])
        return s
    ids = [ctx.bem_mesh_upload(v, t, case["basis"]) for v, t in meshes]
    s.mesh = ids[0]
    if work in ("dense", "solve"):
        n = len(meshes[0][1] if case["basis"] == "p0" else meshes[0][0])
        s.kernel, s.quad, s.out = _kernel(case, case["kernels"]), _quad(case), _out(case["kernels"], n * n)
        if work == "solve":
            ctx.bem_assemble_dense(ids[0], s.kernel, s.quad, 0, s.out)
            s.half_mass, s.rhs, s.points = (_dev(x, d) for x, d in _solve_inputs(case, seed))
            s.x = torch.zeros(n, dtype=torch.complex128, device=DEVICE)
            s.field = torch.zeros(len(s.points), dtype=torch.complex128, device=DEVICE)
    elif work in ("blocks", "plan", "learned"):
        s.jobs, s.outs = _jobs(case, ids)
        if work == "learned":
            mlp = _order_model(ctx)
            ctx.bem_set_order_model(mlp, 0.999)
        if work != "blocks":
            s.plan = ctx.bem_plan_create(s.jobs["near"], s.jobs["far"], bem.PLAN_GRAPH)
            s.release.append((ctx.bem_plan_destroy, s.plan))
        if work == "learned":
            s.release.append((ctx.bem_mlp_destroy, mlp))
    else:
        g = _green_inputs(case, seed)
        s.out = _out(case["kernels"], int(g["off"][-1]))
        f = {k: _dev(g[k], torch.float64) for k in ("z", "nz", "sp", "sm")}
        i = {k: _dev(g[k], torch.int32) for k in ("row_ptr", "rows", "pt_ptr")}
        s.job = bem.GreenJob(ids[0], i["row_ptr"], i["rows"], i["pt_ptr"], f["z"], f["nz"],
                             _dev(g["off"][:-1], torch.int64), s.out, f["sp"], f["sm"],
                             _kernel(case, case["kernels"]), case["rule"], case["q"])
    return s


def _solve_inputs(case, seed):
    """Half the mass matrix's diagonal, a point source's right-hand side (one-point rule), and
    points off the surface."""
    v, t = _mesh(case["mesh"].split("+")[0], seed)
    w = v[t]
    area = 0.5 * np.linalg.norm(np.cross(w[:, 1] - w[:, 0], w[:, 2] - w[:, 1]), axis=1)
    rng = np.random.default_rng(seed)
    centre = v.mean(0)
    r = np.linalg.norm(w.mean(1) - (centre + rng.uniform(-0.05, 0.05, 3)), axis=1)
    d = rng.standard_normal((case["points"], 3))
    z = centre + d / np.linalg.norm(d, axis=1, keepdims=True) * rng.uniform(2, 4, (len(d), 1))
    return ((0.5 * area + 0j, torch.complex128),
            (area * np.exp(1j * case["kappa"] * r) / (4 * np.pi * r), torch.complex128),
            (z, torch.float64))


def run(s):
    ctx, work = s.ctx, s.case["work"]
    if work == "dense":
        ctx.bem_assemble_dense(s.mesh, s.kernel, s.quad, 0, s.out)
        return s.out
    if work == "solve":
        ctx.bem_dense_gmres(s.out, s.rhs, s.x, diag=s.half_mass, tol=1e-10)
        ctx.bem_potentials(s.mesh, s.kernel, s.points, s.x, s.field)
        return {"density": s.x, "field": s.field}
    if work == "blocks":
        ctx.bem_near_field(s.jobs["near"])
        ctx.bem_coupling_blocks(s.jobs["far"])
        return s.outs
    if work == "upload":
        mesh = ctx.bem_mesh_upload(*s.mesh, s.case["basis"])
        for j in s.jobs["near"] + s.jobs["far"]:
            j.mesh_id = mesh
        ctx.bem_near_field(s.jobs["near"])
        ctx.bem_coupling_blocks(s.jobs["far"])
        ctx.bem_mesh_free(mesh)
        return s.outs
    if work in ("plan", "learned"):
        ctx.bem_plan_run(s.plan)
        return s.outs
    if work == "green":
        ctx.bem_green_matrices(s.job)
        return s.out
    ctx.bem_h2_matvec(s.h2, s.x, s.y)
    return s.y


# ---------------------------------------------------------------------------
# What a pass cannot do without
# ---------------------------------------------------------------------------
_FLOPS = {"laplace_slp": 11, "laplace_dlp": 13, "helmholtz_slp": 19, "helmholtz_dlp": 27,
          "helmholtz_bw": 31}   # per quadrature point: difference, distance, kernel, weighted sum


def work(case):
    kind, bodies = case["work"], case["mesh"].split("+")
    kernels = case["kernels"].split("+")
    nt = sum(len(_surface(b)[1]) for b in bodies)
    np2 = 7 if case["rule"] == "tri7" else case["q"] ** 2
    width = {k: 16 if k in COMPLEX else 8 for k in kernels}
    if kind == "h2":
        lists = _lists(bodies[0], "p0", case["rank"])
        n = lists["near"][5] + lists["far"][5]
        n += 2 * sum(len(i) * case["rank"] for i in _tree(bodies[0], "p0").idx if len(i) <= LEAF)
        return {"bytes": 8.0 * n + 16.0 * nt, "flops": 2.0 * n}
    if kind == "solve":   # about 28 products of the matrix, and the field
        return {"bytes": 16.0 * nt * nt + 32.0 * nt,
                "flops": 28 * 8.0 * nt * nt + 31.0 * case["points"] * nt * 16}
    if kind == "green":
        g = _green_inputs(case, 0)
        n, per = int(g["off"][-1]), 6 if case["basis"] == "p1" else 1
        return {"bytes": n * width[kernels[0]] + 64.0 * len(g["sp"]) + 52.0 * nt,
                "flops": n / 2 * per * np2 * (_FLOPS[kernels[0]] + 8.0)}
    if kind == "dense":
        n = (nt if case["basis"] == "p0" else len(_surface(bodies[0])[0])) ** 2
        index = 0
    else:
        lists = [x for b in bodies for x in _lists(b, case["basis"], case["rank"]).values()]
        n = sum(x[5] for x in lists)
        index = sum(4.0 * len(x[1]) + 16.0 * len(x[2]) for x in lists)
    # triangle pairs per entry: the 36 pairs of two vertices' supports, shared by 9 neighbours in
    # the dense matrix and the near field
    pairs = float(n)
    if case["basis"] == "p1":
        near = n if kind == "dense" else sum(_lists(b, "p1", case["rank"])["near"][5] for b in bodies)
        pairs = 4.0 * near + 36.0 * (n - near)
    points = 49 if kind == "learned" else np2 * np2
    return {"bytes": n * float(sum(width.values())) + index + 52.0 * nt,
            "flops": pairs * points * sum(_FLOPS[k] for k in kernels)}


# ---------------------------------------------------------------------------
# The same in 64 bits
# ---------------------------------------------------------------------------
def _gauss(q):
    x, w = np.polynomial.legendre.leggauss(q)
    return 0.5 + 0.5 * x, 0.5 * w


def _rule2(rule, q):
    """(s, t, w) on {0 <= t <= s <= 1}: Duffy's product rule, or Radon's 7 points."""
    if rule == "duffy":
        g, w = _gauss(q)
        return np.repeat(g, q), np.outer(g, g).ravel(), np.outer(w * g, w).ravel()
    r = math.sqrt(15.0)
    bary, weight = [(1 / 3, 1 / 3)], [9 / 80]
    for p, w in (((6 - r) / 21, (155 - r) / 2400), ((6 + r) / 21, (155 + r) / 2400)):
        bary += [(p, p), (1 - 2 * p, p), (p, 1 - 2 * p)]
        weight += [w] * 3
    b = np.array(bary)
    return b.sum(1), b[:, 1], np.array(weight)


def _rule4(shared, q):
    """Sauter-Schwab rule (x1, x2, y1, y2, x1 - y1, x2 - y2, w) for pairs sharing 1, 2, 3 vertices."""
    g, w = _gauss(q)
    xi, a, b, c = (x.ravel() for x in np.meshgrid(g, g, g, g, indexing="ij"))
    wt = np.einsum("i,j,k,l->ijkl", w, w, w, w).ravel() * xi ** 3
    one = np.ones_like(xi)
    if shared == 1:   # x = (1, a), y = (b, b c)
        parts = [(a, b, b * c, 1 - b, a - b * c, b)]
    elif shared == 2:   # x = (1, u), y = (1 - p, r): cones from u = p = r = 0
        parts = [(u, 1 - p, r, p, u - r, j) for u, p, r, j in (
            (a, a * b * (1 - c), a * b * c, a * a * b), (a * b, a * c, a * (1 - c), a * a))]
    else:   # x = (1, u), y = (1 - p, u - r): cones from p = r = 0
        parts = [(u, 1 - p, u - r, p, r, a * (1 - a)) for p, r, u in (
            (a * b, a, a + (1 - a) * c), (a, a * b, a * b + (1 - a) * c),
            (a * (1 - b), -a * b, (1 - a) * c))]
    got = []
    for x2, y1, y2, d1, d2, j in parts:
        got.append(np.stack([xi * one, xi * x2, xi * y1, xi * y2, xi * d1, xi * d2, wt * j]))
        got.append(np.stack([xi * y1, xi * y2, xi * one, xi * x2, -xi * d1, -xi * d2, wt * j]))
    return np.concatenate(got, 1)


def _values(kernel, kappa, r2, height):
    """4 pi k(x, y) from |x - y|^2 and (x - y) . n_y."""
    r = r2.sqrt()
    if kernel == "laplace_slp":
        return 1 / r
    if kernel == "laplace_dlp":
        return height / (r2 * r)
    wave = torch.polar(1 / r, kappa * r)
    if kernel == "helmholtz_slp":
        return wave
    double = wave * torch.complex(height / r2, -kappa * height / r)
    return double - 1j * kappa * wave if kernel == "helmholtz_bw" else double


class _Exact:
    """Integrals over pairs of triangles of one mesh."""

    def __init__(self, v, t):
        self.t = _dev(t, torch.int64)
        self.v = _dev(v, torch.float64)[self.t]
        n = torch.linalg.cross(self.v[:, 1] - self.v[:, 0], self.v[:, 2] - self.v[:, 1])
        self.gram = torch.linalg.vector_norm(n, dim=1)
        self.normal = n / self.gram[:, None]

    @staticmethod
    def _hat(local, s, t):
        """Hat function of the vertex at position `local` (n,) at the points (s, t)."""
        h = torch.stack([1 - s, s - t, t])
        return h[local]

    def pairs(self, case, kernels, a, b, la=None, lb=None):
        """One tensor per kernel: the integral over triangles a x b (n,), times the hats la, lb."""
        share = (self.t[a][:, :, None] == self.t[b][:, None, :])
        count = share.sum((1, 2))
        outs = [torch.zeros(len(a), device=DEVICE, dtype=torch.complex128
                            if k in COMPLEX else torch.float64) for k in kernels]
        for shared in range(4):
            at = torch.nonzero(count == shared)[:, 0]
            points = len(_rule2(case["rule"], case["q"])[0]) ** 2 if shared == 0 else \
                (2, 4, 6)[shared - 1] * case["singular"] ** 4
            for part in torch.split(at, max(1, (1 << 25) // points)):
                if len(part):
                    self._some(case, kernels, shared, part, a[part], b[part],
                               None if la is None else la[part], None if lb is None else lb[part],
                               share[part], outs)
        return outs

    def _some(self, case, kernels, shared, part, a, b, la, lb, share, outs):
        va, vb, n = self.v[a], self.v[b], self.normal[b]
        rows = torch.arange(len(a), device=DEVICE)
        if shared == 0:
            s, t, w = (_dev(x, torch.float64) for x in _rule2(case["rule"], case["q"]))

            def mapped(v):
                return (v[:, :1] - vb[:, :1] + s[None, :, None] * (v[:, 1] - v[:, 0])[:, None]
                        + t[None, :, None] * (v[:, 2] - v[:, 1])[:, None])

            x, y = mapped(va), mapped(vb)
            height = torch.einsum("npc,nc->np", x, n)[:, :, None]
            r2 = 0
            for c in range(3):
                r2 = r2 + (x[:, :, None, c] - y[:, None, :, c]) ** 2
            wx = w if la is None else w * self._hat(la, s, t)
            wy = w if lb is None else w * self._hat(lb, s, t)
        else:
            if shared == 3:
                pa = pb = torch.arange(3, device=DEVICE).expand(len(a), 3)
            else:   # the shared vertex, or the shared edge in a's direction, first
                hit = share.any(2)
                first = hit.to(torch.int64).argmax(1)
                if shared == 2:
                    first = torch.where(hit[rows, first] & hit[rows, (first + 1) % 3], first, (first + 2) % 3)
                pa = (first[:, None] + torch.arange(3, device=DEVICE)) % 3
                pb0 = share[rows, first].to(torch.int64).argmax(1)
                pb1 = share[rows, pa[:, 1]].to(torch.int64).argmax(1) if shared == 2 else (pb0 + 1) % 3
                pb = torch.stack([pb0, pb1, 3 - pb0 - pb1], 1)
            x1, x2, y1, y2, d1, d2, w = (_dev(r, torch.float64) for r in _rule4(shared, case["singular"]))
            va, vb = va[rows[:, None], pa], vb[rows[:, None], pb]
            e1a, e2a = va[:, 1] - va[:, 0], va[:, 2] - va[:, 1]
            e1b, e2b = vb[:, 1] - vb[:, 0], vb[:, 2] - vb[:, 1]
            r2, height = 0, 0
            h1, h2 = ((e * n).sum(1, keepdim=True) for e in (e1a, e2a))
            height = torch.zeros(len(a), 1, device=DEVICE, dtype=torch.float64) if shared == 3 else \
                x2 * h2 if shared == 2 else x1 * h1 + x2 * h2
            for c in range(3):
                p, q, r, u = (e[:, c, None] for e in (e1a, e2a, e1b, e2b))
                d = d1 * p + d2 * q if shared == 3 else d1 * p + x2 * q - y2 * u if shared == 2 else \
                    x1 * p + x2 * q - y1 * r - y2 * u
                r2 = r2 + d * d
            wx = w
            if la is not None:
                la = (pa == la[:, None]).to(torch.int64).argmax(1)
                lb = (pb == lb[:, None]).to(torch.int64).argmax(1)
                wx = w * self._hat(la, x1, x2) * self._hat(lb, y1, y2)
        scale = self.gram[a] * self.gram[b] / (4 * math.pi)
        for out, k in zip(outs, kernels):
            val = _values(k, case["kappa"], r2, height)
            if shared == 0:
                val = (val * (wy if wy.dim() == 1 else wy[:, None, :])).sum(2)
            out[part] = (val * wx).sum(1) * scale

    def entries(self, case, kernels, rows, cols):
        """Matrix entries of one mesh, one tensor per kernel."""
        rows, cols = _dev(rows, torch.int64), _dev(cols, torch.int64)
        if case["basis"] == "p0":
            step = 1 << 24
            got = [self.pairs(case, kernels, r, c) for r, c in zip(rows.split(step), cols.split(step))]
            return [torch.cat(g) for g in zip(*got)]
        flat = self.t.reshape(-1)
        order = torch.argsort(flat, stable=True)
        deg = torch.bincount(flat)
        start = torch.cumsum(deg, 0) - deg
        outs = [torch.zeros(len(rows), device=DEVICE, dtype=torch.complex128
                            if k in COMPLEX else torch.float64) for k in kernels]
        for lo in range(0, len(rows), 1 << 19):
            i, j = rows[lo:lo + (1 << 19)], cols[lo:lo + (1 << 19)]
            n = deg[i] * deg[j]
            e = torch.repeat_interleave(torch.arange(len(i), device=DEVICE), n)
            local = torch.arange(len(e), device=DEVICE) - (torch.cumsum(n, 0) - n)[e]
            a = order[start[i[e]] + local // deg[j[e]]]
            b = order[start[j[e]] + local % deg[j[e]]]
            vals = self.pairs(case, kernels, a // 3, b // 3, a % 3, b % 3)
            for out, v in zip(outs, vals):
                out[lo:lo + len(i)].index_add_(0, e, v)
        return outs


def _exact_dense(case, seed):
    v, t = _mesh(case["mesh"], seed)
    n = len(t if case["basis"] == "p0" else v)
    return _Exact(v, t).entries(case, [case["kernels"]], np.tile(np.arange(n), n),
                                np.repeat(np.arange(n), n))[0]


def _exact_green(case, seed):
    v, t = _mesh(case["mesh"], seed)
    E, g = _Exact(v, t), _green_inputs(case, seed)
    s, tt, w = (_dev(x, torch.float64) for x in _rule2(case["rule"], case["q"]))
    helm = case["kernels"] == "helmholtz_slp"
    x = (E.v[:, :1] + s[None, :, None] * (E.v[:, 1] - E.v[:, 0])[:, None]
         + tt[None, :, None] * (E.v[:, 2] - E.v[:, 1])[:, None])
    n_of, size = np.diff(g["row_ptr"]), int(g["off"][-1])
    z, nz, sp, sm = (_dev(g[k], torch.float64) for k in ("z", "nz", "sp", "sm"))
    out = torch.zeros(size, device=DEVICE, dtype=torch.complex128 if helm else torch.float64)
    c = np.repeat(np.arange(len(n_of)), n_of)
    row, k = g["rows"].astype(np.int64), np.arange(len(g["rows"])) - g["row_ptr"][c]
    if case["basis"] == "p0":
        tri, src, weight = row, np.arange(len(row)), (w * E.gram[:, None])[:, None]
        local = np.zeros(len(row), np.int64)
    else:
        order = np.argsort(t.ravel(), kind="stable")
        deg = np.bincount(t.ravel())
        src = np.repeat(np.arange(len(row)), deg[row])
        at = np.arange(len(src)) - np.repeat(np.cumsum(deg[row]) - deg[row], deg[row])
        tri, local = np.divmod(order[(np.cumsum(deg) - deg)[row[src]] + at], 3)
        weight = torch.stack([1 - s, s - tt, tt])[None] * (w * E.gram[:, None])[:, None]
    for part in np.array_split(np.arange(len(src)), max(1, len(src) // 20000)):
        p = _dev(c[src[part]][:, None] * 96 + np.arange(96), torch.int64)
        T = _dev(tri[part], torch.int64)
        d = x[T][:, None] - z[p][:, :, None]
        r2 = (d * d).sum(3)
        wt = weight[T, _dev(local[part], torch.int64)][:, None]
        dn = torch.einsum("nmqc,nmc->nmq", d, nz[p])
        plus = _values(case["kernels"], case["kappa"], r2, dn)
        minus = _values("helmholtz_dlp" if helm else "laplace_dlp", case["kappa"], r2, dn)
        at = _dev((g["off"][c] + k)[src[part]][:, None] + np.arange(96) * n_of[c[src[part]]][:, None],
                  torch.int64)
        skip = _dev(96 * n_of[c[src[part]]][:, None], torch.int64)
        for val, f, o in ((plus, sp, at), (minus, sm, at + skip)):
            out.index_put_((o.reshape(-1),), ((val * wt).sum(2) * f[p] / (4 * math.pi)).reshape(-1),
                           accumulate=True)
    return out


def _exact_h2(case, seed):
    tree, piv, mats, lists, vals, x = _h2_inputs(case, seed)
    hat, y = [None] * tree.nc, torch.zeros_like(x)
    i, j = _h2_index(case["mesh"], case["rank"], "near")
    y.index_add_(0, i, vals["near"] * x[j])
    xh, y = x.cpu().numpy(), y.cpu().numpy()
    deepest = sorted(range(tree.nc), key=lambda c: -tree.depth[c])
    for c in deepest:
        v = np.concatenate([hat[s] for s in tree.sons[c]]) if tree.sons[c] else xh[tree.idx[c]]
        hat[c] = mats[c].T @ v
    at = np.concatenate([[0], np.cumsum([len(p) for p in piv])])
    ptr, _, row, col, off, n = lists["far"]
    i, j = (_dev(a, torch.int64) for a in _entries(ptr, np.arange(at[-1], dtype=np.int32), row, col,
                                                   off, n))
    yh = torch.zeros(int(at[-1]), device=DEVICE, dtype=torch.float64)
    yh = yh.index_add_(0, i, vals["far"] * _dev(np.concatenate(hat), torch.float64)[j]).cpu().numpy()
    for c in reversed(deepest):
        up = mats[c] @ yh[at[c]:at[c + 1]]
        for s in tree.sons[c]:
            yh[at[s]:at[s + 1]] += up[:len(piv[s])]
            up = up[len(piv[s]):]
        if not tree.sons[c]:
            y[tree.idx[c]] += up
    return _dev(y, torch.float64)


def exact(case, seed):
    kind, kernels = case["work"], case["kernels"].split("+")
    if kind == "learned":   # the order model works in 16 bits
        return None
    if kind == "dense":
        return _exact_dense(case, seed)
    if kind == "green":
        return _exact_green(case, seed)
    if kind == "h2":
        return _exact_h2(case, seed)
    if kind == "solve":
        A = _exact_dense(case, seed)
        mass, rhs, z = (_dev(x, d) for x, d in _solve_inputs(case, seed))
        n = len(mass)
        x = torch.linalg.solve(A.reshape(n, n).T + torch.diag(mass), rhs)
        E = _Exact(*_mesh(case["mesh"], seed))
        s, t, w = (_dev(p, torch.float64) for p in _rule2("duffy", 4))
        y = (E.v[:, :1] + s[None, :, None] * (E.v[:, 1] - E.v[:, 0])[:, None]
             + t[None, :, None] * (E.v[:, 2] - E.v[:, 1])[:, None])
        field = []
        for p in z:
            d = p - y
            k = _values("helmholtz_bw", case["kappa"], (d * d).sum(2),
                        torch.einsum("nqc,nc->nq", d, E.normal))
            field.append(((k * w).sum(1) * E.gram / (4 * math.pi) * x).sum())
        return {"density": x, "field": torch.stack(field)}
    outs = {}
    for part in ("near", "far"):
        got = []
        for b, body in enumerate(case["mesh"].split("+")):
            v, t = _mesh(body, seed + 101 * b)
            got.append(_Exact(v, t).entries(case, kernels, *_entries(*_lists(body, case["basis"],
                                                                             case["rank"])[part])))
        outs.update({part + "_" + k: torch.cat(v) for k, v in zip(kernels, zip(*got))})
    return outs
