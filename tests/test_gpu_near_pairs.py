"""GPU: disjoint pairs in the FP64 form, one block each, whose nearest points are
4, 8 or 16 times closer than the pair's extent and lie in the trial plane, so
that the largest values of 1/r^3 take the smallest heights.  Against the oracle,
relative to the sum of the magnitudes of an entry's terms.

Tolerance 6 b 2^-53 for an extent S of at most b distances: coordinate
differences of up to S are rounded to 2^-53 S, 1/r^3 takes three times the
relative error of r, and both sides carry it."""
import numpy as np
import pytest

import oracle
from parity_util import to_dev
from test_gpu_h2 import env  # noqa: F401  (fixture)

pytestmark = pytest.mark.gpu


def _pairs(n, near, seed):
    """Triangle pairs (2 k, 2 k + 1), test and trial, with S / r in (near / 2, near]."""
    rng = np.random.default_rng(seed)
    x = 0.5 + 0.5 * np.polynomial.legendre.leggauss(3)[0]
    s, t = np.repeat(x, 3)[:, None], np.outer(x, x).ravel()[:, None]
    out = []
    for _ in range(100 * n):
        B = np.array([[0, 0, 0], [1, 0, 0], [0.3, 0.8, 0]]) + np.c_[rng.uniform(-0.15, 0.15, (3, 2)), np.zeros(3)]
        k = rng.integers(3)
        away = B[k] - B.mean(0)
        away /= np.linalg.norm(away)
        A = np.array([B[k] + rng.uniform(0.002, 2.0 / near) * away] * 3)
        for j in (1, 2):
            A[j] += (rng.uniform(0.3, 1.0) * away + np.r_[rng.uniform(-0.5, 0.5, 2), 0.0]
                     + [0.0, 0.0, rng.uniform(0.1, 0.8)])
        A = np.roll(A, rng.integers(3), 0)
        if np.linalg.norm(np.cross(A[1] - A[0], A[2] - A[1])) < 0.05:
            continue
        p, q = (v[0] + s * (v[1] - v[0]) + t * (v[2] - v[1]) for v in (A, B))
        r = np.linalg.norm(p[:, None] - q[None], axis=2).min()
        size = (np.abs(A - B[0]).max(0) + np.abs(B - B[0]).max(0)).max()
        if near / 2 < 2.0 ** np.ceil(np.log2(size)) / r <= near:
            out += [A, B]
        if len(out) == 2 * n:
            break
    v = np.array(out).reshape(-1, 3)
    return v, np.arange(len(v), dtype=np.int32).reshape(-1, 3)


@pytest.mark.parametrize("near", [4, 8, 16])
@pytest.mark.parametrize("kernel", ["laplace_slp", "laplace_dlp", "helmholtz_dlp"])
@pytest.mark.parametrize("basis", ["p0", "p1"])
def test_near_pairs(env, basis, kernel, near):  # noqa: F811
    import torch
    pkg, ctx = env
    kappa = 3.0 if kernel.startswith("helmholtz") else 0.0
    quad = dict(q_regular=3, regular_rule="duffy", q_identical=3, q_edge=3, q_vertex=3)
    v, tris = _pairs(200, near, near)
    n = len(tris) // 2
    assert n == 200
    mid = ctx.bem_mesh_upload(v, tris, basis)
    side = 1 if basis == "p0" else 3
    ptr, idx = side * np.arange(2 * n + 1), np.arange(2 * n * side)
    out = torch.zeros(n * side * side, dtype=torch.complex128 if kappa else torch.float64, device="cuda")
    d = lambda a: to_dev(a, torch.int32)  # noqa: E731
    ctx.bem_near_field([pkg.BlockJob(mid, d(ptr), d(idx), d(ptr), d(idx), d(2 * np.arange(n)),
                                     d(2 * np.arange(n) + 1), to_dev(np.arange(n) * side * side, torch.int64),
                                     out, kernel=pkg.kernel_desc(kernel, kappa), quad=pkg.quad_desc(**quad))])
    ctx.bem_sync()
    ctx.bem_mesh_free(mid)
    k, c, r = np.meshgrid(np.arange(n), np.arange(side), np.arange(side), indexing="ij")
    rows, cols = (2 * k * side + r).ravel(), ((2 * k + 1) * side + c).ravel()
    kw = dict(kernel=kernel, kappa=kappa, basis=basis, **quad)
    ref = oracle.entries(v, tris, rows, cols, **kw)
    A = oracle.entries_absolute(v, tris, rows, cols, **kw)
    err = np.abs(out.cpu().numpy() - (ref if kappa else ref.real)) / A
    assert err.max() < 6 * near * 2.0 ** -53, err.max()


@pytest.mark.parametrize("length", [3.0, 100.0])
def test_plan_of_stretched_triangles(env, length):  # noqa: F811
    """Both piecewise-linear Laplace layers of a plan, fused, have the bits of single calls where
    most pairs are out of the fixed-point range, and where none is."""
    import torch
    import synth
    from parity_util import block_job
    pkg, ctx = env
    m = synth.jitter(synth.torus(9, 5), 0.05, 5)
    bs = synth.workloads.h2_blocks(m, "p1")[1]
    mid = ctx.bem_mesh_upload(np.array(m.verts) * [1.0, length, 1.0], m.tris, "p1")
    quad = dict(q_regular=3, q_identical=3, q_edge=3, q_vertex=3)

    def jobs():
        return [block_job(pkg, mid, bs, k, 0.0, quad, torch.zeros(bs.n_entries, dtype=torch.float64, device="cuda"))
                for k in ("laplace_slp", "laplace_dlp")]

    planned, single = jobs(), jobs()
    plan = ctx.bem_plan_create(planned, [], pkg.PLAN_GRAPH)
    ctx.bem_plan_run(plan)
    for j in single:
        ctx.bem_near_field([j])
    ctx.bem_sync()
    for a, b in zip(planned, single):
        assert torch.equal(a.out, b.out)
    ctx.bem_plan_destroy(plan)
    ctx.bem_mesh_free(mid)
