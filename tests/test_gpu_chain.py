"""GPU: launches that overlap in one stream, and the support records of the
piecewise-linear engine.

- Calls in a row without a synchronisation between them, each overwriting the
  touching table and the tile prefix sums that the one before still reads, give
  the bits of the same calls with a synchronisation after each; so does a plan
  of the same jobs, run twice, with and without a graph.
- Clusters of 1, 31, 32, 33 and 40 vertices in shuffled order over a bipyramid
  whose apexes have the largest degree (16): blocks of the single call and of a
  plan against the entry kernel, which takes no supports.  Both are FP64 sums of
  the same at most 16 * 16 * 6 * 5^4 terms of one sign (single layer): 1e-11 of
  the entry bounds their rounding."""
import numpy as np
import pytest

import synth
from parity_util import block_job, to_dev
from test_gpu_h2 import env  # noqa: F401  (fixture)

pytestmark = pytest.mark.gpu

QUAD = dict(q_regular=3, regular_rule="duffy", q_identical=5, q_edge=4, q_vertex=3)


def _all_pairs(ptr, idx):
    nc = len(ptr) - 1
    t, s = (a.ravel().astype(np.int32) for a in np.meshgrid(np.arange(nc), np.arange(nc), indexing="ij"))
    size = np.diff(ptr)[t].astype(np.int64) * np.diff(ptr)[s]
    off = np.concatenate([[0], np.cumsum(size)]).astype(np.int64)
    return synth.workloads.BlockSet(ptr, idx, ptr, idx, t, s, off[:-1], int(off[-1]))


@pytest.mark.parametrize("basis,precision", [("p0", "fp64"), ("p0", "mixed_full"), ("p1", "fp64"), ("p1", "mixed_full")])
def test_calls_in_a_row(env, basis, precision):  # noqa: F811
    import torch
    pkg, ctx = env
    mesh = synth.jitter(synth.icosphere(2), 0.05, 5)
    n = mesh.nt if basis == "p0" else mesh.nv
    cuts = np.unique(np.concatenate([np.arange(0, n, 29), [n]])).astype(np.int32)
    bs = _all_pairs(cuts, np.random.default_rng(2).permutation(n).astype(np.int32))
    mid = ctx.bem_mesh_upload(mesh.verts, mesh.tris, basis)
    kinds = ["laplace_slp", "laplace_dlp", "laplace_slp", "laplace_dlp"]
    quads = [dict(QUAD, precision=precision), dict(QUAD, precision=precision, q_regular=2)]

    def jobs():
        return [block_job(pkg, mid, bs, k, 0.0, quads[i // 2],
                          torch.zeros(bs.n_entries, dtype=torch.float64, device="cuda"))
                for i, k in enumerate(kinds)]

    alone, row = jobs(), jobs()
    for j in alone:
        ctx.bem_near_field([j])
        ctx.bem_sync()
    for _ in range(3):
        for j in row:
            ctx.bem_near_field([j])
    ctx.bem_sync()
    for a, b in zip(alone, row):
        assert torch.equal(a.out, b.out)
    for flags in (0, pkg.PLAN_GRAPH):
        planned = jobs()
        plan = ctx.bem_plan_create(planned, [], flags)
        for _ in range(2):
            for j in planned:
                j.out.zero_()
            torch.cuda.synchronize()
            ctx.bem_plan_run(plan)
            ctx.bem_plan_run(plan)
            ctx.bem_sync()
            for a, b in zip(alone, planned):
                assert torch.equal(a.out, b.out)
        ctx.bem_plan_destroy(plan)
    ctx.bem_mesh_free(mid)


@pytest.mark.parametrize("planned", [False, True])
def test_supports(env, planned):  # noqa: F811
    import torch
    pkg, ctx = env
    a = 2.0 * np.pi * np.arange(16) / 16.0
    levels = [(0.6, -0.5), (1.0, 0.0), (0.7, 0.45)]
    verts = [[r * np.cos(x), r * np.sin(x), z] for r, z in levels for x in a] + [[0, 0, -0.9], [0, 0, 0.8]]
    tris = []
    for k in range(16):
        m = (k + 1) % 16
        tris += [[48, m, k], [49, 32 + k, 32 + m]]
        for l in (0, 16):
            tris += [[l + k, l + m, l + 16 + m], [l + k, l + 16 + m, l + 16 + k]]
    verts, tris = np.array(verts, np.float64), np.array(tris, np.int32)
    rng = np.random.default_rng(9)
    sets = [rng.permutation(50)[:k] for k in (1, 31, 32, 33, 40)] + [np.array([49, 48])]
    ptr = np.concatenate([[0], np.cumsum([len(s) for s in sets])]).astype(np.int32)
    bs = _all_pairs(ptr, np.concatenate(sets).astype(np.int32))
    mid = ctx.bem_mesh_upload(verts, tris, "p1")
    out = torch.zeros(bs.n_entries, dtype=torch.float64, device="cuda")
    job = block_job(pkg, mid, bs, "laplace_slp", 0.0, QUAD, out)
    if planned:
        plan = ctx.bem_plan_create([job], [], pkg.PLAN_GRAPH)
        ctx.bem_plan_run(plan)
        ctx.bem_sync()
        ctx.bem_plan_destroy(plan)
    else:
        ctx.bem_near_field([job])
    rows, cols = bs.entry_indices()
    ref = torch.zeros_like(out)
    ctx.bem_pivot_entries(mid, pkg.kernel_desc("laplace_slp", 0.0), pkg.quad_desc(**QUAD),
                          to_dev(rows, torch.int32), to_dev(cols, torch.int32), ref)
    ctx.bem_sync()
    ctx.bem_mesh_free(mid)
    assert float(ref.min()) > 0.0
    assert float(((out - ref).abs() / ref).max()) <= 1e-11


@pytest.mark.parametrize("sizes", [
    [1] * 90,                                   # many blocks of one entry
    [3, 0, 0, 5, 1, 0, 17, 0, 2, 33, 0, 0],     # empty blocks between, and at the end
    [0] * 40 + [7] + [0] * 70 + [9, 40],        # runs of empty blocks longer than a window
    [320],                                      # one block
    [16, 16, 31, 32, 33, 64],
])
def test_flat_entries(env, sizes):  # noqa: F811
    """Entries of block lists with small, empty and large blocks, taken by a
    single call and by a plan, against the entry kernel: both are FP64 forms of
    the same sums (81 terms of one sign, or one touching rule), 1e-11 of the entry."""
    import torch
    pkg, ctx = env
    mesh = synth.jitter(synth.icosphere(2), 0.05, 7)
    rng = np.random.default_rng(len(sizes))
    ptr = np.concatenate([[0], np.cumsum(sizes)]).astype(np.int32)
    idx = rng.integers(0, mesh.nt, ptr[-1]).astype(np.int32)
    bs = _all_pairs(ptr, idx)
    mid = ctx.bem_mesh_upload(mesh.verts, mesh.tris, "p0")
    outs = [torch.zeros(bs.n_entries, dtype=torch.float64, device="cuda") for _ in range(2)]
    jobs = [block_job(pkg, mid, bs, "laplace_slp", 0.0, QUAD, o) for o in outs]
    ctx.bem_near_field([jobs[0]])
    plan = ctx.bem_plan_create([jobs[1]], [], pkg.PLAN_GRAPH)
    ctx.bem_plan_run(plan)
    ctx.bem_sync()
    ctx.bem_plan_destroy(plan)
    rows, cols = bs.entry_indices()
    ref = torch.zeros_like(outs[0])
    ctx.bem_pivot_entries(mid, pkg.kernel_desc("laplace_slp", 0.0), pkg.quad_desc(**QUAD),
                          to_dev(rows, torch.int32), to_dev(cols, torch.int32), ref)
    ctx.bem_sync()
    ctx.bem_mesh_free(mid)
    for o in outs:
        assert float(((o - ref).abs() / ref).max()) <= 1e-11


@pytest.mark.parametrize("n", [1, 31, 33, 70, 257])
@pytest.mark.parametrize("restart", [1, 3, 40])
def test_gmres_sizes(env, n, restart):  # noqa: F811
    """Dense GMRES at sizes around the kernels' tiles (32 rows, 64 columns) and at
    restarts after one, a few and all steps, against a direct solve.  |A - 3 I| is
    below 0.5 in the spectral norm, so the condition number is below 1.5 and a
    residual of 1e-12 bounds the error by 1.5e-12 of |x|."""
    import torch
    pkg, ctx = env
    rng = np.random.default_rng(n)
    A = rng.standard_normal((n, n)) + 1j * rng.standard_normal((n, n))
    A = 3.0 * np.eye(n) + 0.45 * A / np.linalg.norm(A, 2)
    b = rng.standard_normal(n) + 1j * rng.standard_normal(n)
    x = torch.empty(n, dtype=torch.complex128, device="cuda")
    it, res = ctx.bem_dense_gmres(to_dev(A.T.ravel(), torch.complex128), to_dev(b, torch.complex128), x,
                                  tol=1e-12, restart=restart, maxit=200)
    ref = np.linalg.solve(A, b)
    assert res <= 1e-12 and 0 < it < 200
    assert np.linalg.norm(x.cpu().numpy() - ref) <= 3e-12 * np.linalg.norm(ref)
    _, res = ctx.bem_dense_gmres(to_dev(A.T.ravel(), torch.complex128), to_dev(b, torch.complex128), x,
                                 tol=1e-300, restart=restart, maxit=2)
    assert np.isfinite(x.cpu().numpy()).all()


def test_guard_splits(env):  # noqa: F811
    """The double layer's guard over one block, 400 blocks and 65536 blocks of the same
    entries (all warps in a block, a few, one): every entry has the same bits, since
    the row maxima, and so the entries that are recomputed, are the same."""
    import torch
    pkg, ctx = env
    mesh = synth.jitter(synth.icosphere(3), 0.05, 8)
    n = mesh.nt
    idx = np.random.default_rng(4).permutation(n).astype(np.int32)
    mid = ctx.bem_mesh_upload(mesh.verts, mesh.tris, "p0")
    quad = dict(QUAD, precision="mixed_full")
    mats = []
    for size in (n, n // 20, n // 256):
        bs = _all_pairs(np.arange(0, n + 1, size, dtype=np.int32), idx)
        out = torch.zeros(bs.n_entries, dtype=torch.float64, device="cuda")
        ctx.bem_near_field([block_job(pkg, mid, bs, "laplace_dlp", 0.0, quad, out)])
        ctx.bem_sync()
        rows, cols = bs.entry_indices()
        mat = np.empty((n, n))
        mat[rows, cols] = out.cpu().numpy()
        mats.append(mat)
    ctx.bem_mesh_free(mid)
    assert np.isfinite(mats[0]).all() and np.abs(mats[0]).max() > 0.0
    assert np.array_equal(mats[0], mats[1]) and np.array_equal(mats[0], mats[2])
