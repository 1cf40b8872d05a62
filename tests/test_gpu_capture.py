"""GPU: calls captured into a CUDA graph by the caller and replayed later.

- Potentials: a captured call holds no scratch of the library's, so it replays
  with the eager call's bits after a solve has grown (and replaced) the solver's
  scratch.  Also against numpy for 1 to 1300 points, which changes the CTAs per
  point; tolerance 1e-12 of the sum of the terms' magnitudes (320 terms of 16
  points, each rounded to a few 2^-53).
- A dense FP64 matrix after a call in a float form (Laplace kernels) or of the
  entry kernel (Helmholtz): the singular rules that the first call loaded serve
  the second, which then allocates nothing."""
import numpy as np
import pytest

import synth
from parity_util import to_dev

pytestmark = pytest.mark.gpu


@pytest.fixture()
def env():
    import torch
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    import __graft_entry__
    __graft_entry__.build()
    import paper_1510_07244_gb300 as pkg
    stream = torch.cuda.Stream()
    ctx = pkg.Context(0, stream)
    yield pkg, ctx, stream
    ctx.close()


def _solve(ctx, n):
    import torch
    rng = np.random.default_rng(n)
    A = np.eye(n) + 0.1 / n * rng.standard_normal((n, n))
    b = rng.standard_normal(n) + 0j
    x = torch.empty(n, dtype=torch.complex128, device="cuda")
    ctx.bem_dense_gmres(to_dev(A.T.ravel() + 0j, torch.complex128), to_dev(b, torch.complex128), x,
                        tol=1e-10, restart=30)
    return np.abs(x.cpu().numpy() - np.linalg.solve(A, b)).max()


@pytest.mark.parametrize("points", [1, 40, 1300])
def test_potentials(env, points):
    import torch
    pkg, ctx, stream = env
    mesh = synth.jitter(synth.icosphere(2), 0.05, 91)
    rng = np.random.default_rng(points)
    w = rng.standard_normal(mesh.nt) + 1j * rng.standard_normal(mesh.nt)
    d = rng.standard_normal((points, 3))
    z = d / np.linalg.norm(d, axis=1)[:, None] * rng.uniform(1.6, 3.0, points)[:, None]
    mid = ctx.bem_mesh_upload(mesh.verts, mesh.tris, "p0")
    zd, wd = to_dev(z, torch.float64), to_dev(w, torch.complex128)
    out = torch.empty(points, dtype=torch.complex128, device="cuda")
    kd = pkg.kernel_desc("helmholtz_slp", 3.0)
    torch.cuda.synchronize()
    _solve(ctx, 200)
    ctx.bem_potentials(mid, kd, zd, wd, out, q=4)
    ctx.bem_sync()
    eager = out.clone()
    g = torch.cuda.CUDAGraph()
    with torch.cuda.graph(g, stream=stream):
        ctx.bem_potentials(mid, kd, zd, wd, out, q=4)
    assert _solve(ctx, 1500) < 1e-8
    out.zero_()
    torch.cuda.synchronize()
    g.replay()
    torch.cuda.synchronize()
    assert torch.equal(out, eager)
    x, gw = np.polynomial.legendre.leggauss(4)
    x, gw = 0.5 + 0.5 * x, 0.5 * gw
    s, t, qw = np.repeat(x, 4), np.outer(x, x).ravel(), np.outer(gw * x, gw).ravel()
    v = mesh.verts[mesh.tris]
    e1, e2 = v[:, 1] - v[:, 0], v[:, 2] - v[:, 1]
    gram = np.linalg.norm(np.cross(e1, e2), axis=1)
    y = (v[:, None, 0] + s[:, None] * e1[:, None] + t[:, None] * e2[:, None]).reshape(-1, 3)
    wt = (qw[None] * (w * gram)[:, None] / (4 * np.pi)).ravel()
    for k in range(0, points, 100):
        r = np.linalg.norm(z[k:k + 100, None] - y[None], axis=2)
        ref, A = (np.exp(3j * r) / r) @ wt, (1 / r) @ np.abs(wt)
        assert (np.abs(eager[k:k + 100].cpu().numpy() - ref) / A).max() < 1e-12
    ctx.bem_mesh_free(mid)


@pytest.mark.parametrize("basis,kernel", [("p0", "laplace_slp"), ("p0", "laplace_dlp"), ("p1", "laplace_slp"),
                                          ("p1", "laplace_dlp"), ("p0", "helmholtz_slp")])
def test_fp64_captured_after_another_call(env, basis, kernel):
    import torch
    pkg, ctx, stream = env
    mesh = synth.jitter(synth.icosphere(1), 0.05, 7)
    n = mesh.nt if basis == "p0" else mesh.nv
    quad = dict(q_regular=3, q_identical=5, q_edge=4, q_vertex=3)
    if basis == "p1":       # the rules' first call is one of the other basis
        other = ctx.bem_mesh_upload(mesh.verts, mesh.tris, "p0")
        o = torch.zeros(mesh.nt ** 2, dtype=torch.float64, device="cuda")
        torch.cuda.synchronize()
        ctx.bem_assemble_dense(other, pkg.kernel_desc(kernel), pkg.quad_desc(precision="mixed_full", **quad), 0, o)
        ctx.bem_sync()
    mid = ctx.bem_mesh_upload(mesh.verts, mesh.tris, basis)
    cplx = kernel.startswith("helmholtz")
    out = torch.zeros(n * n, dtype=torch.complex128 if cplx else torch.float64, device="cuda")
    kd = pkg.kernel_desc(kernel, 2.0 if cplx else 0.0)
    torch.cuda.synchronize()
    if cplx:
        # the dense call's other buffers; then other orders, whose rules only the entry kernel has loaded
        ctx.bem_assemble_dense(mid, kd, pkg.quad_desc(q_regular=3, q_identical=3, q_edge=3, q_vertex=2), 0, out)
        i = torch.arange(32, dtype=torch.int32, device="cuda")
        ctx.bem_pivot_entries(mid, kd, pkg.quad_desc(**quad), i, i, torch.zeros(32, dtype=out.dtype, device="cuda"))
    else:
        ctx.bem_assemble_dense(mid, pkg.kernel_desc("laplace_slp"), pkg.quad_desc(precision="mixed_full", **quad), 0, out)
    ctx.bem_sync()
    g = torch.cuda.CUDAGraph()
    with torch.cuda.graph(g, stream=stream):
        ctx.bem_assemble_dense(mid, kd, pkg.quad_desc(**quad), 0, out)
    g.replay()
    torch.cuda.synchronize()
    got = out.clone()
    out.zero_()
    torch.cuda.synchronize()
    ctx.bem_assemble_dense(mid, kd, pkg.quad_desc(**quad), 0, out)
    ctx.bem_sync()
    assert torch.equal(got, out)
    ctx.bem_mesh_free(mid)
