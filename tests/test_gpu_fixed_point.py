"""The FP64 form in fixed point (bem_fixed_pair.cuh, bem_touch_fixed.cuh)
against the oracle where its ranges end: meshes of very small and very large
size and far from the origin (the pair's scale), flattened and stretched ones
(distances below a sixteenth of a pair's scale, which take the FP64 path, and
slivers), every regular rule's point count, and singular orders on both sides of
the complex kinds' limit.

Tolerance 1e-11 of the sum of the magnitudes of an entry's terms (or a
thousandth of its row's largest): both sides carry about 2^-50 of a term for
regular shapes, and 2^-53 S / r where a pair's coordinate differences S exceed
its distances r, with S / r up to some 10^3 on the flattened meshes."""
import numpy as np
import pytest

import oracle
import synth
from parity_util import rel_err_abs

pytestmark = pytest.mark.gpu

TOL = 1e-11
SHAPES = {"unit": (1.0, (1.0, 1.0, 1.0), 0.0), "tiny": (1e-6, (1.0, 1.0, 1.0), 0.0),
          "huge": (3e7, (1.0, 1.0, 1.0), 0.0), "far": (0.01, (1.0, 1.0, 1.0), 5.0),
          "flat": (1.0, (1.0, 1.0, 0.01), 0.0), "long": (1.0, (1.0, 30.0, 1.0), 0.0)}
KERNELS = ("laplace_slp", "laplace_dlp", "helmholtz_slp", "helmholtz_dlp")


@pytest.fixture(scope="module")
def pkg():
    import torch
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    import __graft_entry__
    __graft_entry__.build()
    import paper_1510_07244_gb300 as p
    return p


@pytest.fixture(scope="module")
def ctx(pkg):
    c = pkg.Context(0)
    yield c
    c.close()


def _check(pkg, ctx, mesh, basis, kernel, kappa, quad):
    import torch
    mid = ctx.bem_mesh_upload(mesh.verts, mesh.tris, basis)
    n = mesh.nt if basis == "p0" else mesh.nv
    cplx = kernel.startswith("helmholtz")
    out = torch.zeros(n * n, dtype=torch.complex128 if cplx else torch.float64, device="cuda")
    ctx.bem_assemble_dense(mid, pkg.kernel_desc(kernel, kappa), pkg.quad_desc(**quad), 0, out)
    ctx.bem_sync()
    ctx.bem_mesh_free(mid)
    rows, cols = np.tile(np.arange(n), n), np.repeat(np.arange(n), n)
    kw = dict(kernel=kernel, kappa=kappa, basis=basis, **quad)
    ref = oracle.entries(mesh.verts, mesh.tris, rows, cols, **kw)
    A = oracle.entries_absolute(mesh.verts, mesh.tris, rows, cols, **kw)
    got = out.cpu().numpy()
    err = rel_err_abs(got, ref if cplx else ref.real, A, rows).max()
    assert err <= TOL, err


@pytest.mark.parametrize("shape", sorted(SHAPES))
@pytest.mark.parametrize("kernel", KERNELS)
@pytest.mark.parametrize("basis", ["p0", "p1"])
def test_scales_and_shapes(pkg, ctx, basis, kernel, shape):
    scale, stretch, shift = SHAPES[shape]
    m = synth.jitter(synth.torus(7, 5), 0.05, 5)
    mesh = type(m)((m.verts * np.array(stretch) + shift) * scale, m.tris, m.name)
    quad = dict(q_regular=3, regular_rule="duffy", q_identical=4, q_edge=3, q_vertex=3)
    _check(pkg, ctx, mesh, basis, kernel, 4.0 / scale, quad)


@pytest.mark.parametrize("kernel", KERNELS)
@pytest.mark.parametrize("rule,q,singular", [("duffy", 2, 1), ("tri7", 3, 2), ("duffy", 4, 9),
                                             ("duffy", 3, 10)])
def test_rules(pkg, ctx, kernel, rule, q, singular):
    mesh = synth.jitter(synth.icosphere(0), 0.05, 6)
    quad = dict(q_regular=q, regular_rule=rule, q_identical=singular, q_edge=singular,
                q_vertex=singular)
    _check(pkg, ctx, mesh, "p0", kernel, 40.0, quad)


def _duffy(q):
    x, w = np.polynomial.legendre.leggauss(q)
    x, w = 0.5 + 0.5 * x, 0.5 * w
    return np.repeat(x, q), np.outer(x, x).ravel(), np.outer(w * x, w).ravel()


@pytest.mark.parametrize("away", [3.0, 0.3, 0.01])
@pytest.mark.parametrize("kernel", ["laplace_slp", "helmholtz_slp", "helmholtz_bw"])
def test_points_towards_the_surface(pkg, ctx, kernel, away):
    """Green matrices and potentials for points at a distance down to a hundredth of the edge
    length (below S / 16, the FP64 path), against numpy with the same rule; normals longer than 1
    leave the fixed-point range too.  Tolerance 1e-12 of the sum of the terms' magnitudes."""
    import torch
    kappa = 0.0 if kernel == "laplace_slp" else 3.0
    mesh = synth.jitter(synth.torus(7, 5), 0.05, 5)
    v = mesh.verts[mesh.tris]
    n = np.cross(v[:, 1] - v[:, 0], v[:, 2] - v[:, 1])
    gram = np.linalg.norm(n, axis=1)
    n /= gram[:, None]
    h = np.sqrt(gram.mean())
    z = v.mean(1) + away * h * n
    s, t, w = _duffy(3)
    y = (v[:, None, 0] + s[None, :, None] * (v[:, 1] - v[:, 0])[:, None]
         + t[None, :, None] * (v[:, 2] - v[:, 1])[:, None])
    d = z[:, None, None] - y[None]
    r = np.linalg.norm(d, axis=3)
    wave = np.exp(1j * kappa * r) / r
    wt = w[None, None] * gram[None, :, None] / (4 * np.pi)
    double = (d * n[None, :, None]).sum(3) / r ** 2 * (1 - 1j * kappa * r) * wave
    mid = ctx.bem_mesh_upload(mesh.verts, mesh.tris, "p0")
    dens = np.exp(1j * np.arange(mesh.nt))
    val = double - 1j * kappa * wave if kernel == "helmholtz_bw" else wave
    out = torch.zeros(mesh.nt, dtype=torch.complex128, device="cuda")
    ctx.bem_potentials(mid, pkg.kernel_desc(kernel, kappa, kappa), torch.as_tensor(z).cuda(),
                       torch.as_tensor(dens).cuda(), out, q=3)
    ctx.bem_sync()
    ref = (val * wt).sum(2) @ dens
    A = (np.abs(val) * wt).sum((1, 2))
    assert (np.abs(out.cpu().numpy() - ref) / A).max() < 1e-12
    if kernel != "helmholtz_bw":
        # every triangle a row of one cluster, normals of length 1 and of length 7
        nz = n * np.where(np.arange(mesh.nt) % 40 < 35, 1.0, 7.0)[:, None]
        cols = 2 * mesh.nt
        cplx = kernel == "helmholtz_slp"
        o = torch.zeros(mesh.nt * cols, dtype=torch.complex128 if cplx else torch.float64, device="cuda")
        i32 = lambda a: torch.as_tensor(np.ascontiguousarray(a), dtype=torch.int32).cuda()
        ctx.bem_green_matrices(pkg.GreenJob(mid, i32([0, mesh.nt]), i32(np.arange(mesh.nt)),
                                            i32([0, mesh.nt]), torch.as_tensor(z).cuda(),
                                            torch.as_tensor(nz).cuda(),
                                            torch.zeros(1, dtype=torch.int64, device="cuda"), o,
                                            kernel=pkg.kernel_desc(kernel, kappa), rule="duffy", q=3))
        ctx.bem_sync()
        got = o.cpu().numpy().reshape(cols, mesh.nt).T
        minus = -(d * nz[:, None, None]).sum(3) / r ** 2 * (1 - 1j * kappa * r) * wave
        for k, f in ((0, wave), (1, minus)):
            ref, A = (f * wt).sum(2).T, (np.abs(f) * wt).sum(2).T
            err = np.abs(got[:, k * mesh.nt:(k + 1) * mesh.nt] - (ref if cplx else ref.real))
            assert (err / A.max(1, keepdims=True)).max() < 1e-12
    ctx.bem_mesh_free(mid)
