"""GPU: double layers between two parallel plates 1e-6 apart in the FP64 form.

The plates are parallel to a coordinate plane, so the heights of a pair are one
component's differences, exact in FP64 arithmetic; a form with one absolute
scale for all components loses them.  Entries between interior triangles
(vertices) of the two plates against the oracle, relative to the sum of the
magnitudes of an entry's terms.  Tolerance 1e-13: lateral differences of up to
S are rounded to 2^-53 S, distances of different points are at least S / 100 or
the gap alone, and 1/r^3 takes three times their relative error, on both sides:
6 * 100 * 2^-53 = 7e-14."""
import numpy as np
import pytest

import oracle
import synth
from test_gpu_h2 import env  # noqa: F401  (fixture)

pytestmark = pytest.mark.gpu


def _plates(gap):
    m = synth.cube_surface(4)
    v = np.array(m.verts)
    v = (v - v.min(0)) / (v.max(0) - v.min(0)) * [1.0, 1.3, 1.0]
    top, bottom = v[:, 2] > 0.99, v[:, 2] < 0.01
    v[:, 0] += 0.07 * np.sin(3.0 * v[:, 1])
    v[:, 1] += 0.05 * np.cos(2.0 * v[:, 0])
    v[:, 2] = np.where(top, 0.8234567 * gap, 0.61 * gap * v[:, 2])
    return type(m)(v, m.tris, "plates"), top, bottom


@pytest.mark.parametrize("q,rule", [(2, "duffy"), (3, "duffy"), (4, "duffy"), (3, "tri7")])
@pytest.mark.parametrize("kernel", ["laplace_dlp", "helmholtz_dlp"])
@pytest.mark.parametrize("basis", ["p0", "p1"])
def test_heights(env, basis, kernel, q, rule):  # noqa: F811
    import torch
    pkg, ctx = env
    mesh, top, bottom = _plates(1e-6)
    kappa = 3.0 if kernel.startswith("helmholtz") else 0.0
    quad = dict(q_regular=q, regular_rule=rule, q_identical=3, q_edge=3, q_vertex=3)
    mid = ctx.bem_mesh_upload(mesh.verts, mesh.tris, basis)
    n = mesh.nt if basis == "p0" else mesh.nv
    out = torch.zeros(n * n, dtype=torch.complex128 if kappa else torch.float64, device="cuda")
    ctx.bem_assemble_dense(mid, pkg.kernel_desc(kernel, kappa), pkg.quad_desc(**quad), 0, out)
    ctx.bem_sync()
    ctx.bem_mesh_free(mid)
    got = out.cpu().numpy().reshape(n, n).T
    if basis == "p0":
        t, b = (np.nonzero(s[mesh.tris].all(1))[0] for s in (top, bottom))
    else:       # vertices all of whose triangles lie in their plate
        inner = [s & ~np.isin(np.arange(n), mesh.tris[~s[mesh.tris].all(1)]) for s in (top, bottom)]
        t, b = (np.nonzero(s)[0] for s in inner)
    assert len(t) and len(b)
    rows, cols = np.repeat(b, len(t)), np.tile(t, len(b))
    kw = dict(kernel=kernel, kappa=kappa, basis=basis, **quad)
    ref = oracle.entries(mesh.verts, mesh.tris, rows, cols, **kw)
    A = oracle.entries_absolute(mesh.verts, mesh.tris, rows, cols, **kw)
    err = np.abs(got[rows, cols] - (ref if kappa else ref.real)) / A
    assert err.max() < 1e-13, err.max()
