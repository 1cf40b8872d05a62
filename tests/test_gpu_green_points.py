"""GPU: Green matrices with points and normals outside the fixed-point range.

One cluster whose points hold a NaN or infinite coordinate (not the first
point's), a NaN normal, and normals of length 1e-9 and sqrt(3): columns that
plain arithmetic makes NaN are NaN (every entry, real or imaginary part), and
all the others are numpy's with the same rule, to 1e-12 of the sum of the terms'
magnitudes (16 terms of a few 2^-53 each).  An infinite point has r = infinity:
its plus entries are 0 or NaN in plain arithmetic, so only the other columns are
compared."""
import numpy as np
import pytest

import synth
from parity_util import to_dev
from test_gpu_h2 import env  # noqa: F401  (fixture)

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("infinite", [False, True])
@pytest.mark.parametrize("kernel", ["laplace_slp", "helmholtz_slp"])
def test_outside_the_range(env, kernel, infinite):  # noqa: F811
    import torch
    pkg, ctx = env
    kappa = 0.0 if kernel == "laplace_slp" else 3.0
    mesh = synth.jitter(synth.octasphere(4), 0.05, 5)
    v = mesh.verts[mesh.tris]
    n = np.cross(v[:, 1] - v[:, 0], v[:, 2] - v[:, 1])
    gram = np.linalg.norm(n, axis=1)
    m = 96
    rng = np.random.default_rng(2)
    nz = rng.standard_normal((m, 3))
    nz /= np.linalg.norm(nz, axis=1)[:, None]
    z = 2.0 * nz + 0.1 * rng.standard_normal((m, 3))
    z[40, 1] = np.inf if infinite else np.nan
    nz[50, 2] = np.nan
    nz[70] *= 1e-9
    nz[90] = 1.0
    x, w = np.polynomial.legendre.leggauss(4)
    x, w = 0.5 + 0.5 * x, 0.5 * w
    s, t, w = np.repeat(x, 4), np.outer(x, x).ravel(), np.outer(w * x, w).ravel()
    y = (v[:, None, 0] + s[None, :, None] * (v[:, 1] - v[:, 0])[:, None]
         + t[None, :, None] * (v[:, 2] - v[:, 1])[:, None])
    d = y[:, None] - z[None, :, None]
    r = np.linalg.norm(d, axis=3)
    wt = w * gram[:, None, None] / (4 * np.pi)
    with np.errstate(invalid="ignore"):
        plus = np.exp(1j * kappa * r) / r
        minus = (d * nz[None, :, None]).sum(3) / r ** 2 * (1 - 1j * kappa * r) * plus
    mid = ctx.bem_mesh_upload(mesh.verts, mesh.tris, "p0")
    cplx = kernel == "helmholtz_slp"
    out = torch.zeros(mesh.nt * 2 * m, dtype=torch.complex128 if cplx else torch.float64, device="cuda")
    i32 = lambda a: to_dev(np.asarray(a), torch.int32)  # noqa: E731
    ctx.bem_green_matrices(pkg.GreenJob(mid, i32([0, mesh.nt]), i32(np.arange(mesh.nt)), i32([0, m]),
                                        to_dev(z, torch.float64), to_dev(nz, torch.float64),
                                        to_dev(np.array([0]), torch.int64), out,
                                        kernel=pkg.kernel_desc(kernel, kappa), rule="duffy", q=4))
    ctx.bem_sync()
    ctx.bem_mesh_free(mid)
    got = out.cpu().numpy().reshape(2 * m, mesh.nt).T
    for k, f in enumerate((plus, minus)):
        col = got[:, k * m:(k + 1) * m]
        with np.errstate(invalid="ignore"):
            ref, A = (f * wt).sum(2), (np.abs(f) * wt).sum(2)
        bad = np.arange(m) == 40
        if k == 1:
            bad |= np.arange(m) == 50
        for c in np.nonzero(bad)[0]:
            if not (infinite and c == 40):
                assert np.isnan(col[:, c]).all(), (k, c)
        ok = ~bad
        err = np.abs(col - (ref if cplx else ref.real))[:, ok] / A[:, ok].max(0)
        assert err.max() < 1e-12, (k, np.nonzero(ok)[0][err.max(0).argmax()], err.max())
