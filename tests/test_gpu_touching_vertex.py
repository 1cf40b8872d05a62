"""GPU: double layers of pairs with a common vertex in the FP64 form, against the
Sauter-Schwab rule in long double, relative to the sum of the magnitudes of an
entry's terms, on a torus and the same flattened to a tenth and stretched six
times.  (The oracle adds its 512 terms in sequence in double, which costs more
than what is looked for here.)

Root mean square tolerance 2^-51 (2^-50 for the flattened and the stretched
one): a term carries a few roundings of 2^-53 (the difference's three components
relative to the distance, its power, the height, the phase), their mean over
the entries a few 2^-53, and twice that where edges differ in length by ten."""
import numpy as np
import pytest

import synth
from test_gpu_h2 import env  # noqa: F401  (fixture)

pytestmark = pytest.mark.gpu


def _gauss():
    """Four Gauss points on [0, 1] in long double (Newton steps on P4)."""
    x = np.polynomial.legendre.leggauss(4)[0].astype(np.longdouble)
    for _ in range(3):
        x = x - (35 * x ** 4 - 30 * x ** 2 + 3) / (140 * x ** 3 - 60 * x)
    d = (140 * x ** 3 - 60 * x) / 8
    return (x + 1) / 2, 1 / ((1 - x * x) * d * d)


def _reference(v, t, rows, cols, kernel, kappa):
    """Entries of pairs with one common vertex and their terms' magnitudes."""
    v = v.astype(np.longdouble)
    g, w = _gauss()
    xi, a, b, c = (x.ravel() for x in np.meshgrid(g, g, g, g, indexing="ij"))
    wt = np.einsum("i,j,k,l->ijkl", w, w, w, w).ravel() * xi ** 3 * b
    one, two = (xi, xi * a), (xi * b, xi * b * c)      # the pair's points, and swapped
    (x1, x2), (y1, y2) = ([np.concatenate([p, q]) for p, q in zip(one, two)],
                          [np.concatenate([q, p]) for p, q in zip(one, two)])
    wt = np.concatenate([wt, wt])
    turned = []
    for tri, other in ((t[rows], t[cols]), (t[cols], t[rows])):
        first = (tri[:, :, None] == other[:, None, :]).any(2).argmax(1)
        turned.append(v[np.take_along_axis(tri, (first[:, None] + np.arange(3)) % 3, 1)])
    A, B = turned
    na, nb = (np.cross(T[:, 1] - T[:, 0], T[:, 2] - T[:, 1]) for T in (A, B))
    ga, gb = (np.sqrt((n * n).sum(1)) for n in (na, nb))
    d = (x1[:, None] * (A[:, 1] - A[:, 0])[:, None] + x2[:, None] * (A[:, 2] - A[:, 1])[:, None]
         - y1[:, None] * (B[:, 1] - B[:, 0])[:, None] - y2[:, None] * (B[:, 2] - B[:, 1])[:, None])
    r = np.sqrt((d * d).sum(2))
    dn = (d * (nb / gb[:, None])[:, None]).sum(2)
    c, s, p = np.cos(kappa * r), np.sin(kappa * r), kappa * r
    k = dn / r ** 3 * ((c + p * s) + 1j * (s - p * c))
    if kernel == "helmholtz_bw":
        k = k - 1j * kappa * (c + 1j * s) / r
    f = ga * gb / (16 * np.arctan(np.longdouble(1)))
    return (k * wt).sum(1) * f, (np.abs(k) * wt).sum(1) * f


@pytest.mark.parametrize("stretch,bits", [((1, 1, 1), 51), ((1, 1, 0.1), 50), ((1, 6, 1), 50)])
@pytest.mark.parametrize("kernel", ["laplace_dlp", "helmholtz_dlp", "helmholtz_bw"])
def test_common_vertex(env, kernel, stretch, bits):  # noqa: F811
    import torch
    pkg, ctx = env
    m = synth.jitter(synth.torus(8, 6), 0.08, 3)
    v, t, n = np.array(m.verts) * stretch, m.tris, m.nt
    kappa = 2.0 if kernel.startswith("helmholtz") else 0.0
    quad = dict(q_regular=3, q_identical=4, q_edge=4, q_vertex=4)
    mid = ctx.bem_mesh_upload(v, t, "p0")
    out = torch.zeros(n * n, dtype=torch.complex128 if kappa else torch.float64, device="cuda")
    ctx.bem_assemble_dense(mid, pkg.kernel_desc(kernel, kappa, kappa), pkg.quad_desc(**quad), 0, out)
    ctx.bem_sync()
    ctx.bem_mesh_free(mid)
    shared = (t[:, None, :, None] == t[None, :, None, :]).any(3).sum(2)
    rows, cols = np.nonzero(shared == 1)
    ref, A = _reference(v, t, rows, cols, kernel, kappa)
    err = (np.abs(out.cpu().numpy().reshape(n, n).T[rows, cols] - (ref if kappa else ref.real)) / A).astype(float)
    assert np.sqrt((err ** 2).mean()) < 2.0 ** -bits, np.sqrt((err ** 2).mean())
