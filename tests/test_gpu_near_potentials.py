"""GPU: potentials at points beside a triangle, whose distances to the rule's
points are at least a quarter of the extent S but about those from the
triangle's centroid to its vertices (no bound of S / r from the centroid).

One triangle at a time, against numpy with the same rule, relative to the sum of
the magnitudes of both layers' terms.  Tolerance (6 * 4 + 4 * 5) 2^-53: coordinate
differences are rounded to 2^-53 S, 1/r^3 takes three times the relative error of
r, the phase kappa r (at most 5) its absolute one, and both sides carry them."""
import numpy as np
import pytest

from parity_util import to_dev
from test_gpu_h2 import env  # noqa: F401  (fixture)

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("kernel", ["laplace_dlp", "helmholtz_dlp", "helmholtz_bw"])
def test_beside_a_triangle(env, kernel):  # noqa: F811
    import torch
    pkg, ctx = env
    kappa = eta = 1.0 if kernel.startswith("helmholtz") else 0.0
    if kernel != "helmholtz_bw":
        eta = 0.0
    rng = np.random.default_rng(4)
    x, w = np.polynomial.legendre.leggauss(4)
    x, w = 0.5 + 0.5 * x, 0.5 * w
    s, t, w = np.repeat(x, 4)[:, None], np.outer(x, x).ravel()[:, None], np.outer(w * x, w).ravel()
    worst = points = 0
    for _ in range(20):
        T = np.array([[0, 0, 0], [1, 0, 0], [0.4, 0.8, 0]]) + rng.uniform(-0.2, 0.2, (3, 3))
        n = np.cross(T[1] - T[0], T[2] - T[1])
        gram = np.linalg.norm(n)
        n /= gram
        y = T[0] + s * (T[1] - T[0]) + t * (T[2] - T[1])
        z = rng.dirichlet([1, 1, 1], 200) @ T + rng.uniform(0.25, 0.7, (200, 1)) * n * rng.choice([-1, 1], (200, 1))
        size = (np.abs(z - T[0]) + np.abs(T - T[0]).max(0)).max(1)
        z = z[2.0 ** np.ceil(np.log2(size)) < 4 * np.linalg.norm(z[:, None] - y[None], axis=2).min(1)]
        d = z[:, None] - y[None]
        r = np.linalg.norm(d, axis=2)
        assert (kappa * r <= 5).all()
        single = np.exp(1j * kappa * r) / r
        double = (d @ n) / r ** 2 * (1 - 1j * kappa * r) * single
        mid = ctx.bem_mesh_upload(T, np.array([[0, 1, 2]], np.int32), "p0")
        out = torch.zeros(len(z), dtype=torch.complex128, device="cuda")
        ctx.bem_potentials(mid, pkg.kernel_desc(kernel, kappa, eta), to_dev(z, torch.float64),
                           torch.ones(1, dtype=torch.complex128, device="cuda"), out, q=4)
        ctx.bem_sync()
        ctx.bem_mesh_free(mid)
        f = w * gram / (4 * np.pi)
        err = np.abs(out.cpu().numpy() - (double - 1j * eta * single) @ f)
        worst = max(worst, (err / ((np.abs(double) + eta * np.abs(single)) @ f)).max())
        points += len(z)
    assert points > 500
    assert worst < 44 * 2.0 ** -53, worst
