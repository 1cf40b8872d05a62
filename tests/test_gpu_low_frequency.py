"""GPU: Helmholtz entries far below the first resonance in the FP64 form: the
imaginary parts, about kappa / (4 pi) of the areas' product and so down to 1e-6
of the real ones, against the oracle relative to themselves.

Tolerance 2e-13: the oracle adds up to 6 * 4^4 terms of one sign in sequence,
each step rounding to 2^-53 of the sum."""
import numpy as np
import pytest

import oracle
import synth
from test_gpu_h2 import env  # noqa: F401  (fixture)

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("kappa", [0.1, 1e-2, 1e-3, 1e-6])
@pytest.mark.parametrize("basis", ["p0", "p1"])
def test_imaginary_parts(env, basis, kappa):  # noqa: F811
    import torch
    pkg, ctx = env
    m = synth.jitter(synth.icosphere(1), 0.05, 3)
    n = m.nt if basis == "p0" else m.nv
    quad = dict(q_regular=3, regular_rule="duffy", q_identical=4, q_edge=4, q_vertex=4)
    mid = ctx.bem_mesh_upload(m.verts, m.tris, basis)
    out = torch.zeros(n * n, dtype=torch.complex128, device="cuda")
    ctx.bem_assemble_dense(mid, pkg.kernel_desc("helmholtz_slp", kappa), pkg.quad_desc(**quad), 0, out)
    ctx.bem_sync()
    ctx.bem_mesh_free(mid)
    ref = oracle.entries(m.verts, m.tris, np.tile(np.arange(n), n), np.repeat(np.arange(n), n),
                         kernel="helmholtz_slp", kappa=kappa, basis=basis, **quad)
    got = out.cpu().numpy()
    assert (np.abs(got.imag - ref.imag) < 2e-13 * np.abs(ref.imag)).all()
    assert (np.abs(got.real - ref.real) < 2e-13 * np.abs(ref.real)).all()
