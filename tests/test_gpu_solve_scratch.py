"""GPU: dense GMRES gives its scratch back where it is large (9000 unknowns, 500
Krylov vectors: 72 MB), and solves on with what it keeps."""
import pytest

from test_gpu_h2 import env  # noqa: F401  (fixture)

pytestmark = pytest.mark.gpu


def test_large_scratch_is_freed(env):  # noqa: F811
    import torch
    pkg, ctx = env

    def solve(n, restart):
        A = torch.eye(n, dtype=torch.complex128, device="cuda").reshape(-1)
        b = torch.ones(n, dtype=torch.complex128, device="cuda")
        x = torch.zeros_like(b)
        torch.cuda.synchronize()
        ctx.bem_dense_gmres(A, b, x, tol=1e-12, restart=restart)
        free = torch.cuda.mem_get_info()[0]
        assert torch.allclose(x, b)
        return free

    # the same tensors each time: torch keeps their memory
    solve(9000, 30)
    before = solve(9000, 30)
    after = solve(9000, 500)
    assert before - after < 16 << 20
    solve(300, 20)
