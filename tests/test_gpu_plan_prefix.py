"""GPU: plans whose jobs are long enough for a cluster of CTAs to sum their blocks
(above 4096), beside short ones in the same bucket, with empty blocks among them:
the bits of single calls."""
import numpy as np
import pytest

import synth
from parity_util import block_job
from test_gpu_h2 import env  # noqa: F401  (fixture)

pytestmark = pytest.mark.gpu


def _blocks(n, count, rng):
    """`count` blocks of clusters of 0 to 3 triangles out of n."""
    size = rng.integers(0, 4, 64)
    ptr = np.concatenate([[0], np.cumsum(size)]).astype(np.int32)
    idx = rng.integers(0, n, ptr[-1]).astype(np.int32)
    row, col = (rng.integers(0, 64, count).astype(np.int32) for _ in range(2))
    off = np.concatenate([[0], np.cumsum(size[row] * size[col])]).astype(np.int64)
    return synth.workloads.BlockSet(ptr, idx, ptr, idx, row, col, off[:-1], int(off[-1]))


@pytest.mark.parametrize("counts", [(4097, 1), (3, 20000, 7, 4099), (4096,)])
@pytest.mark.parametrize("precision", ["fp64", "mixed_full"])
def test_long_jobs(env, precision, counts):  # noqa: F811
    import torch
    pkg, ctx = env
    rng = np.random.default_rng(len(counts))
    mesh = synth.jitter(synth.icosphere(1), 0.05, 3)
    mid = ctx.bem_mesh_upload(mesh.verts, mesh.tris, "p0")
    sets = [_blocks(mesh.nt, c, rng) for c in counts]
    quad = dict(q_regular=2, q_identical=3, q_edge=3, q_vertex=3, precision=precision)

    def jobs():
        return [block_job(pkg, mid, bs, "laplace_slp", 0.0, quad,
                          torch.zeros(max(1, bs.n_entries), dtype=torch.float64, device="cuda")) for bs in sets]

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
