"""GPU: the order of the H2 product's sums where one summand is much larger than
the others.  Four leaves of 32 indices, bases of unit entries, and blocks whose
sums are exact in double as long as the small summands (2^-54) are added to one
another before they meet the large one (1): a father's part beside 32
admissible blocks of a leaf, and a leaf's near field beside its 32 basis
columns.  Both results are 1 + 2^-49, bit for bit."""
import numpy as np
import pytest

from parity_util import to_dev
from test_gpu_h2 import env  # noqa: F401  (fixture)

pytestmark = pytest.mark.gpu


def test_small_summands_first(env):  # noqa: F811
    import torch
    pkg, ctx = env
    r, tiny = 32, 2.0 ** -54
    n = 4 * r
    # clusters 0 (root), 1, 2, leaves 3 to 6
    sets = [np.arange(n), np.arange(2 * r), np.arange(2 * r, n)] + [np.arange(k * r, (k + 1) * r) for k in range(4)]
    son = np.array([[1, 2], [3, 4], [5, 6]] + 4 * [[-1, -1]], np.int32)
    ptr = np.concatenate([[0], np.cumsum([len(s) for s in sets])]).astype(np.int32)
    rank = [0] + 6 * [r]
    pp = np.concatenate([[0], np.cumsum(rank)]).astype(np.int32)
    eye, first = np.eye(r), np.zeros((r, r))
    first[0, 0] = 1.0
    up = np.concatenate([eye, np.zeros((r, r))])       # y^ of the first son, nothing of the second
    mats = [np.zeros((2 * r, 0)), up, up, eye, np.concatenate([np.ones((1, r)), np.zeros((r - 1, r))]), eye, eye]
    far = [(1, 2, first)] + 32 * [(3, 5, tiny * first)] + [(4, 6, tiny * eye)]
    near = [(4, 4, first)]

    def blocks(b):
        return ((np.array([t for t, _, _ in b], np.int32), np.array([s for _, s, _ in b], np.int32),
                 np.arange(len(b), dtype=np.int64) * r * r),
                to_dev(np.concatenate([m.T.ravel() for _, _, m in b]), torch.float64))

    (nl, nv), (fl, fv) = blocks(near), blocks(far)
    h = ctx.bem_h2_create(n, ptr, np.concatenate(sets).astype(np.int32), son, pp, np.zeros(pp[-1], np.int32),
                          mats, nl, nv, fl, fv)
    y = torch.empty(n, dtype=torch.float64, device="cuda")
    ctx.bem_h2_matvec(h, torch.ones(n, dtype=torch.float64, device="cuda"), y)
    ctx.bem_sync()
    ctx.bem_h2_destroy(h)
    y = y.cpu().numpy()
    assert y[0] == 1.0 + 2.0 ** -49        # leaf 3: the father's part and its blocks
    assert y[r] == 1.0 + 2.0 ** -49        # leaf 4: its near field and its basis
