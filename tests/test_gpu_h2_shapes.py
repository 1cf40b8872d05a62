"""GPU: the H2 product on trees and blocks of random entries, at the edges of
its kernels: leaves of more than 64 indices, blocks of more than 32 rows or
columns, ranks 0 and 32, odd ranks, coupling at one level only (the clusters
above take part in neither transformation), and no coupling at all.  The
reference is the oracle's product.  Tolerance: every entry is a chain of at
most 4 nested sums of fewer than 2^11 terms, so its rounding error is below
2^14 * 2^-53 = 2e-12 of the same product of absolute values."""
import numpy as np
import pytest

from oracle import h2 as oh2
from parity_util import to_dev
from test_gpu_h2 import env  # noqa: F401  (fixture)

pytestmark = pytest.mark.gpu


def _tree(sizes):
    """Balanced binary tree over leaves of the given sizes (a power of two):
    clusters numbered leaves last, index sets contiguous per leaf."""
    n_leaf = len(sizes)
    perm = np.random.default_rng(5).permutation(sum(sizes)).astype(np.int32)
    ends = np.concatenate([[0], np.cumsum(sizes)])
    sets, son = [], []
    for c in range(2 * n_leaf - 1):
        d = int(np.log2(c + 1))
        w = n_leaf >> d
        k = c + 1 - (1 << d)
        sets.append(perm[ends[k * w]:ends[(k + 1) * w]])
        son.append([2 * c + 1, 2 * c + 2] if c < n_leaf - 1 else [-1, -1])
    return sets, np.array(son, np.int32)


@pytest.mark.parametrize("sizes,ranks,far_depth", [
    ([65, 64, 33, 32], (32, 31), 1),
    ([1, 130, 7, 70, 31, 2, 90, 40], (5, 17, 32), 2),
    ([96] * 8, (0, 9, 16), 3),
    ([20, 50, 33, 12], (8,), None),
])
def test_h2_product_shapes(env, sizes, ranks, far_depth):  # noqa: F811
    import torch
    pkg, ctx = env
    rng = np.random.default_rng(11)
    sets, son = _tree(sizes)
    n, nc = sum(sizes), len(sets)
    ptr = np.concatenate([[0], np.cumsum([len(s) for s in sets])]).astype(np.int32)
    rank = [ranks[c % len(ranks)] for c in range(nc)]
    pp = np.concatenate([[0], np.cumsum(rank)]).astype(np.int32)
    rows = [sum(rank[s] for s in son[c]) if son[c][0] >= 0 else len(sets[c]) for c in range(nc)]
    mats = [rng.standard_normal((rows[c], rank[c])) for c in range(nc)]
    leaves = [c for c in range(nc) if son[c][0] < 0]

    def blocks(pairs, size):
        off = np.concatenate([[0], np.cumsum([size(t) * size(s) for t, s in pairs])])
        vals = rng.standard_normal(max(1, int(off[-1])))
        mats_ = [vals[off[k]:off[k + 1]].reshape(size(s), size(t)).T
                 for k, (t, s) in enumerate(pairs)]
        t, s = (np.array([p[j] for p in pairs], np.int32) for j in (0, 1))
        return (t, s, off[:-1].astype(np.int64)), vals, mats_

    # near: every leaf with itself, the leaf before it and the root (many columns)
    near, nv, nm = blocks([(t, s) for i, t in enumerate(leaves) for s in (t, leaves[i - 1], 0)],
                          lambda c: len(sets[c]))
    level = [] if far_depth is None else range((1 << far_depth) - 1, (2 << far_depth) - 1)
    far, fv, fm = blocks([(t, s) for t in level for s in level if t != s and (t + s) % 3],
                         lambda c: rank[c])
    diag = rng.standard_normal(n)
    x = rng.standard_normal(n)
    nvd, fvd = to_dev(nv, torch.float64), to_dev(fv, torch.float64)
    h = ctx.bem_h2_create(n, ptr, np.concatenate(sets), son, pp, np.zeros(pp[-1], np.int32), mats,
                          near, nvd, far, fvd, diag=diag)
    y = torch.empty(n, dtype=torch.float64, device="cuda")
    ctx.bem_h2_matvec(h, to_dev(x, torch.float64), y)
    ctx.bem_sync()
    ctx.bem_h2_destroy(h)

    def product(f, x):
        V = [None] * nc
        for c in reversed(range(nc)):
            if son[c][0] < 0:
                V[c] = f(mats[c])
            else:
                a, b = son[c]
                V[c] = np.concatenate([V[a] @ f(mats[c])[:rank[a]], V[b] @ f(mats[c])[rank[a]:]])
        return f(diag) * x + oh2.h2_matvec(
            n, x, [(sets[t], sets[s], f(m)) for t, s, m in zip(near[0], near[1], nm)],
            [(t, s, f(m)) for t, s, m in zip(far[0], far[1], fm)],
            [(sets[c], V[c]) for c in range(nc)], pp)

    err = np.abs(y.cpu().numpy() - product(lambda a: a, x))
    assert (err <= 2e-12 * product(np.abs, np.abs(x))).all()
