"""Runs of equal lower bounds in the d = 1 tree's order (GPU).

The set is sorted by the lower bound; equal ones are then put in the order of
their upper bound, ties of both by id: in runs of up to 64 by the elements, of
up to 128 by a warp, longer ones by a CTA (up to 2,048 on chip).  If a sample of
1,024 bounds promises much more of one value, the set is sorted by both bounds.
Planted runs of every length around those limits in sets of otherwise distinct
bounds, their members away from the sampled positions (so that the sample sees
none of them) or everywhere; upper bounds that descend with the id, equal ones
and signed zeros among them; sizes of each form of the sort.  The tree order is
numpy's stable sort.
"""
import numpy as np
import pytest

import paper_1309_3458_gb300 as ddm
from tests.helpers import to_dev
from tests.test_gpu_parity import order_key

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def ctx():
    import __graft_entry__
    __graft_entry__.build()
    h = ddm.ddm_create(0)
    yield h
    ddm.ddm_destroy(h)


def tree_order(ctx, lo, hi):
    import torch
    S = to_dev((lo, hi))
    ddm.ddm_build(ctx, S[0], S[1])
    order = torch.empty(lo.shape[1], dtype=torch.int32, device="cuda")
    ddm.ddm_tree_export(ctx, order)
    return order.cpu().numpy()


def wanted(lo, hi):
    return np.lexsort((np.arange(lo.shape[1]), order_key(hi[0]), order_key(lo[0])))


def planted(n, lengths, seed):
    """Distinct lower bounds but for runs of the given lengths."""
    rng = np.random.default_rng(seed)
    lo = rng.permutation(n).astype(np.float32) - np.float32(n // 2)  # distinct: n < 2**24
    hi = lo + rng.integers(0, 5, n).astype(np.float32)
    sampled = (np.arange(1024, dtype=np.uint64) * np.uint64(n) // np.uint64(1024)).astype(np.int64)
    free = np.setdiff1d(np.arange(n), sampled)
    free = rng.permutation(free)
    at = 0
    for j, r in enumerate(lengths):
        m = np.sort(free[at:at + r])
        at += r
        v = np.float32(-0.0) if j == 0 else lo[m[0]]
        lo[m] = v
        up = np.arange(r, 0, -1).astype(np.float32) // (1 + j % 3)  # descending, some equal
        if j % 4 == 3:
            up = rng.integers(0, 1 << 20, r).astype(np.float32)
        hi[m] = np.maximum(v + up, v)
    assert (np.bincount(np.unique(lo, return_inverse=True)[1]) > 1).sum() <= len(lengths) + 1
    return lo[None, :], hi[None, :]


@pytest.mark.parametrize("n", [8193, 40001, 300007, 700001, 1600007])
def test_short_runs_keep_the_first_sort(ctx, n):
    """Runs of 2 to 32: nothing else puts them in order."""
    lo, hi = planted(n, [2, 3, 31, 32] + [2, 17, 32] * 20, seed=n)
    _, counts = np.unique(lo, return_counts=True)
    assert counts.max() == 32
    assert np.array_equal(tree_order(ctx, lo, hi), wanted(lo, hi))


@pytest.mark.parametrize("n,lengths", [(8193, [33, 40, 63, 64, 65, 127, 128, 129, 255, 256, 257, 1000]), (8200, [6000, 33]),
                                       (40001, [33, 256, 257, 1024, 1025, 2048, 2049, 8191]),
                                       (40001, [34] * 700), (40001, [64, 65, 128, 129] * 60), (300007, [8192, 8193, 20000, 33, 257]),
                                       (1600007, [256] * 2000 + [257] * 500 + [30000])])
def test_longer_runs(ctx, n, lengths):
    lo, hi = planted(n, lengths, seed=len(lengths))
    assert np.array_equal(tree_order(ctx, lo, hi), wanted(lo, hi))


@pytest.mark.parametrize("n", [8193, 40001, 300007, 700001, 1600007])
@pytest.mark.parametrize("values", [1, 2, 30, 500, 0])
def test_values_that_abound(ctx, n, values):
    """Few values, or (0) one for three quarters of the set."""
    rng = np.random.default_rng(n + values)
    if values:
        lo = rng.integers(0, values, size=(1, n)).astype(np.float32)
    else:
        lo = rng.permutation(n).astype(np.float32)[None, :]
        lo[0, rng.random(n) < 0.75] = 5.0
    hi = lo + rng.integers(0, 1 << 22, size=(1, n)).astype(np.float32)
    assert np.array_equal(tree_order(ctx, lo, hi), wanted(lo, hi))
