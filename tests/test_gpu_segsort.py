"""Re-sorts inside groups (GPU).

The updates' plan order for d >= 2 is the stable order of the top 24 bits of
the dimension-0 lower bound's key, then, dimension by dimension, a stable
re-sort by that dimension's key inside aligned groups of 2^g positions.  It
is compared with numpy's stable sorts at sizes around the chunks of 4,096 and
8,192 positions, with one and several groups per chunk, and beyond the groups
a CTA holds (the radix sort over the whole set).  A batch with an instance
whose groups exceed a CTA gives every instance's pairs of the plain call.
"""
import math

import numpy as np
import pytest

import paper_1309_3458_gb300 as ddm
from paper_1309_3458_gb300 import workloads as W
from tests.helpers import gpu_match, keys, to_dev
from tests.test_gpu_parity import order_key

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def ctx():
    import __graft_entry__
    __graft_entry__.build()
    h = ddm.ddm_create(0)
    yield h
    ddm.ddm_destroy(h)


def groups(n, d):
    """Group exponents by dimension (sort-tile-recursive sizes)."""
    out, prev = [0] * d, 64
    for k in range(1, d):
        if n < 64:
            continue
        nb = (n + 31) // 32
        g = int(math.floor(math.log2(32.0 * nb ** ((d - k) / d)) + 0.5))
        if 6 <= g < prev and (1 << g) < n:
            out[k], prev = g, g
    return out


def plan_order(lo, d):
    n = lo.shape[1]
    order = np.argsort(order_key(lo[0]) >> np.uint32(8), kind="stable")
    for k, g in enumerate(groups(n, d)):
        if not g:
            continue
        grp = np.arange(n) >> g
        key = (grp.astype(np.uint64) << np.uint64(32)) | (order_key(lo[k])[order] >> np.uint32(8))
        order = order[np.argsort(key, kind="stable")]
    return order.astype(np.uint32)


@pytest.mark.parametrize("d,n", [(2, 65), (2, 129), (2, 4095), (2, 4097), (2, 12289), (2, 70001),
                                 (2, 700001), (2, 1500007), (3, 5001), (3, 100003), (3, 250007),
                                 (5, 33333)])
def test_plan_order(ctx, d, n):
    import torch
    rng = np.random.default_rng(n + d)
    lo = (rng.integers(-4000, 4000, size=(d, n)) * np.float32(0.25)).astype(np.float32)  # ties
    lo[:, :2] = -0.0
    hi = lo + np.float32(0.5)
    U = to_dev((lo, hi))
    ddm.ddm_build(ctx, U[0][:, :100].contiguous(), U[1][:, :100].contiguous())
    ddm.ddm_plan(ctx, U[0], U[1])
    order = torch.empty(n, dtype=torch.int32, device="cuda")
    ddm.ddm_plan_order(ctx, order)
    assert np.array_equal(order.cpu().numpy().view(np.uint32), plan_order(lo, d))


def test_batch_with_large_groups(ctx):
    """An instance of 300,000 extents (d = 3) has groups of 2^14 positions."""
    import torch
    inst = [W.uniform_fixed_length(n, m, 3, 2.0, seed=i) for i, (n, m) in
            enumerate([(40, 70), (300000, 260000), (5000, 1), (1, 4097)])]
    assert max(groups(300000, 3)) > 13
    ulo, uhi, uoff, slo, shi, soff = W.concat_instances(inst)
    U = to_dev((ulo, uhi, slo, shi))
    uo = torch.from_numpy(uoff.astype(np.int64)).cuda()
    so = torch.from_numpy(soff.astype(np.int64)).cuda()
    pairs = torch.empty((4000000, 2), dtype=torch.int32, device="cuda")
    po = torch.empty(len(inst) + 1, dtype=torch.int64, device="cuda")
    K = ddm.ddm_batch_match(ctx, U[0], U[1], uo, U[2], U[3], so, pairs, po)
    p, o = pairs[:K].cpu().numpy().view(np.uint32), po.cpu().numpy()
    for i, a in enumerate(inst):
        k, pu, ps = gpu_match(ctx, a)
        assert k == o[i + 1] - o[i]
        assert np.array_equal(p[o[i]:o[i + 1], 0], pu)
        assert np.array_equal(np.sort(keys(p[o[i]:o[i + 1], 0], p[o[i]:o[i + 1], 1])),
                              np.sort(keys(pu, ps)))
