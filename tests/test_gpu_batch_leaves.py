"""Batches whose instances start leaves of their own (GPU).

With 128 or more subscriptions per instance on average, every instance's
subscriptions start a new leaf and its last leaf is filled up with empty
positions.  Instances of 0, 1, 31, 32, 33 ... subscriptions, unbounded extents
(an empty position must not meet a query reaching to infinity) and signed
zeros, both rules, replay and walking write, the compare loops (d > 3) and the
rank tables (d <= 3): each instance's pairs are the oracle's, grouped by update
and, for d = 1, in the order of the batched sort.
"""
import numpy as np
import pytest

import oracle
import paper_1309_3458_gb300 as ddm
from paper_1309_3458_gb300 import workloads as W
from tests.helpers import keys, to_dev
from tests.test_gpu_parity import order_key

pytestmark = pytest.mark.gpu

SUBS = [0, 1, 31, 32, 33, 64, 65, 0, 0, 1023, 1025, 300, 5, 2]
UPDS = [3, 40, 0, 33, 700, 1, 64, 9, 0, 2000, 31, 300, 5, 1]


@pytest.fixture(scope="module")
def ctx():
    import __graft_entry__
    __graft_entry__.build()
    h = ddm.ddm_create(0)
    yield h
    ddm.ddm_set_tuning(h)
    ddm.ddm_set_tiling(h)
    ddm.ddm_destroy(h)


def instances(d, seed):
    rng = np.random.default_rng(seed)

    def one(k):
        lo = rng.integers(-20, 20, size=(d, k)).astype(np.float32)
        hi = lo + rng.integers(0, 30, size=(d, k)).astype(np.float32)
        lo[:, rng.random(k) < 0.1] = -0.0
        hi = np.maximum(lo, hi)
        lo[:, rng.random(k) < 0.1] = -np.inf
        hi[:, rng.random(k) < 0.1] = np.inf
        up = rng.random(k) < 0.05     # the point at infinity
        lo[:, up] = hi[:, up] = np.inf
        return np.ascontiguousarray(lo), np.ascontiguousarray(hi)
    return [one(m) + one(n) for n, m in zip(SUBS, UPDS)]


@pytest.mark.parametrize("flags", [ddm.DDM_CLOSED, ddm.DDM_OPEN])
@pytest.mark.parametrize("d", [1, 2, 3, 4])
@pytest.mark.parametrize("replay,swap_min", [(1, 12), (1, 1), (0, 33)])
def test_instances_on_whole_leaves(ctx, d, flags, replay, swap_min):
    import torch
    assert sum(SUBS) >= 128 * len(SUBS)
    inst = instances(d, seed=10 * d + flags)
    ulo, uhi, uoff, slo, shi, soff = W.concat_instances(inst)
    U = to_dev((ulo, uhi, slo, shi))
    uo = torch.from_numpy(uoff.astype(np.int64)).cuda()
    so = torch.from_numpy(soff.astype(np.int64)).cuda()
    ddm.ddm_set_tuning(ctx, replay=replay)
    ddm.ddm_set_tiling(ctx, swap_min=swap_min)
    pairs = torch.empty((4000000, 2), dtype=torch.int32, device="cuda")
    po = torch.empty(len(inst) + 1, dtype=torch.int64, device="cuda")
    K = ddm.ddm_batch_match(ctx, U[0], U[1], uo, U[2], U[3], so, pairs, po, flags=flags)
    p, o = pairs[:K].cpu().numpy().view(np.uint32), po.cpu().numpy()
    assert o[-1] == K
    for i, a in enumerate(inst):
        got = p[o[i]:o[i + 1]]
        if UPDS[i] == 0 or SUBS[i] == 0:
            assert len(got) == 0
            continue
        _, ou, os_ = oracle.itm_pairs(*a, flags=flags)
        assert np.array_equal(np.sort(keys(got[:, 0], got[:, 1])), np.sort(keys(ou, os_)))
        assert (np.diff(got[:, 0].astype(np.int64)) >= 0).all()
        if d == 1:  # the batched order: by the top 24 bits of the lower bound's key, ties by id
            rank = np.argsort(np.argsort(order_key(a[2][0]) >> np.uint32(8), kind="stable"))
            at = got[:, 0].astype(np.int64) * (1 << 20) + rank[got[:, 1]]
            assert (np.diff(at) > 0).all()
