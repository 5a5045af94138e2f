"""The two forms of the write pass from records (GPU).

Whether a plan's record entries count as short (few pairs each on average: a
packet's two first blocks are then one entry) is decided by the whole plan, and
every range of it follows.  Plans on both sides of the limit that mix updates
meeting almost everything with updates meeting almost nothing, so that ranges of
the plan order are far denser or sparser than the plan: pairs in plan order, the
compressed output and pairs by update id equal the walking write pass.
"""
import numpy as np
import pytest

import oracle
import paper_1309_3458_gb300 as ddm
from tests.helpers import gpu_match, keys, to_dev

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def ctx():
    import __graft_entry__
    __graft_entry__.build()
    h = ddm.ddm_create(0)
    yield h
    ddm.ddm_destroy(h)


def mixed(d, m, n, wide, seed):
    """`wide` updates over most of the space's first half, the others short; the
    lower bounds of the wide ones come first in the plan order."""
    rng = np.random.default_rng(seed)
    side = np.float32(1000.0 * (1.0 / n) ** (1.0 / d))
    slo = rng.uniform(0, 1000.0, size=(d, n)).astype(np.float32)
    ulo = rng.uniform(0, 1000.0, size=(d, m)).astype(np.float32)
    uhi = ulo + side
    ulo[:, :wide] = rng.uniform(0, 1.0, size=(d, wide)).astype(np.float32)
    uhi[:, :wide] = np.float32(500.0)
    p = rng.permutation(m)
    return tuple(np.ascontiguousarray(a) for a in (ulo[:, p], uhi[:, p], slo, slo + side))


def written(ctx, U, K, m, ranges):
    import torch
    order = torch.empty(m, dtype=torch.int32, device="cuda")
    offs = torch.empty(m + 1, dtype=torch.int64, device="cuda")
    ddm.ddm_build(ctx, U[2], U[3])
    assert ddm.ddm_plan(ctx, U[0], U[1]) == K
    ddm.ddm_plan_order(ctx, order, offs)
    out = [order.cpu().numpy(), offs.cpu().numpy()]
    for b, e in ranges:
        k = int(offs[e] - offs[b])
        pairs = torch.full((k + 1, 2), -1, dtype=torch.int32, device="cuda")
        ids = torch.full((k + 1,), -1, dtype=torch.int32, device="cuda")
        assert ddm.ddm_write_ordered(ctx, b, e, pairs[:k]) == k
        assert ddm.ddm_write_ordered_ids(ctx, b, e, ids[:k]) == k
        out += [pairs.cpu().numpy(), ids.cpu().numpy()]
        assert np.array_equal(out[-2][:, 1], out[-1])
    whole = torch.empty((K, 2), dtype=torch.int32, device="cuda")
    assert ddm.ddm_write(ctx, 0, m, whole) == K
    part = torch.empty((K, 2), dtype=torch.int32, device="cuda")
    k = ddm.ddm_write(ctx, m // 3, m // 2, part)
    return out + [whole.cpu().numpy(), part[:k].cpu().numpy()]


@pytest.mark.parametrize("d,m,n,wide", [(1, 3, 5000, 2), (1, 81000, 9000, 0), (1, 81000, 9000, 17),
                                        (1, 81000, 9000, 60), (1, 81000, 9000, 137), (1, 81000, 9000, 2000),
                                        (2, 2500, 30011, 100), (3, 79000, 12000, 900)])
def test_ranges_of_mixed_plans(ctx, d, m, n, wide):
    arrays = mixed(d, m, n, wide, seed=m + wide)
    U = to_dev(arrays)
    K = ddm.ddm_count(ctx, *U)
    cut = max(wide, 1)
    ranges = [(0, m), (0, cut), (cut // 2, min(cut + 40, m)), (min(cut, m - 1), m), (m // 2, m // 2)]
    ddm.ddm_set_tuning(ctx, replay=1)
    got = written(ctx, U, K, m, ranges)
    ddm.ddm_set_tuning(ctx, replay=0)
    want = written(ctx, U, K, m, ranges)
    ddm.ddm_set_tuning(ctx)
    for a, b in zip(got, want):
        assert np.array_equal(a, b)
    Km, pu, ps = gpu_match(ctx, arrays)
    Ko, ou, os_ = oracle.itm_pairs(*arrays)
    assert Km == Ko == K
    assert np.array_equal(np.sort(keys(pu, ps)), np.sort(keys(ou, os_)))
