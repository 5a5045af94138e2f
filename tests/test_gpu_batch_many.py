"""Batches of more instances than one CTA plans (GPU).

Up to 4,096 instances are planned by one CTA, more by one CTA per 4,096 with the
sums of those before.  A batch on either side of the limit gives, instance by
instance and pair by pair, what its two halves give in calls of their own (one
CTA each): instances of a few extents, thousands of empty ones in a row (behind
which the instance of a position is searched, not walked to) and some with
several re-sort groups, with and without whole leaves per instance.
"""
import numpy as np
import pytest

import oracle
import paper_1309_3458_gb300 as ddm
from tests.helpers import keys, to_dev

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def ctx():
    import __graft_entry__
    __graft_entry__.build()
    h = ddm.ddm_create(0)
    yield h
    ddm.ddm_destroy(h)


def extents(rng, d, n):
    lo = rng.integers(0, 3000, size=(d, n)).astype(np.float32)
    return lo, lo + rng.integers(0, 40, size=(d, n)).astype(np.float32)


def call(ctx, d, u, su, s, ss):
    """Batched match of instances of sizes su / ss; pairs and instance offsets."""
    import torch
    off = [torch.from_numpy(np.concatenate([[0], np.cumsum(x)]).astype(np.int64)).cuda() for x in (su, ss)]
    U, S = to_dev(u), to_dev(s)
    po = torch.empty(len(su) + 1, dtype=torch.int64, device="cuda")
    pairs = torch.empty((40000000 if d == 1 else 3000000, 2), dtype=torch.int32, device="cuda")
    K = ddm.ddm_batch_match(ctx, U[0], U[1], off[0], S[0], S[1], off[1], pairs, po)
    return pairs[:K].cpu().numpy().view(np.uint32), po.cpu().numpy()


@pytest.mark.parametrize("d,count,mean", [(1, 4097, 3), (2, 4096, 3), (2, 4097, 3), (2, 8193, 5), (3, 12289, 2),
                                          (2, 4099, 140), (5, 4097, 3)])
def test_many_instances(ctx, d, count, mean):
    rng = np.random.default_rng(count + d)
    ss, su = rng.integers(0, 2 * mean + 1, count), rng.integers(0, 8, count)
    if mean < 128:  # a long run of empty instances, then large ones
        ss[count // 4: count // 4 + 3000] = 0
        su[count // 4: count // 4 + 3000] = 0
    else:
        ss = np.maximum(ss, 129)
    for i, n in ((0, 20011), (count // 4 + 3000, 9001), (count - 2, 70001)):
        ss[i], su[i] = n, n // 2
    u, s = extents(rng, d, su.sum()), extents(rng, d, ss.sum())
    pairs, off = call(ctx, d, u, su, s, ss)
    h = count // 2
    cu, cs = su[:h].sum(), ss[:h].sum()
    a, ao = call(ctx, d, [x[:, :cu] for x in u], su[:h], [x[:, :cs] for x in s], ss[:h])
    b, bo = call(ctx, d, [x[:, cu:] for x in u], su[h:], [x[:, cs:] for x in s], ss[h:])
    assert np.array_equal(off, np.concatenate([ao, ao[-1] + bo[1:]]))
    assert np.array_equal(pairs, np.concatenate([a, b]))
    if d == 1:  # 3.3e7 pairs
        return
    i = count - 2  # one large instance against the oracle
    eu, es = su[:i].sum(), ss[:i].sum()
    _, ou, os_ = oracle.itm_pairs(*[np.ascontiguousarray(x[:, e:e + n]) for x, e, n in
                                    ((u[0], eu, su[i]), (u[1], eu, su[i]), (s[0], es, ss[i]), (s[1], es, ss[i]))])
    got = pairs[off[i]:off[i + 1]]
    assert np.array_equal(np.sort(keys(got[:, 0], got[:, 1])), np.sort(keys(ou, os_)))
