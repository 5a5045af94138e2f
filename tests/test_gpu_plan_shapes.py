"""Packets of few updates and short record entries (GPU).

A plan of few updates walks the tree in packets of 4, 8 or 16 queries, by the
number of updates and SMs; the two record blocks of a packet are one entry of
the write pass while their records fit one block.  Both sides of every
threshold: update counts around each change of the packet size, and sets in
which some packets keep to short entries while a wide update fills blocks.
The replayed pairs equal the walking write pass element by element and the
oracle as a set; ordered chunks cut packets in the middle.
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
    ddm.ddm_set_tuning(h)
    ddm.ddm_destroy(h)


def sparse_with_wide(m, n, d, wide, seed):
    """About one hit per update, except `wide` updates that meet many."""
    rng = np.random.default_rng(seed)
    side = 1000.0 * (1.0 / n) ** (1.0 / d)

    def one(k):
        lo = rng.uniform(0, 1000.0, size=(d, k)).astype(np.float32)
        return lo, lo + np.float32(side)
    (slo, shi), (ulo, uhi) = one(n), one(m)
    w = rng.choice(m, size=min(wide, m), replace=False)
    ulo[:, w] = rng.uniform(0, 200.0, size=(d, len(w))).astype(np.float32)
    uhi[:, w] = np.float32(900.0)
    return tuple(np.ascontiguousarray(a) for a in (ulo, uhi, slo, shi))


def sizes():
    import torch
    sms = torch.cuda.get_device_properties(0).multi_processor_count if torch.cuda.is_available() else 152
    t = sms * 16
    return [1, 5, 8 * (t - 1), 8 * (t - 1) + 1, 16 * (t - 1) + 1, 32 * (t - 1), 32 * (t - 1) + 1]


@pytest.mark.parametrize("which", range(7))
@pytest.mark.parametrize("d", [1, 2])
def test_packet_sizes(ctx, which, d):
    import torch
    m, n = sizes()[which], 20011
    arrays = sparse_with_wide(m, n, d, wide=7, seed=which)
    K, pu, ps = gpu_match(ctx, arrays)
    ddm.ddm_set_tuning(ctx, replay=0)
    Kw, wu, ws = gpu_match(ctx, arrays)
    ddm.ddm_set_tuning(ctx)
    assert K == Kw and np.array_equal(pu, wu) and np.array_equal(ps, ws)
    if m < 40000:
        _, ou, os_ = oracle.itm_pairs(*arrays)
        assert np.array_equal(np.sort(keys(pu, ps)), np.sort(keys(ou, os_)))
    # ordered chunks whose ends fall inside packets
    U = to_dev(arrays)
    ddm.ddm_build(ctx, U[2], U[3])
    assert ddm.ddm_plan(ctx, U[0], U[1]) == K
    order = torch.empty(m, dtype=torch.int32, device="cuda")
    offs = torch.empty(m + 1, dtype=torch.int64, device="cuda")
    ddm.ddm_plan_order(ctx, order, offs)
    oo = offs.cpu().numpy()
    want = np.argsort(np.argsort(order.cpu().numpy())[pu], kind="stable")
    ids = torch.empty(max(K, 1), dtype=torch.int32, device="cuda")
    for b, e in [(0, m), (m // 3, m // 3 + 3), (m // 2 + 1, m)]:
        e = min(e, m)
        b = min(b, e)
        k = ddm.ddm_write_ordered_ids(ctx, b, e, ids)
        assert k == oo[e] - oo[b]
        assert np.array_equal(ids[:k].cpu().numpy().view(np.uint32), ps[want][oo[b]:oo[e]])


@pytest.mark.parametrize("records", [511, 512, 513, 1024, 1025])
def test_entry_limit(ctx, records):
    """One packet whose records just fit one block, or do not: two updates of
    different halves share them; every leaf gives each a record."""
    leaves = (records + 1) // 2
    n = leaves * 32
    slo = np.arange(n, dtype=np.float32)[None, :]
    shi = slo.copy()
    # plan order is by lower bound: positions 0 and 16 of the first packet hold
    # the wide updates; the others lie outside, enough of them for packets of 32
    m = sizes()[-1]
    ulo = (n + 10.0 + np.arange(m, dtype=np.float64)).astype(np.float32)[None, :].copy()
    ulo[0, :20] = -20 + np.arange(20)
    uhi = ulo.copy()
    uhi[0, 0] = n
    uhi[0, 16] = n if records % 2 == 0 else n - 33   # one leaf less
    arrays = (ulo, uhi, slo, shi)
    K, pu, ps = gpu_match(ctx, arrays)
    _, ou, os_ = oracle.itm_pairs(*arrays)
    assert K == len(ou)
    assert np.array_equal(np.sort(keys(pu, ps)), np.sort(keys(ou, os_)))


@pytest.mark.parametrize("n", [1, 2, 3, 4, 5, 31, 63, 64, 65, 2047, 2049, 2051, 6144, 6145, 8191, 8192, 8193])
def test_order_by_counting(ctx, n):
    """Tree and plan order of small sets, around the staged chunk of keys, the
    extents of a CTA and the switch to the radix sort, with ties and signed
    zeros, against numpy's stable sorts (d = 1) and the oracle (d = 2)."""
    import torch
    from tests.test_gpu_parity import order_key
    rng = np.random.default_rng(n)
    lo = rng.integers(-9, 9, size=(1, n)).astype(np.float32) * np.float32(0.5)
    hi = lo + rng.integers(0, 3, size=(1, n)).astype(np.float32)
    lo[0, : n // 7] = -0.0
    hi = np.maximum(lo, hi)
    S = to_dev((lo, hi))
    ddm.ddm_build(ctx, S[0], S[1])
    order = torch.empty(n, dtype=torch.int32, device="cuda")
    ddm.ddm_tree_export(ctx, order)
    want = np.lexsort((np.arange(n), order_key(hi[0]), order_key(lo[0])))
    assert np.array_equal(order.cpu().numpy(), want)
    ddm.ddm_plan(ctx, S[0], S[1])
    ddm.ddm_plan_order(ctx, order)
    want = np.argsort(order_key(lo[0]) >> np.uint32(8), kind="stable")
    assert np.array_equal(order.cpu().numpy(), want)
    bad = S[1].clone()
    bad[0, n - 1] = float("nan")
    with pytest.raises(ddm.DDMError) as e:
        ddm.ddm_build(ctx, S[0], bad)
    assert e.value.code == ddm.DDM_ERR_EXTENT
    arrays = sparse_with_wide(n, n, 2, wide=1, seed=n)
    K, pu, ps = gpu_match(ctx, arrays)
    _, ou, os_ = oracle.itm_pairs(*arrays)
    assert np.array_equal(np.sort(keys(pu, ps)), np.sort(keys(ou, os_)))
