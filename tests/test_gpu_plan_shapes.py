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


def test_staged_calls_after_one_shot(ctx):
    """A one-shot call leaves a plan whose order's offsets and entries are made
    by the first staged call that needs them: the same as ddm_plan's."""
    import torch
    m, n = 5003, 4001
    U = to_dev(sparse_with_wide(m, n, 2, wide=9, seed=3))
    order = [torch.empty(m, dtype=torch.int32, device="cuda") for _ in range(3)]
    offs = [torch.empty(m + 1, dtype=torch.int64, device="cuda") for _ in range(3)]
    ids = [None] * 3
    for i in range(3):
        if i == 0:
            ddm.ddm_build(ctx, U[2], U[3])
            K = ddm.ddm_plan(ctx, U[0], U[1])
        elif i == 1:
            pairs = torch.empty((K, 2), dtype=torch.int32, device="cuda")
            assert ddm.ddm_match(ctx, *U, pairs) == K
        else:
            assert ddm.ddm_count(ctx, *U) == K
        ids[i] = torch.empty(K, dtype=torch.int32, device="cuda")
        e = ddm.ddm_chunk_end_ordered(ctx, 0, K // 2)
        k = ddm.ddm_write_ordered_ids(ctx, 0, e, ids[i])
        ddm.ddm_plan_order(ctx, order[i], offs[i])
        ddm.ddm_write_ordered_ids(ctx, e, m, ids[i][k:])
    for i in (1, 2):
        assert torch.equal(order[i], order[0]) and torch.equal(offs[i], offs[0])
        assert torch.equal(ids[i], ids[0])


def test_scratch_limits():
    """With room for one ordering workspace but not for two, a one-shot call
    orders its sets one after the other: under every limit it gives the pairs
    of the unlimited call or DDM_ERR_NOMEM, and the context stays usable."""
    import torch
    U = to_dev(sparse_with_wide(20011, 30011, 2, wide=5, seed=8))
    h = ddm.ddm_create(0)
    K = ddm.ddm_count(h, *U)
    want = torch.empty((K, 2), dtype=torch.int32, device="cuda")
    assert ddm.ddm_match(h, *U, want) == K
    ddm.ddm_destroy(h)
    ok = failed = 0
    for mib in [1, 2, 3, 4, 5, 6, 7, 8, 10, 12, 16, 24, 32, 64]:
        h = ddm.ddm_create(0)
        ddm.ddm_debug_set_alloc_limit(h, mib << 20)
        pairs = torch.empty((K, 2), dtype=torch.int32, device="cuda")
        try:
            assert ddm.ddm_match(h, *U, pairs) == K
            assert torch.equal(pairs, want)
            ok += 1
        except ddm.DDMError as e:
            assert e.code == ddm.DDM_ERR_NOMEM
            failed += 1
        ddm.ddm_debug_set_alloc_limit(h, 0)
        assert ddm.ddm_match(h, *U, pairs) == K and torch.equal(pairs, want)
        ddm.ddm_destroy(h)
    assert ok >= 3 and failed >= 1


@pytest.mark.parametrize("n", [8193, 10000, 40007, 1300001])
@pytest.mark.parametrize("values", [1, 60, 2000, 100000])
def test_d1_tree_order_with_ties(ctx, n, values):
    """Lower bounds that tie in runs of every length around the limit of the
    short way, sampled as heavily tied or not: the exact (lower, upper, id)
    order either way."""
    import torch
    from tests.test_gpu_parity import order_key
    rng = np.random.default_rng(n + values)
    lo = (rng.integers(0, values, size=(1, n)) - values // 2).astype(np.float32)
    lo[0, :40] = values            # one run of 40 among shorter ones
    hi = lo + rng.integers(0, 4, size=(1, n)).astype(np.float32)
    S = to_dev((lo, hi))
    ddm.ddm_build(ctx, S[0], S[1])
    order = torch.empty(n, dtype=torch.int32, device="cuda")
    ddm.ddm_tree_export(ctx, order)
    want = np.lexsort((np.arange(n), order_key(hi[0]), order_key(lo[0])))
    assert np.array_equal(order.cpu().numpy(), want)
