"""Record budgets below a first block for every chain of packets (GPU).

With room for them every chain of a plan's packets owns a block from the start;
with less, every block is handed out, so that a plan whose hits lie in few
packets is still recorded (its write launches the replay alone).  Pairs by
update id, in plan order, of sub-ranges and the compressed output are those of
the walking write pass at every budget.
"""
import numpy as np
import pytest

import paper_1309_3458_gb300 as ddm
from tests.helpers import to_dev

pytestmark = pytest.mark.gpu
BLOCK = 5184 + 4 + 8 + 16  # bytes of the arena per block


def sets(d, m, n, hits, seed):
    """`hits` updates that meet about a quarter of the subscriptions, neighbours
    in the plan order, and the rest meeting none."""
    rng = np.random.default_rng(seed)
    slo = rng.uniform(0, 1000.0, size=(d, n)).astype(np.float32)
    ulo = rng.uniform(2000.0, 9000.0, size=(d, m)).astype(np.float32)
    uhi = ulo + np.float32(1.0)
    ulo[:, :hits] = rng.uniform(0, 5.0, size=(d, hits)).astype(np.float32)
    uhi[:, :hits] = np.float32(1000.0 * 0.25 ** (1.0 / d))
    p = rng.permutation(m)
    return tuple(np.ascontiguousarray(x) for x in (ulo[:, p], uhi[:, p], slo, slo + np.float32(1.0)))


def outputs(h, U, m, ranges):
    """Pairs by id (all and a part), and pairs and ids of ranges of the plan order."""
    import torch
    ddm.ddm_build(h, U[2], U[3])
    K = ddm.ddm_plan(h, U[0], U[1])
    pairs = torch.empty((K + 1, 2), dtype=torch.int32, device="cuda")
    ids = torch.empty(K + 1, dtype=torch.int32, device="cuda")
    out = []
    for b, e in ranges:
        for call, buf in ((ddm.ddm_write_ordered, pairs), (ddm.ddm_write_ordered_ids, ids)):
            out.append(buf[:call(h, b, e, buf)].cpu().numpy().copy())
    out.append(pairs[:ddm.ddm_write(h, m // 3, m, pairs)].cpu().numpy().copy())
    a = ddm.ddm_debug_launch_count()
    assert ddm.ddm_write(h, 0, m, pairs) == K
    launches = ddm.ddm_debug_launch_count() - a
    return out + [pairs[:K].cpu().numpy()], launches


@pytest.mark.parametrize("d,m,n,hits", [(1, 90001, 2000, 0), (1, 90001, 2000, 40), (2, 90001, 3000, 33), (3, 90001, 3000, 3),
                                        (2, 90001, 3000, 400)])
def test_budgets(d, m, n, hits):
    import __graft_entry__
    __graft_entry__.build()
    U = to_dev(sets(d, m, n, hits, seed=hits))
    ranges = [(0, m), (0, hits + 7), (3, 40), (m // 2, m)]
    chains = 2 * ((m + 31) // 32)

    def run(budget, replay=1):
        h = ddm.ddm_create(0)
        try:
            ddm.ddm_set_replay_budget(h, budget)
            ddm.ddm_set_tuning(h, replay=replay)
            outputs(h, U, m, ranges)  # the second plan sizes its records by the first
            return outputs(h, U, m, ranges)
        finally:
            ddm.ddm_destroy(h)

    want, _ = run(0, replay=0)
    for blocks in (1, 17, 300, chains - 1, chains, chains + 3, 3 * chains):
        got, launches = run(blocks * BLOCK)
        for x, y in zip(got, want):
            assert np.array_equal(x, y)
        # 2,000 subscriptions are 63 leaves: a record of every update with hits
        # and leaf, in blocks of 512 per half packet
        need = (hits * ((n + 31) // 32) // 512 + 2 * (hits // 32 + 2)) if hits else 0
        if chains > blocks >= 2 * need and blocks > 1:
            assert launches == 1, (blocks, launches)
