"""The workspace of the one-shot calls' second ordering is given back (GPU).

A one-shot call orders its two sets side by side, with a workspace for each.
Afterwards the second one must not stand in the way of what fits without it:
under an allocation limit that just admits a staged build and plan (after a
smaller staged one), the same build and plan fit after a smaller one-shot call.
"""
import pytest

import paper_1309_3458_gb300 as ddm
from paper_1309_3458_gb300 import workloads as W

pytestmark = pytest.mark.gpu
MIB = 1 << 20


def attempt(limit, small, large, one_shot):
    """K of the large staged matching under the limit, None if it does not fit."""
    import torch
    h = ddm.ddm_create(0)
    try:
        ddm.ddm_set_replay_budget(h, 0)
        ddm.ddm_debug_set_alloc_limit(h, limit)
        if one_shot:
            pairs = torch.empty((1000000, 2), dtype=torch.int32, device="cuda")
            ddm.ddm_match(h, *small, pairs)
        else:
            ddm.ddm_build(h, small[2], small[3])
            ddm.ddm_plan(h, small[0], small[1])
        ddm.ddm_build(h, large[2], large[3])
        return ddm.ddm_plan(h, large[0], large[1])
    except ddm.DDMError as e:
        assert e.code == ddm.DDM_ERR_NOMEM
        return None
    finally:
        ddm.ddm_destroy(h)


@pytest.mark.parametrize("d", [1, 2])
def test_staged_call_after_a_one_shot_call(d):
    import __graft_entry__
    from tests.helpers import to_dev
    __graft_entry__.build()
    small = to_dev(W.uniform_fixed_length(90000, 90000, d, 1.0, seed=1))
    large = to_dev(W.uniform_fixed_length(130000, 130000, d, 1.0, seed=2))
    K = attempt(0, small, large, one_shot=False)
    lo, hi = 1, 256  # MiB: lo does not fit, hi does
    while hi - lo > 1:
        mid = (lo + hi) // 2
        lo, hi = (lo, mid) if attempt(mid * MIB, small, large, one_shot=False) == K else (mid, hi)
    assert attempt(hi * MIB, small, large, one_shot=True) == K
