"""A wait of the plan's scan that runs out (failure detection without a fault).

The tiles of a plan's offset scan wait for the tiles before them, boundedly.
With offsets that miss a tile's sum the total is too small and later offsets
too large against it, so no write may place pairs by them: every write form
reports the timeout and leaves the output buffer (and the words behind it) as
it was, until the next plan.
"""
import pytest

import paper_1309_3458_gb300 as ddm
from paper_1309_3458_gb300 import workloads as W


def test_null_and_range_errors_without_gpu():
    lib = ddm.lib()
    assert lib.ddm_debug_scan_timeout(None, 1, None) == ddm.DDM_ERR_ARG


def timed_out(call, *args, **kw):
    with pytest.raises(ddm.DDMError) as e:
        call(*args, **kw)
    assert e.value.code == ddm.DDM_ERR_TIMEOUT


@pytest.mark.gpu
@pytest.mark.parametrize("replay", [1, 0])
@pytest.mark.parametrize("m", [4097, 3 * 4096, 150001])
def test_writes_after_a_failed_scan(m, replay):
    import torch
    from tests.helpers import to_dev
    ctx = ddm.ddm_create(0)
    try:
        ddm.ddm_set_tuning(ctx, replay=replay)
        U = to_dev(W.uniform_fixed_length(3000, m, 2, 50.0, seed=m))
        ddm.ddm_build(ctx, U[2], U[3])
        with pytest.raises(ddm.DDMError) as e:
            ddm.ddm_debug_scan_timeout(ctx, 64)
        assert e.value.code == ddm.DDM_ERR_STATE
        K = ddm.ddm_plan(ctx, U[0], U[1])
        want = torch.full((K + 64, 2), -7, dtype=torch.int32, device="cuda")
        assert ddm.ddm_write(ctx, 0, m, want[:K]) == K and int((want[K:] != -7).sum()) == 0

        timed_out(ddm.ddm_debug_scan_timeout, ctx, 64)
        out = torch.full((K + 64, 2), -7, dtype=torch.int32, device="cuda")
        k = torch.zeros(1, dtype=torch.int64, device="cuda")
        err = torch.zeros(1, dtype=torch.int32, device="cuda")
        timed_out(ddm.ddm_write, ctx, 0, m, out[:K])
        timed_out(ddm.ddm_write, ctx, m // 2, m, out[:K])
        timed_out(ddm.ddm_write_ordered, ctx, 0, m, out[:K])
        timed_out(ddm.ddm_write_ordered_ids, ctx, 1, m, out.view(-1)[:K])
        timed_out(ddm.ddm_chunk_end, ctx, 0, K)
        timed_out(ddm.ddm_chunk_end_ordered, ctx, 0, K)
        ddm.ddm_write_async(ctx, 0, m, out[:K], k, err)
        assert int(err[0]) & 2
        assert int((out != -7).sum()) == 0

        assert ddm.ddm_plan(ctx, U[0], U[1]) == K  # the next plan is whole again
        assert ddm.ddm_write(ctx, 0, m, out[:K]) == K
        assert torch.equal(out, want)
    finally:
        ddm.ddm_destroy(ctx)
