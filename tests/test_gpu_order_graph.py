"""ddm_plan_order in a CUDA graph (GPU): a replay gives the order and offsets of
the context's latest plan of that size, whether a staged call or a one-shot call
made it, and whichever had made the plan at capture."""
import pytest

import paper_1309_3458_gb300 as ddm
from paper_1309_3458_gb300 import workloads as W

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("m", [300, 9001])
@pytest.mark.parametrize("first", ["staged", "one-shot"])
def test_replay_after_plans_of_either_kind(first, m):
    import __graft_entry__
    import torch
    from tests.helpers import to_dev
    __graft_entry__.build()
    sets = [to_dev(W.uniform_fixed_length(4000, m, 2, 20.0, seed=s)) for s in range(3)]
    h = ddm.ddm_create(0)
    try:
        pairs = torch.empty((2000000, 2), dtype=torch.int32, device="cuda")

        def plan(kind, x):
            if kind == "staged":
                ddm.ddm_build(h, x[2], x[3])
                ddm.ddm_plan(h, x[0], x[1])
            else:
                ddm.ddm_match(h, *x, pairs)

        plan(first, sets[0])
        order = torch.zeros(m, dtype=torch.int32, device="cuda")
        offs = torch.zeros(m + 1, dtype=torch.int64, device="cuda")
        stream, graph = torch.cuda.Stream(), torch.cuda.CUDAGraph()
        torch.cuda.synchronize()
        with torch.cuda.graph(graph, stream=stream):
            ddm.ddm_plan_order(h, order, offs, stream=stream)
        for kind, x in [("one-shot", sets[1]), ("staged", sets[2]), ("one-shot", sets[0]), ("one-shot", sets[2])]:
            plan(kind, x)
            graph.replay()
            torch.cuda.synchronize()
            want = [torch.zeros_like(order), torch.zeros_like(offs)]
            ddm.ddm_plan_order(h, *want)
            torch.cuda.synchronize()
            assert torch.equal(order, want[0]) and torch.equal(offs, want[1])
            k = int(offs[-1])
            out = torch.empty((k, 2), dtype=torch.int32, device="cuda")
            assert ddm.ddm_write_ordered(h, 0, m, out) == k
    finally:
        ddm.ddm_destroy(h)
