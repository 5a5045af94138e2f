"""Performance cases: matching as a user of the library runs it.

Every case draws its extents on the GPU from the seed, in the shapes of
``paper_1309_3458_gb300/workloads.py`` (uniform extents of equal length with
overlapping degree alpha, log-normal extents around Gaussian clusters, batches
of independent problems), and makes one call or one short sequence of calls of
the public API.  Outputs are whole: every pair (or subscription id), the
offsets and orders a staged call hands out, and the counts.  They are whole
numbers, so there is nothing to compare in 64 bits: they have to be equal.

A case's fields:

* ``kind``  -- the call sequence (see the ``_run_*`` functions);
* ``dist``  -- "uniform" or "clustered";
* ``d``, ``m``, ``n`` -- dimensions, updates, subscriptions; ``alpha``;
* further fields of single kinds (flags, chunks, instances, moved extents).
"""
import math
import random

import numpy as np
import torch

import paper_1309_3458_gb300 as ddm
from paper_1309_3458_gb300.dynamic import DynamicMatching

L = 1.0e6  # side of the routing space
CLUSTERS, CLUSTER_SIGMA, LN_SIGMA = 64, 0.02, 1.0
# Pairs of the clustered d = 3 workload at N = 1e7, alpha = 100 (n = m = 5e6):
# the hit probability at another size scales with alpha / N.
CLUSTERED_P = 4.4147e10 / 2.5e13


def listed():
    return [
        # one small problem: the size of the paper's smallest experiment, where
        # launches and latencies count
        {"name": "match_d1_1e4", "kind": "match", "dist": "uniform", "d": 1, "m": 5000, "n": 5000,
         "alpha": 1.0, "open": False, "swap": False},
        # the paper's N = 1e6 setting with the densest overlap it uses
        {"name": "match_d1_1e6_a100", "kind": "match", "dist": "uniform", "d": 1, "m": 500000,
         "n": 500000, "alpha": 100.0, "open": False, "swap": False},
        # the largest d = 1 sweep point (Fig. 7's shape), sparse output
        {"name": "match_d1_5e7", "kind": "match", "dist": "uniform", "d": 1, "m": 25000000,
         "n": 25000000, "alpha": 1.0, "open": False, "swap": False},
        # two-dimensional regions, N = 1e6
        {"name": "match_d2_1e6", "kind": "match", "dist": "uniform", "d": 2, "m": 500000,
         "n": 500000, "alpha": 1.0, "open": False, "swap": False},
        # few subscribers against many updates: the tree over the updates, odd sizes
        {"name": "match_d2_swapped", "kind": "match", "dist": "uniform", "d": 2, "m": 600011,
         "n": 30011, "alpha": 10.0, "open": False, "swap": True},
        # more than three dimensions (the runtime-d kernels), strict comparison, odd sizes
        {"name": "match_d5_open", "kind": "match", "dist": "uniform", "d": 5, "m": 33333, "n": 70001,
         "alpha": 50.0, "open": True, "swap": False},
        # dense clustered regions in space, all pairs in one call
        {"name": "match_d3_clustered", "kind": "match", "dist": "clustered", "d": 3, "m": 250000,
         "n": 250000, "alpha": 100.0, "open": False, "swap": False},
        # the same kind of regions staged: build, plan, compressed output in chunks
        {"name": "stream_ids_d3", "kind": "stream", "dist": "clustered", "d": 3, "m": 500000,
         "n": 500000, "alpha": 100.0, "chunks": 3},
        # thousands of independent problems in one call
        {"name": "batch_4096", "kind": "batch", "d": 2, "instances": 4096, "size_lo": 100,
         "size_hi": 100000, "alpha": 1.0, "graph": False},
        # a real-time loop's batch of small problems, recorded in a CUDA graph
        {"name": "batch_graph_256", "kind": "batch", "d": 2, "instances": 256, "size_lo": 50,
         "size_hi": 5000, "alpha": 1.0, "graph": True},
        # one launch of the server: several requests against resident regions
        {"name": "serve_1e6", "kind": "serve", "dist": "uniform", "d": 2, "m": 31627, "n": 1000000,
         "alpha": 2.0, "requests": 4},
        # a tick of a simulation: some updates move, their rows are matched again
        {"name": "moved_2e5", "kind": "moved", "dist": "uniform", "d": 2, "m": 200000, "n": 200000,
         "alpha": 4.0, "moved": 3001},
    ]


def _log(rng, a, b):
    """A whole number, log-uniform in [a, b]."""
    return int(round(math.exp(rng.uniform(math.log(a), math.log(b)))))


def draw(rng):
    kind = rng.choice(["match", "match", "match", "clustered", "stream", "batch", "graph", "serve",
                       "moved"])
    if kind == "match":
        d = rng.choice([1, 1, 2, 2, 3, 5])
        top = {1: 20000000, 2: 4000000, 3: 1000000, 5: 60000}[d]
        m, n = _log(rng, 1000, top), _log(rng, 1000, top)
        # alpha up to 100, at most about 2e8 pairs
        case = {"kind": "match", "dist": "uniform", "d": d, "m": m, "n": n, "alpha": 1.0,
                "open": rng.random() < 0.25, "swap": rng.random() < 0.25}
        most = min(100.0, 2.0e8 / max(_expected_pairs(case), 1.0))
        case["alpha"] = round(math.exp(rng.uniform(math.log(0.01), math.log(max(most, 0.02)))), 4)
        return case
    if kind in ("clustered", "stream"):
        m, n = _log(rng, 20000, 400000), _log(rng, 20000, 400000)
        case = {"kind": "match" if kind == "clustered" else "stream", "dist": "clustered", "d": 3,
                "m": m, "n": n, "alpha": round(math.exp(rng.uniform(0.0, math.log(100.0))), 3)}
        if kind == "stream":
            case["chunks"] = rng.randint(1, 5)
        else:
            case["open"] = rng.random() < 0.25
            case["swap"] = False
        return case
    if kind in ("batch", "graph"):
        return {"kind": "batch", "d": rng.choice([1, 2, 2, 3]), "instances": _log(rng, 8, 2048),
                "size_lo": _log(rng, 20, 200), "size_hi": _log(rng, 400, 20000),
                "alpha": round(math.exp(rng.uniform(math.log(0.1), math.log(20.0))), 3),
                "graph": kind == "graph"}
    if kind == "serve":
        n = _log(rng, 50000, 2000000)
        return {"kind": "serve", "dist": "uniform", "d": rng.choice([1, 2, 3]),
                "m": _log(rng, 1000, 1000000), "n": n, "alpha": 2.0, "requests": rng.randint(1, 16)}
    n = _log(rng, 20000, 1000000)
    return {"kind": "moved", "dist": "uniform", "d": rng.choice([1, 2, 3]), "m": n,
            "n": _log(rng, 20000, 1000000), "alpha": round(rng.uniform(0.5, 20.0), 3),
            "moved": _log(rng, 16, n // 4)}


# ---- inputs ---------------------------------------------------------------

def _generator(seed):
    g = torch.Generator(device="cuda")
    g.manual_seed(seed)
    return g


def _side(case):
    """Length of a uniform extent: alpha = N * l**d / L**d."""
    return L * (case["alpha"] / (case["m"] + case["n"])) ** (1.0 / case["d"])


def _uniform(case, size, g):
    l = min(_side(case), 0.5 * L)
    # drawn in 64 bits and rounded, as the numpy generators do
    lo = (torch.rand((case["d"], size), generator=g, device="cuda", dtype=torch.float64) * (L - l)).float()
    return lo, lo + l


def _clustered(case, centres, size, g):
    d = case["d"]
    mu = (math.log(case["alpha"] * L ** d / (case["m"] + case["n"])) - d * LN_SIGMA ** 2 / 2.0) / d
    which = torch.randint(0, CLUSTERS, (size,), generator=g, device="cuda")
    c = centres[:, which] + CLUSTER_SIGMA * L * torch.randn((d, size), generator=g, device="cuda")
    c = c.clamp_(0.0, float(np.nextafter(np.float32(L), np.float32(0.0))))
    half = 0.5 * torch.exp(mu + LN_SIGMA * torch.randn((d, size), generator=g, device="cuda"))
    return c - half, c + half


def _sets(case, seed):
    """(upd_lo, upd_hi, sub_lo, sub_hi), float32 (d, count) on the GPU."""
    g = _generator(seed)
    if case["dist"] == "clustered":
        centres = L * torch.rand((case["d"], CLUSTERS), generator=g, device="cuda")
        s = _clustered(case, centres, case["n"], g)
        u = _clustered(case, centres, case["m"], g)
    else:
        s = _uniform(case, case["n"], g)
        u = _uniform(case, case["m"], g)
    return u[0], u[1], s[0], s[1]


def _batch_sizes(case):
    """Updates and subscriptions of every instance: sizes log-uniform, the
    same for every seed (only the extents are drawn from it)."""
    r = random.Random(case["instances"] * 1000003 + case["size_hi"])
    sizes = [_log(r, case["size_lo"], case["size_hi"]) for _ in range(case["instances"])]
    return [s // 2 for s in sizes], [s - s // 2 for s in sizes]


def _batch_set(case, counts, lengths, g):
    total, d = sum(counts), case["d"]
    l = torch.repeat_interleave(torch.tensor(lengths, device="cuda"),
                                torch.tensor(counts, device="cuda"), output_size=total)
    lo = torch.rand((d, total), generator=g, device="cuda") * (L - l)
    off = torch.from_numpy(np.concatenate([[0], np.cumsum(counts)]).astype(np.int64)).cuda()
    return lo, lo + l, off


class _Handle:
    """A context that goes with its state."""

    def __init__(self):
        self.h = ddm.ddm_create(torch.cuda.current_device())

    def __del__(self):
        ddm.ddm_destroy(self.h)


class _Dynamic:
    def __init__(self, *a, **k):
        self.dm = DynamicMatching(*a, **k)

    def __del__(self):
        self.dm.close()


def _room(expected):
    """Capacity of an output buffer: the expected pairs and some slack, as a
    program that knows its density allocates it (a call says when it is too
    small).  Passes return the whole buffer; its slack stays zero."""
    return int(1.25 * expected) + 20000


def _pairs(k):
    return torch.zeros((k, 2), dtype=torch.int32, device="cuda")


def prepare(case, seed):
    return {"match": _prep_match, "stream": _prep_stream, "batch": _prep_batch, "serve": _prep_serve,
            "moved": _prep_moved}[case["kind"]](case, seed)


def run(state):
    return state["run"](state)


# ---- one call for the whole matching --------------------------------------

def _prep_match(case, seed):
    ctx, sets = _Handle(), _sets(case, seed)
    flags = (ddm.DDM_OPEN if case["open"] else 0) | (ddm.DDM_SWAP_ROLES if case["swap"] else 0)
    return {"run": _run_match, "ctx": ctx, "sets": sets, "flags": flags,
            "pairs": _pairs(_room(_expected_pairs(case)))}


def _run_match(s):
    k = ddm.ddm_match(s["ctx"].h, *s["sets"], s["pairs"], flags=s["flags"])
    return {"k": k, "pairs": s["pairs"]}


# ---- resident tree, plan, compressed output in chunks of the plan's order --

def _prep_stream(case, seed):
    ctx, sets = _Handle(), _sets(case, seed)
    room, m = _room(_expected_pairs(case)), case["m"]
    return {"run": _run_stream, "ctx": ctx, "sets": sets, "chunk": room // case["chunks"] + case["n"],
            "ids": torch.zeros(room, dtype=torch.int32, device="cuda"),
            "order": torch.zeros(m, dtype=torch.int32, device="cuda"),
            "offsets": torch.zeros(m + 1, dtype=torch.int64, device="cuda")}


def _run_stream(s):
    h, (ulo, uhi, slo, shi) = s["ctx"].h, s["sets"]
    m = ulo.shape[1]
    ddm.ddm_build(h, slo, shi)
    k = ddm.ddm_plan(h, ulo, uhi)
    ddm.ddm_plan_order(h, s["order"], s["offsets"])
    at = written = 0
    while at < m:
        end = ddm.ddm_chunk_end_ordered(h, at, s["chunk"])
        written += ddm.ddm_write_ordered_ids(h, at, end, s["ids"][written:written + s["chunk"]])
        at = end
    return {"k": k, "order": s["order"], "offsets": s["offsets"], "ids": s["ids"]}


# ---- many independent problems in one call --------------------------------

def _prep_batch(case, seed):
    g, (ms, ns) = _generator(seed), _batch_sizes(case)
    lengths = [min(0.5 * L, L * (case["alpha"] / max(a + b, 1)) ** (1.0 / case["d"]))
               for a, b in zip(ms, ns)]
    slo, shi, soff = _batch_set(case, ns, lengths, g)
    ulo, uhi, uoff = _batch_set(case, ms, lengths, g)
    ctx = _Handle()
    s = {"run": _run_batch, "ctx": ctx, "args": (ulo, uhi, uoff, slo, shi, soff),
         "pairs": _pairs(_room(_expected_pairs(case))),
         "pair_off": torch.zeros(case["instances"] + 1, dtype=torch.int64, device="cuda")}
    if case["graph"]:
        s["run"] = _run_graph
        s["k"] = torch.zeros(1, dtype=torch.int64, device="cuda")
        s["err"] = torch.zeros(1, dtype=torch.int32, device="cuda")
        stream = torch.cuda.Stream()
        stream.wait_stream(torch.cuda.current_stream())

        def call():
            ddm.ddm_batch_match_async(ctx.h, *s["args"], s["pairs"], s["pair_off"], s["k"], s["err"],
                                      stream=stream)

        with torch.cuda.stream(stream):
            call()  # the workspace grows here, not while recording
        torch.cuda.synchronize()
        s["graph"] = torch.cuda.CUDAGraph()
        with torch.cuda.graph(s["graph"], stream=stream):
            call()
        torch.cuda.synchronize()
    return s


def _run_batch(s):
    k = ddm.ddm_batch_match(s["ctx"].h, *s["args"], s["pairs"], s["pair_off"])
    return {"k": k, "pairs": s["pairs"], "pair_off": s["pair_off"]}


def _run_graph(s):
    s["graph"].replay()
    return {"k": s["k"], "err": s["err"], "pairs": s["pairs"], "pair_off": s["pair_off"]}


# ---- a server's launch: requests against resident regions -----------------

def _prep_serve(case, seed):
    tree, ctx, (ulo, uhi, slo, shi) = _Handle(), _Handle(), _sets(case, seed)
    ddm.ddm_build(tree.h, slo, shi)
    ddm.ddm_attach(ctx.h, tree.h)
    r = case["requests"]
    cuts = np.array([case["m"] * (i * i) // (r * r) for i in range(r + 1)], dtype=np.int64)
    return {"run": _run_serve, "tree": tree, "ctx": ctx, "regions": (slo, shi), "updates": (ulo, uhi),
            "upd_off": torch.from_numpy(cuts).cuda(),
            "pair_off": torch.zeros(r + 1, dtype=torch.int64, device="cuda"),
            "pairs": _pairs(_room(_expected_pairs(case))), "k": torch.zeros(1, dtype=torch.int64, device="cuda"),
            "err": torch.zeros(1, dtype=torch.int32, device="cuda")}


def _run_serve(s):
    h, (ulo, uhi) = s["ctx"].h, s["updates"]
    ddm.ddm_plan_async(h, ulo, uhi)
    ddm.ddm_write_async(h, 0, ulo.shape[1], s["pairs"], s["k"], s["err"])
    ddm.ddm_pair_offsets_async(h, s["upd_off"], s["pair_off"])
    return {"k": s["k"], "err": s["err"], "pairs": s["pairs"], "pair_off": s["pair_off"]}


# ---- moved extents against the resident tree of the other set -------------

def _prep_moved(case, seed):
    ulo, uhi, slo, shi = _sets(case, seed)
    g = _generator(seed + 1)
    ids = torch.randperm(case["m"], generator=g, device="cuda")[:case["moved"]]
    step = _side(case) * torch.randn((case["d"], case["moved"]), generator=g, device="cuda")
    lo, hi = ulo[:, ids] + step, uhi[:, ids] + step
    hi = torch.maximum(lo, hi)
    return {"run": _run_moved, "dyn": _Dynamic(ulo, uhi, slo, shi), "ids": ids.to(torch.int32),
            "lo": lo, "hi": hi, "pairs": _pairs(_room(_expected_pairs(case) * case["moved"] / case["m"]))}


def _run_moved(s):
    dm = s["dyn"].dm
    k = dm.move_updates(s["ids"], s["lo"], s["hi"], s["pairs"])
    return {"k": k, "pairs": s["pairs"], "upd_lo": dm.U[0], "upd_hi": dm.U[1]}


# ---- what a pass cannot do without ----------------------------------------

def _expected_pairs(case):
    d = case["d"]
    if case["kind"] == "batch":
        return sum(_expected_pairs({"kind": "match", "dist": "uniform", "d": d, "m": a, "n": b,
                                    "alpha": case["alpha"]}) for a, b in zip(*_batch_sizes(case)))
    if case["dist"] == "clustered":
        N = case["m"] + case["n"]
        return case["m"] * case["n"] * CLUSTERED_P * (case["alpha"] / 100.0) * (1.0e7 / N)
    l = min(_side(case), 0.5 * L)
    # coordinates near L lie 0.03 to 0.06 apart: rounding widens short extents
    r = (l + 0.015) / (L - l)
    return case["m"] * case["n"] * (2 * r - r * r) ** d


def work(case):
    """Every coordinate the call takes read once, every pair (8 bytes, or 4
    of compressed output) and offset written once."""
    d = case["d"]
    if case["kind"] == "batch":
        ms, ns = _batch_sizes(case)
        return {"bytes": 8.0 * d * (sum(ms) + sum(ns)) + 8.0 * _expected_pairs(case)
                + 24.0 * (len(ms) + 1), "flops": 0.0}
    k, m, n = _expected_pairs(case), case["m"], case["n"]
    if case["kind"] == "stream":
        return {"bytes": 8.0 * d * (m + n) + 4.0 * k + 12.0 * m, "flops": 0.0}
    if case["kind"] == "serve":  # the regions are resident: only their hits have to be looked at
        return {"bytes": 8.0 * d * m + 8.0 * d * min(n, k) + 8.0 * k, "flops": 0.0}
    if case["kind"] == "moved":  # moved extents in, their own tree's coordinates and their rows out
        v = case["moved"]
        return {"bytes": 8.0 * d * (2 * v + 2 * m) + 8.0 * k * v / m, "flops": 0.0}
    return {"bytes": 8.0 * d * (m + n) + 8.0 * k, "flops": 0.0}
