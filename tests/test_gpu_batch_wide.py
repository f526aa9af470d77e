"""Plans that meet two large motif tables, in batches of warp walks (k_batch_wide): graphs on both sides
of a bitmap's width, one and two join keys, first tables that end inside a tile, no survivors and many,
and a scratch budget that leaves no room for the bitmaps. Exact against the same plans one at a time,
which the step-by-step joins answer, and against the oracle on the smallest graph."""
import numpy as np
import pytest

import oracle
from paper_2508_21287_gb300 import inputs as I

pytestmark = pytest.mark.gpu

PATTERNS = [I.path(9), I.path(12), I.path(13), I.cycle(10), I.cycle(12), I.cycle(13), I.cycle(16),
            I.cycle_with_chords(14, 3, 1)]


@pytest.fixture(scope="module")
def B():
    from paper_2508_21287_gb300 import build
    build.build()
    from paper_2508_21287_gb300 import binding
    return binding


def wide(B, plan):
    d = B.dm_plan_describe(plan)
    return (len(d) == 2 and len(d[1]["slice"]) - d[1]["n_keys"] > 4 and not d[0]["backedges"]
            and not d[1]["backedges"])


@pytest.mark.parametrize("graph", ["ring40", "rr254", "rr256", "rr258", "rr512", "rr514", "rr768", "rr1024", "rr1026",
                                   "hex12x6", "small_budget"])
def test_wide_plans_match_single_runs(B, graph):
    if graph == "ring40":
        g = I.cycle(40)
    elif graph.startswith("rr"):
        g = I.random_regular3(int(graph[2:]), 7)
    else:
        g = I.heavy_hex(12, 6)
    with B.Context(0, (4 << 20) if graph == "small_budget" else 0) as ctx:
        gid = ctx.load(g, False)
        plans, pats = [], []
        for p in PATTERNS:
            for plan in B.dm_plan_candidates(ctx.h, gid, p.n, p.row_ptr, p.col_idx):
                plans.append(plan)
                pats.append(p)
        assert any(wide(B, plan) for plan in plans)
        single = [B.dm_match(ctx.h, plan, B.DM_COUNT) for plan in plans]
        B.dm_set_tuning(ctx.h, autotune=False)
        B.dm_set_batch_shape(ctx.h, 32)
        only = [i for i, plan in enumerate(plans) if wide(B, plan)]
        for sel in (list(range(len(plans))), only, only[:1]):
            for _ in range(2):  # built, then replayed
                counts, sums = B.dm_match_batch(ctx.h, [plans[i] for i in sel])
                assert counts.tolist() == [int(single[i][0]) for i in sel]
                assert sums.tolist() == [int(single[i][1]) for i in sel]
            assert np.all((B.dm_batch_latency(ctx.h, len(sel)) > 0) | (counts == 0))  # no first rows: no items
        if graph == "ring40":
            for i in only:
                ref = oracle.enumerate(g, pats[i], rows=False)
                assert (int(single[i][0]), int(single[i][1])) == (ref.count, ref.checksum)
        for plan in plans:
            B.dm_plan_free(plan)
