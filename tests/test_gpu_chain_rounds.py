"""Plans of one to five launches whose first launch leaves part of the first table to further rounds
(dm_set_launch_limit): tables between launches start anew in each round, and rows that are there stay.
Exact against the oracle, with the arena growing and with the arena at its budget."""
import numpy as np
import pytest

import oracle
from paper_2508_21287_gb300 import inputs as I

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def B():
    from paper_2508_21287_gb300 import build
    build.build()
    from paper_2508_21287_gb300 import binding
    return binding


@pytest.fixture(scope="module")
def comb():
    """A path of 16 000 vertices with three leaves each: first tables far larger than the warps of a launch
    take in at once, and 32 embeddings of a long path for each of its edges."""
    n = 16000
    g = I.from_edges(4 * n, [(i, i + 1) for i in range(n - 1)] + [(i, n + 3 * i + j) for i in range(n) for j in range(3)])
    return I.lognormal_weights(g, 3)


@pytest.mark.parametrize("length", [8, 16, 20, 30, 40, 50])
@pytest.mark.parametrize("limit", [1, 300])
def test_counts(B, comb, length, limit):
    p = I.path(length)
    ref = oracle.enumerate(comb, p, threads=8, rows=False)
    with B.Context(0) as c:
        plan = c.plan(c.load(comb, False), p)
        assert plan.count() == (ref.count, ref.checksum)
        whole = c.stats()
        B.dm_set_launch_limit(c.h, limit)
        assert plan.count() == (ref.count, ref.checksum)
        parts = c.stats()
        assert parts["kernel_launches"] >= 2 * whole["kernel_launches"] - 1  # the candidate tables are made once
        assert parts["rows"] == whole["rows"] and parts["candidates"] == whole["candidates"]
        with pytest.raises(RuntimeError):
            B.dm_set_launch_limit(c.h, -1)


@pytest.mark.parametrize("budget", [0, 800 << 20])
@pytest.mark.parametrize("length", [8, 16, 20, 24, 30])
def test_rows_and_best_rows(B, comb, length, budget):
    p = I.path(length)
    ref = oracle.enumerate(comb, p, threads=8)
    with B.Context(0, budget) as c:
        plan = c.plan(c.load(comb), p)
        first = plan.all()
        assert c.stats()["chunks"] == c.stats()["n_steps"]
        best = plan.topk(50)
        B.dm_set_launch_limit(c.h, 1)
        rows, scores, cnt, cs = plan.all()
        assert c.stats()["chunks"] > c.stats()["n_steps"]  # some steps ran in more than one round
        assert (cnt, cs) == (ref.count, ref.checksum) and np.array_equal(rows, ref.rows)
        assert np.array_equal(first[0], ref.rows) and np.array_equal(first[1], scores)
        for _ in range(2):
            again = plan.topk(50)
            assert np.array_equal(again[0], best[0]) and np.array_equal(again[1], best[1])
        order = np.lexsort((np.arange(len(scores)), scores))[:50]
        assert np.array_equal(best[0], rows[order]) and np.array_equal(best[1], scores[order])


def test_arena_that_overflows_in_a_later_round(B):
    """61 M rows of 44 bytes in three rounds: two fit the first arena (rows in its half, 2 GB), the third does
    not, and the joins begin again in a larger one."""
    g, p = I.random_regular3(40000, 3), I.path(11)
    ref = oracle.enumerate(g, p, threads=8, rows=False)
    with B.Context(0) as c:
        plan = c.plan(c.load(g), p)
        B.dm_set_launch_limit(c.h, 1)
        got = []
        count, checksum = B.dm_match(c.h, plan.h, B.DM_ALL | B.DM_DEVICE_ROWS, lambda r, s, m, n: got.append((m, n)) or 0)
        assert (count, checksum) == (ref.count, ref.checksum) and sum(m for m, _ in got) == ref.count
        # the arena has grown: one attempt, three rounds
        plan2 = c.plan(c.load(g), I.path(10))
        B.dm_match(c.h, plan2.h, B.DM_ALL | B.DM_DEVICE_ROWS, lambda r, s, m, n: 0)
        assert c.stats()["rows"][-1] == oracle.enumerate(g, I.path(10), threads=8, rows=False).count
