"""Plans that run several steps a launch (chain.cu) against the oracle: graphs that decide which pairs
of vertices are compared (girth, odd cycles), groups of every size the records take, tiles that fill
and drain at every remainder, and the edge of 16-bit ids. Counts, checksums and rows are exact."""
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
def ctx(B):
    c = B.Context(0)
    yield c
    c.close()


def strip(n):
    """Triangles in a row: odd cycles, girth 3."""
    return I.from_edges(n, [(i, i + 1) for i in range(n - 1)] + [(i, i + 2) for i in range(n - 2)])


def bipartite(a, b):
    return I.from_edges(a + b, [(i, a + j) for i in range(a) for j in range(b)])


def torus(a, b):
    return I.from_edges(a * b, sorted({tuple(sorted((r * b + c, q))) for r in range(a) for c in range(b)
                                       for q in (((r + 1) % a) * b + c, r * b + (c + 1) % b)}))


def caterpillar(n):
    """A path with 0, 1 or 2 leaves a vertex: groups of uneven size, no cycle."""
    e, k = [(i, i + 1) for i in range(n - 1)], n
    for i in range(n):
        for _ in range(i % 3):
            e.append((i, k))
            k += 1
    return I.from_edges(k, e)


GRAPHS = {
    "strip": (strip(37), [4, 7, 9]),
    "k7": (I.complete(7), [3, 5, 7]),
    "k33": (bipartite(3, 3), [4, 6]),
    "k45": (bipartite(4, 5), [5, 7]),
    "torus5x7": (torus(5, 7), [6, 9]),
    "torus6x6": (torus(6, 6), [6, 9]),
    "ring13": (I.cycle(13), [5, 12, 13]),
    "ring12": (I.cycle(12), [5, 11, 12]),
    "caterpillar": (caterpillar(23), [6, 11]),
    "heavyhex": (I.heavy_hex(2, 3), [13, 18]),
    "rr3": (I.random_regular3(64, 3), [7, 10]),
}


@pytest.mark.parametrize("name", sorted(GRAPHS))
def test_every_form_equals_the_oracle(ctx, B, name):
    g, lens = GRAPHS[name]
    g = I.lognormal_weights(g, 5, qubits=True)
    gid = ctx.load(g)
    pats = [I.path(k) for k in lens] + [I.star(3), I.cycle(4), I.cycle(6), I.random_tree(8, 2), I.random_tree(9, 7)]
    for p in pats:
        if p.n > g.n:
            continue
        ref = oracle.enumerate(g, p, threads=8)
        want = oracle.scores(g, p, ref.rows)
        for motifs in (None, [2], [4, 2], [104, 2]):
            plan = ctx.plan(gid, p, motifs=motifs)
            assert plan.count() == (ref.count, ref.checksum), (name, p.name, motifs)
            shards = [B.dm_match_shard(ctx.h, plan.h, i, 3) for i in range(3)]
            assert sum(c for c, _ in shards) == ref.count and sum(s for _, s in shards) % 2 ** 64 == ref.checksum
            rows, scores, cnt, cs = plan.all()
            assert (cnt, cs) == (ref.count, ref.checksum) and np.array_equal(rows, ref.rows), (name, p.name, motifs)
            # at most 16 FP32 additions of non-negative terms: relative error below 17 * 2^-24 ~ 1e-6
            if ref.count:
                np.testing.assert_allclose(scores, want, rtol=2e-6, atol=0)
            # the general form (a launch a step, sorted keys) sees the same rows step by step
            stats = ctx.stats()
            ctx.plan(gid, p, motifs=motifs, join_algo=B.DM_JOIN_SORTMERGE).all()
            other = ctx.stats()
            assert stats["rows"] == other["rows"] and stats["candidates"] == other["candidates"], (name, p.name, motifs)


def scrambled(p, seed):
    """p with its vertices renumbered: columns far from their pattern neighbours."""
    return I.relabel(p, np.random.RandomState(seed).permutation(p.n))


@pytest.mark.parametrize("graph,pattern", [
    ((9, 9), scrambled(I.path(20), 1)),     # too many rows share their leading columns: sorted another way
    ((13, 13), scrambled(I.path(12), 2)),   # keys of several words
    ((13, 13), I.path(13)),                 # one word
    ((10, 10), I.sub_patch(I.heavy_hex(10, 10), 30, 4)),
    ((25, 34), scrambled(I.path(9), 3)),
    ((2, 2), I.path(2)),
])
def test_order_of_rows(ctx, B, graph, pattern):
    g = I.lognormal_weights(I.heavy_hex(*graph), 3)
    plan = ctx.plan(ctx.load(g), pattern)
    rows, scores, count, checksum = plan.all()
    ref = oracle.enumerate(g, pattern, threads=8)
    assert (count, checksum) == (ref.count, ref.checksum) and np.array_equal(rows, ref.rows)
    # at most 29 FP32 additions of non-negative terms: relative error below 30 * 2^-24 < 2e-6
    np.testing.assert_allclose(scores, oracle.scores(g, pattern, ref.rows), rtol=2e-6, atol=0)
    top_rows, top, cnt, cs = B.dm_match_topk(ctx.h, plan.h, B.DM_ALL, None, 50, pattern.n)
    assert (cnt, cs) == (ref.count, ref.checksum)
    order = np.lexsort((np.arange(len(scores)), scores))[:50]
    assert np.array_equal(top_rows, rows[order]) and np.array_equal(top, scores[order])


@pytest.mark.parametrize("weights", ["lognormal", "equal", "two", "negative"])
@pytest.mark.parametrize("k", [1, 10, 1000, 1024, 1025])
def test_best_rows(ctx, weights, k):
    # small and large tables, first tables of fewer rows than warps, scores that thousands of rows
    # share (the selection gives up), few distinct scores, and weights that forbid pruning
    for g, p in ((I.heavy_hex(4, 6), I.path(18)), (I.heavy_hex(2, 2), I.path(6)), (I.random_regular3(512, 3), I.path(9)),
                 (I.grid(9, 7), I.sub_patch(I.grid(9, 7), 8, 2))):
        g = I.lognormal_weights(g, 11)
        if weights == "equal":
            g.edge_err[:] = 0.25
        elif weights == "two":
            g.edge_err[:] = np.where(g.edge_err > np.median(g.edge_err), 0.5, 0.25)
        elif weights == "negative":
            g.edge_err -= 0.006
        gid = ctx.load(g)
        rows, scores = ctx.plan(gid, p).topk(k)
        ref = oracle.enumerate(g, p)
        want = oracle.scores(g, p, ref.rows)
        order = oracle.topk(ref.rows, want, k)
        assert len(rows) == min(k, ref.count)
        # sums of at most 17 terms of at most 0.5: FP32 error below 17 * 2^-24 * 8.5 ~ 9e-6
        np.testing.assert_allclose(scores, want[order], rtol=0, atol=9e-6)
        if weights in ("equal", "two"):  # exact in FP32: the rows are decided
            assert np.array_equal(rows, ref.rows[order])
        # the same again, through the form that keeps every row
        r2, s2 = ctx.plan(gid, p, chunk_rows=4000).topk(k)
        np.testing.assert_allclose(s2, scores, rtol=0, atol=9e-6)


@pytest.mark.parametrize("n", [65533, 65534, 65535])
def test_edge_of_16_bit_ids(ctx, n):
    # a path: 2 (n - k + 1) embeddings of the path of k vertices; ids up to n - 1
    gid = ctx.load(I.path(n))
    for k in (3, 7, 12):
        plan = ctx.plan(gid, I.path(k))
        count, checksum = plan.count()
        rows, _, cnt, cs = plan.all()
        assert count == cnt == 2 * (n - k + 1) and checksum == cs
        first = np.arange(n - k + 1)[:, None] + np.arange(k)
        want = np.concatenate([first, first[:, ::-1]])
        assert np.array_equal(rows, want[np.lexsort(want.T[::-1])])


@pytest.mark.parametrize("m,n,length", [(4, 4, 30), (5, 6, 27), (9, 11, 23), (15, 16, 21), (27, 28, 20)])
def test_tables_between_launches(B, ctx, m, n, length):
    """Deep plans, cut into launches: the table between them in shares of four, of two, and whole blocks,
    and first tables of fewer rows than warps and of several a warp."""
    g, p = I.heavy_hex(m, n), I.path(length)
    gid = ctx.load(g, False)
    plan = ctx.plan(gid, p)
    ref = oracle.enumerate(g, p, threads=8, rows=False)
    for _ in range(2):
        assert plan.count() == (ref.count, ref.checksum)


@pytest.mark.parametrize("budget", [2 << 30, 400 << 20, 40 << 20])
def test_rows_of_several_launches_at_the_budget(B, budget):
    """Rows of a plan cut into launches with the arena at its budget: room for the order behind the joins,
    room for the tables only, and too little for one table (streamed)."""
    g, p = I.lognormal_weights(I.heavy_hex(9, 11), 5), I.path(20)
    ref = oracle.enumerate(g, p, threads=8)
    with B.Context(0, budget) as c:
        plan = c.plan(c.load(g), p)
        for _ in range(2):
            rows, scores, cnt, cs = plan.all()
            assert (cnt, cs) == (ref.count, ref.checksum)
            if budget < 400 << 20:  # chunks are sorted one by one
                rows = rows[np.lexsort(rows.T[::-1])]
            assert np.array_equal(rows, ref.rows)
