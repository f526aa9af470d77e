"""Results of more rows than a table that is put in order may have (dm_set_table_limit; 2^31 - 1 unless a test sets
less): delivered in chunks, each in canonical order, with the same rows, count, checksum and best rows."""
import numpy as np
import pytest

import oracle
from paper_2508_21287_gb300 import inputs as I

pytestmark = pytest.mark.gpu
CAPACITY = -4


@pytest.fixture(scope="module")
def B():
    from paper_2508_21287_gb300 import build
    build.build()
    from paper_2508_21287_gb300 import binding
    return binding


# joins of one launch, of several (the 30-vertex path), a launch a step (induced), and sorted ones
@pytest.mark.parametrize("name,n,kw", [("hh", 8, {}), ("hh", 30, {}), ("grid", 6, {}), ("hh", 8, {"induced": 1}),
                                       ("grid", 5, {"join_algo": 2})])
@pytest.mark.parametrize("weights", [False, True])
def test_rows_in_chunks(B, name, n, kw, weights):
    g = I.lognormal_weights(I.heavy_hex(3, 4) if name == "hh" else I.grid(9, 9), 3)
    p = I.path(n)
    ref = oracle.enumerate(g, p, induced=bool(kw.get("induced")))
    with B.Context(0, 64 << 20) as c:
        plan = c.plan(c.load(g, weights=weights), p, **kw)
        for limit in (ref.count + 1, ref.count, ref.count - 1, ref.count // 3, 300):
            B.dm_set_table_limit(c.h, limit)
            got = []

            def take(rows, scores):
                assert [list(r) for r in rows] == sorted(list(r) for r in rows)
                assert (scores is not None) == weights
                got.append(rows.copy())

            cnt, cs = B.dm_match(c.h, plan.h, B.DM_ALL, take)
            assert (cnt, cs) == (ref.count, ref.checksum) == plan.count()
            assert (len(got) == 1) == (limit >= ref.count) and max(map(len, got)) <= limit
            rows = np.concatenate(got)
            assert np.array_equal(rows[np.lexsort(rows.T[::-1])], ref.rows)
            if weights:
                order = oracle.topk(ref.rows, oracle.scores(g, p, ref.rows), 20)
                want = oracle.scores(g, p, ref.rows)[order]
                # sums of at most 29 non-negative terms, each rounded once: within 29 * 2^-24 of the exact ones
                np.testing.assert_allclose(plan.topk(20)[1], want, rtol=2e-6)
                np.testing.assert_allclose(B.dm_match_topk(c.h, plan.h, B.DM_ALL, None, 20, n)[1], want, rtol=2e-6)


def test_one_table(B):
    g, p = I.grid(9, 9), I.path(4)
    want = len({tuple(sorted(r)) for r in oracle.enumerate(g, p).rows.tolist()})
    with B.Context(0, 64 << 20) as c:
        plan = c.plan(c.load(g), p)
        B.dm_set_table_limit(c.h, 100)
        with pytest.raises(B.DMError) as e:
            B.dm_images(c.h, plan.h, 4)
        assert e.value.code == CAPACITY
        with pytest.raises(B.DMError):
            B.dm_set_table_limit(c.h, -1)
        B.dm_set_table_limit(c.h, 0)
        assert len(B.dm_images(c.h, plan.h, 4)) == want
