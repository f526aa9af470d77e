"""What the memory budget bounds besides the tables of the joins: the candidate tables of launches of several
steps. Plans that need more answer step by step, with the same results."""
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


def test_candidate_tables_within_the_budget(B):
    # paths of four vertices on 20 000 vertices of degree 3: 12 candidates a key, 1.9 MB of ids and as much
    # of checksum terms
    g, p = I.random_regular3(20000, 3), I.path(10)  # three steps: one launch behind the tables, or three and more
    ref = oracle.enumerate(g, p, threads=8, rows=False)
    with B.Context(0) as c:
        plan = c.plan(c.load(g), p)
        launches = {}
        for budget in (0, 64 << 20, 16 << 20, 64 << 20):  # the last after tables were given back
            B.dm_set_budget(c.h, budget)
            assert plan.count() == (ref.count, ref.checksum)
            launches.setdefault(budget, c.stats()["kernel_launches"])
            assert c.stats()["kernel_launches"] == launches[budget]
        assert launches[0] == launches[64 << 20] == 2 < launches[16 << 20]


@pytest.mark.parametrize("budget", [1, 600, 1500, 6000, 20000, 65535, 65536, 70000])
def test_budgets_below_a_table(B, budget):
    # wide rows and tables between launches (the long paths), where not even one of them fits
    for g, lengths in ((I.cycle(12), (5, 12)), (I.cycle(70), (31, 60)), (I.heavy_hex(2, 2), (6, 9))):
        g = I.lognormal_weights(g, 4)
        with B.Context(0, budget) as c:
            gid = c.load(g)
            for n in lengths:
                plan, ref = c.plan(gid, I.path(n)), oracle.enumerate(g, I.path(n))
                assert plan.count() == (ref.count, ref.checksum)
                rows, _, cnt, cs = plan.all()
                assert (cnt, cs) == (ref.count, ref.checksum) == (len(rows), ref.checksum)
                assert sorted(map(tuple, rows)) == sorted(map(tuple, ref.rows))
