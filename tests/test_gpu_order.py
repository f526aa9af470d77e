"""Canonical order of rows behind the joins (order.cu) where the buckets of the keys are nearly as wide as
the 32 bits in which a bucket's rows are ranked: the upper buckets' edges, and the widest that is ranked so."""
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


# a 4 x 4 patch of a grid of V vertices: keys below V * 4^15 in 16 384 buckets, V * 2^16 a bucket
@pytest.mark.parametrize("side", [180, 181, 182, 255])
def test_wide_buckets(B, side):
    g, p = I.lognormal_weights(I.grid(side, side), 2), I.grid(4, 4)
    ref = oracle.enumerate(g, p, threads=8)
    with B.Context(0) as c:
        plan = c.plan(c.load(g), p)
        rows, scores, cnt, cs = plan.all()
        launches = c.stats()["kernel_launches"]
        assert (cnt, cs) == (ref.count, ref.checksum) and np.array_equal(rows, ref.rows)
        # 24 FP32 additions of non-negative terms: relative error below 25 * 2^-24 < 1.5e-6
        np.testing.assert_allclose(scores, oracle.scores(g, p, ref.rows), rtol=1.5e-6, atol=0)
        plan.count()
        assert launches <= c.stats()["kernel_launches"] + 6  # ordered behind the joins, not sorted afterwards
