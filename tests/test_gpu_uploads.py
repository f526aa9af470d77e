"""Arrays that a call uploads and its kernels read at once, on a stream of the caller's own as well: graphs whose
arrays are below and above 64 KB (a copy outside the stream returns before the smaller ones have arrived), loaded
one after the other so that the memory of each held another's arrays; and the weights of the model."""
import numpy as np
import pytest
import torch

import oracle
from paper_2508_21287_gb300 import inputs as I

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def B():
    from paper_2508_21287_gb300 import build
    build.build()
    from paper_2508_21287_gb300 import binding
    return binding


@pytest.mark.parametrize("own", [False, True])
def test_graphs_one_after_the_other(B, own):
    graphs = [I.lognormal_weights(g, 7, qubits=True)
              for g in (I.heavy_hex(2, 3), I.random_regular3(8192, 2), I.grid(6, 5), I.heavy_hex(27, 28), I.cycle(40))]
    p = I.path(6)
    refs = [oracle.enumerate(g, p) for g in graphs]
    best = [np.sort(oracle.scores(g, p, r.rows))[:5] for g, r in zip(graphs, refs)]
    stream = torch.cuda.Stream() if own else None
    for _ in range(6):
        with B.Context(0) as c:
            if own:
                B.dm_set_stream(c.h, stream.cuda_stream)
            for g, r, b in zip(graphs, refs, best):
                plan = c.plan(c.load(g), p)
                assert plan.count() == (r.count, r.checksum)
                # sums of 11 non-negative terms, each rounded once: within 11 * 2^-24 of the exact ones
                np.testing.assert_allclose(plan.topk(5)[1], b, rtol=1e-6)


def test_weights_of_the_model(B):
    rng = np.random.default_rng(1)
    X = rng.normal(size=(48, 32)).astype(np.float32)
    with B.Context(0) as c:
        B.dm_model_init(c.h, 3)
        w = B.dm_model_weights(c.h)
        y = B.dm_model_predict(c.h, X)
    for k in range(6):
        with B.Context(0) as c:  # allocated, set and used with nothing in between
            B.dm_model_set_weights(c.h, w)
            assert np.array_equal(B.dm_model_predict(c.h, X), y)
            other = (w * np.float32(k)).astype(np.float32)
            B.dm_model_set_weights(c.h, other)
            assert np.array_equal(B.dm_model_weights(c.h)[:-64], other[:-64])
