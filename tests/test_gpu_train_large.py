"""Training on more samples than are held on the device, on batches larger than a piece of the staging buffer,
and over more steps than losses are held for: the same weights and losses as in one go."""
import numpy as np
import pytest

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def B():
    from paper_2508_21287_gb300 import build
    build.build()
    from paper_2508_21287_gb300 import binding
    return binding


def samples(n):
    rng = np.random.default_rng(n)
    X = rng.normal(size=(n, 32)).astype(np.float32)
    return X, (X[:, :4].sum(axis=1) + 0.1 * rng.normal(size=n)).astype(np.float32)


def train(B, budget, X, t, epochs, batch):
    with B.Context(0, budget) as ctx:
        B.dm_model_init(ctx.h, 5)
        loss = B.dm_model_train(ctx.h, X, t, epochs=epochs, batch=batch, lr=1e-3, seed=3)
        return B.dm_model_weights(ctx.h), np.asarray(loss)


@pytest.mark.parametrize("n,batch", [(520_000, 65_536), (520_000, 300_001), (600_001, 600_000)])
def test_samples_of_each_step(B, n, batch):
    X, t = samples(n)  # more than 64 MB
    w, loss = train(B, 0, X, t, 2, batch)
    w2, loss2 = train(B, 256 << 20, X, t, 2, batch)
    assert np.array_equal(w, w2)
    # sums of n losses in any order, FP32 within a step: relative error below n * 2^-24, and far below it
    # for terms of like size
    np.testing.assert_allclose(loss2, loss, rtol=1e-3)
    assert np.isfinite(w).all() and loss[1] < loss[0]


def test_more_steps_than_losses_are_held_for(B):
    X, t = samples(40)
    epochs = 5500  # three steps each: 16 500 steps, more than 2^14
    w, loss = train(B, 0, X, t, epochs, 16)
    for e in (1, 2, 5461, 5462):  # epoch 5461 ends in the second part
        we, le = train(B, 0, X, t, e, 16)
        np.testing.assert_allclose(loss[:e], le, rtol=1e-5)  # a step adds 16 terms in any order
    assert np.isfinite(w).all() and (loss > 0).all() and loss[-1] < 0.05 * loss[0]
