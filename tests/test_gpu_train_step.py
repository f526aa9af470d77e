"""One training step (k_train_rows, k_train_weights) against Adam on dm_model_grad's gradients, at the edges
of a block's samples, of a product's chunk and of the padding; and fresh weights against the generator."""
import math

import numpy as np
import pytest

pytestmark = pytest.mark.gpu
M64 = (1 << 64) - 1


@pytest.fixture(scope="module")
def B():
    from paper_2508_21287_gb300 import build
    build.build()
    from paper_2508_21287_gb300 import binding
    return binding


def draw(st):
    z = st
    z = ((z ^ (z >> 30)) * 0xBF58476D1CE4E5B9) & M64
    z = ((z ^ (z >> 27)) * 0x94D049BB133111EB) & M64
    return z ^ (z >> 31)


def shuffled(n, seed):
    idx, st = list(range(n)), seed ^ 0xA5A5A5A5
    for i in range(n - 1, 0, -1):
        st = (st + 0x9E3779B97F4A7C15) & M64
        j = draw(st) % (i + 1)
        idx[i], idx[j] = idx[j], idx[i]
    return idx


@pytest.mark.parametrize("n", [16, 17, 31, 127, 128, 129, 255, 256, 257, 300, 512, 600])
def test_one_step_is_adam_on_the_gradients(B, n):
    rng = np.random.default_rng(n)
    X = rng.normal(size=(n, 32)).astype(np.float32)
    t = rng.normal(size=n).astype(np.float32)
    order = shuffled(n, 3)
    with B.Context(0) as ctx:
        B.dm_model_init(ctx.h, 5)
        w = B.dm_model_weights(ctx.h)
        p = len(w) - 64
        B.dm_model_set_weights(ctx.h, w)  # mean 0, deviation 1: inputs are taken as they are
        _, g, loss = B.dm_model_grad(ctx.h, np.ascontiguousarray(X[order]), t[order])
        B.dm_model_init(ctx.h, 5)
        B.dm_model_set_weights(ctx.h, w)
        got_loss = B.dm_model_train(ctx.h, X, t, epochs=1, batch=max(n, 16), lr=2e-3, seed=3)
        got = B.dm_model_weights(ctx.h)[:p].astype(np.float64)
    g = g.astype(np.float64)
    m, v = 0.1 * g / (1 - 0.9), 0.001 * g * g / (1 - 0.999)
    want = w[:p].astype(np.float64) - 2e-3 * m / (np.sqrt(v) + 1e-8)
    # the gradients are the same bits. A weight of at most 1 is rounded once (2^-25), the update of at most
    # lr is off by the FP32 rounding of the corrections 1 - 0.9 and 1 - 0.999 (6e-5 of the second, half of
    # that after the root) and a few more roundings: 2e-3 * 3.1e-5 = 6.2e-8
    np.testing.assert_allclose(got, want, rtol=0, atol=1.2e-7)
    assert abs(float(got_loss[0]) - float(loss)) <= 1e-5 * float(loss)  # n terms added in another order


def test_fresh_weights(B):
    with B.Context(0) as ctx:
        for seed in (0, 3, M64):
            B.dm_model_init(ctx.h, seed)
            w = B.dm_model_weights(ctx.h)
            st, want = seed, []
            for count, a in ((128 * 32, 6 / 32), (128, 0), (128 * 128, 6 / 128), (128, 0), (128, 3 / 128), (1, 0)):
                for _ in range(count):
                    if a == 0:
                        want.append(0.0)
                        continue
                    st = (st + 0x9E3779B97F4A7C15) & M64
                    u = (float(draw(st) >> 11) + 0.5) * (1.0 / 9007199254740992.0) * 2.0 - 1.0
                    want.append(math.sqrt(a) * u)
            assert np.array_equal(w[:len(want)], np.array(want).astype(np.float32))
