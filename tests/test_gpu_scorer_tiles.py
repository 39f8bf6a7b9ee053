"""The scorer's kernels at the edges of their tiles.

Every sum runs in a fixed order whatever the tiling, so a sample's prediction
does not depend on how many others are predicted with it: tiles of 32 samples
(few samples) and of 128 (from 128 times the SM count on, 19,456 on 152 SMs)
give equal bits.  The gradient is compared with the FP64 oracle at the sizes
around a pipeline stage (64) and a segment (2,048), with the tolerance of the
scorer's other gradient test.
"""
import numpy as np
import pytest

from oracle import mlp as M

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def ctx():
    import paper_2510_19608_gb300 as K
    with K.Context(0) as c:
        yield c


def _problem(F, N, seed):
    rng = np.random.default_rng(seed)
    theta = rng.normal(0, 0.12, M.n_params(F)).astype(np.float32)
    return theta, rng.normal(0, 1, (N, F)).astype(np.float32), rng.normal(0, 1, N).astype(np.float32)


@pytest.mark.parametrize("F", [1, 14, 16])
def test_a_prediction_does_not_depend_on_the_tile(ctx, F):
    theta, x, _ = _problem(F, 40001, 5)
    ctx.scorer_init(F, theta)
    y = ctx.scorer_predict(x)
    for lo, hi in ((0, 1), (0, 31), (100, 133), (0, 4865), (7, 19456), (0, 19456), (0, 19457), (1, 40001)):
        assert np.array_equal(ctx.scorer_predict(x[lo:hi]), y[lo:hi]), (lo, hi)


@pytest.mark.parametrize("F,N", [(14, 31), (14, 63), (14, 64), (14, 65), (16, 2047), (3, 2048), (14, 2049), (1, 5000)])
def test_gradient_at_the_edges_of_stages_and_segments(ctx, F, N):
    theta, x, t = _problem(F, N, N)
    ctx.scorer_init(F, theta)
    g, loss = ctx.scorer_gradient(x, t)
    parts = [p.copy() for p in M.unpack(theta, F)]
    for i in (0, 2, 4, 6):
        parts[i] = M.bf16_round(parts[i])
    th = np.concatenate([p.ravel() for p in parts]).astype(np.float64)
    ref = M.grad(th, x.astype(np.float64), t.astype(np.float64))
    assert abs(loss - M.loss(th, x.astype(np.float64), t.astype(np.float64))) <= 1e-4 * max(1.0, loss)
    assert np.abs(g - ref).max() <= 2e-4 * max(1e-3, np.abs(ref).max())


def test_training_repeats_after_another_network_used_the_context(ctx):
    """The scorer's buffers are kept when it is made anew: the same training
    gives the same bits after a network with other features and more samples."""
    theta, x, t = _problem(14, 5000, 9)

    def once():
        ctx.scorer_init(14, theta)
        loss = ctx.scorer_train(x, t, batch=1500, epochs=2, lr=1e-3)
        return loss, ctx.scorer_params()

    l0, p0 = once()
    th2, x2, t2 = _problem(16, 9000, 10)
    ctx.scorer_init(16, th2)
    ctx.scorer_train(x2, t2, batch=9000, epochs=1, lr=1e-3)
    l1, p1 = once()
    assert np.array_equal(l0, l1) and np.array_equal(p0, p1)
