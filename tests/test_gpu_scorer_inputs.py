"""Scorer inference on what a caller may hand over: features in host memory at
any address give the same predictions, whether the kernels read them in place or
from a copy; and an array that ends before the last sample's features is refused
before the GPU reads it."""
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
    return rng.normal(0, 0.12, M.n_params(F)).astype(np.float32), rng.normal(0, 1, (N, F)).astype(np.float32)


def _at(x, shift):
    """x as a contiguous array whose data lies `shift` bytes past a 64-byte boundary."""
    raw = np.zeros(x.nbytes + 128, np.uint8)
    o = -raw.ctypes.data % 64 + shift
    a = raw[o:o + x.nbytes].view(np.float32).reshape(x.shape)
    a[...] = x
    assert a.flags.c_contiguous and a.ctypes.data % 64 == shift
    return a


@pytest.mark.parametrize("F,N", [(14, 1), (14, 333), (1, 20000), (14, 20000), (16, 4096)])
def test_features_at_any_address_give_the_same_predictions(ctx, F, N):
    theta, x = _problem(F, N, 3)
    ctx.scorer_init(F, theta)
    y, ytc = ctx.scorer_predict(_at(x, 0)), ctx.scorer_predict_tc(_at(x, 0))
    for shift in (4, 8, 1, 2, 7, 33):
        a = _at(x, shift)
        assert np.array_equal(ctx.scorer_predict(a), y), shift
        assert np.array_equal(ctx.scorer_predict_tc(a), ytc), shift


def test_too_few_features_are_refused(ctx):
    theta, x = _problem(14, 64, 5)
    ctx.scorer_init(14, theta)
    y = ctx.scorer_predict(x)
    for bad in (x[:, :13], x.reshape(-1), x[:, :0]):
        for f in (ctx.scorer_predict, ctx.scorer_predict_tc):
            with pytest.raises(ValueError):
                f(bad)
    assert np.array_equal(ctx.scorer_predict(x), y)
