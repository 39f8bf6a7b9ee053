"""The launch shape that a caller asks for is the one that runs, in a cluster too:
every eval_warps that okr_set_inc_shape takes with the default thread count (1 ..
11) is in force, alone and in batches, and gives the default shape's run."""
import numpy as np
import pytest

import feedergen as fg

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def ctx():
    import paper_2510_19608_gb300 as K
    with K.Context(0) as c:
        yield c


@pytest.mark.parametrize("precision", [0, 1])
@pytest.mark.parametrize("n", [20, 40, 400])
def test_eval_warps_are_kept(ctx, n, precision):
    import paper_2510_19608_gb300 as K
    f = fg.make_feeder(n, 8000 + n, phase_mode=(0.45, 0.15, 0.4), n_scen=2)
    p = K.default_params(margin=0.005, max_merges=25, precision=precision)
    ctx.reduce(f, p)
    want, sup = ctx.decisions(), ctx.assignment()
    try:
        for threads, top in ((0, 11), (256, 7), (384, 11), (512, 15)):
            for w in (1, 7, 8, 11, 15):
                if w > top:
                    continue
                ctx.set_inc_shape(threads=threads, eval_warps=w)
                ctx.reduce(f, p)
                s = ctx.summary()
                assert s["inc_eval_warps"] == w and s["inc_threads"] in ((threads,) if threads else (256, 384))
                assert all(np.array_equal(want[k], v) for k, v in ctx.decisions().items())
                assert np.array_equal(sup, ctx.assignment())
    finally:
        ctx.reset_inc_shape()


@pytest.mark.parametrize("precision", [0, 1])
@pytest.mark.parametrize("eval_warps", [7, 8, 11])
def test_a_batch_under_many_eval_warps_gives_the_same_runs(ctx, eval_warps, precision):
    import paper_2510_19608_gb300 as K
    fs = [fg.make_feeder(n, 8100 + n, phase_mode=(0.45, 0.15, 0.4), n_scen=2) for n in (700, 520, 90)]
    p = K.default_params(margin=0.005, max_merges=20, precision=precision)
    want = ctx.reduce_batch(fs, p)[:2]
    try:
        ctx.set_inc_shape(eval_warps=eval_warps)
        got = ctx.reduce_batch(fs, p)[:2]
    finally:
        ctx.reset_inc_shape()
    assert want[0] == got[0] and all(np.array_equal(a, b) for a, b in zip(want[1], got[1]))
