"""Objective 1 (the candidate network's largest error) at super-node counts around
the blocks of 32 ranks whose largest MICE are kept: every iteration's decision,
score and largest error against the oracle, both precisions.
"""
import numpy as np
import pytest

import feedergen as fg
from oracle import oracle as O

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def ctx():
    import paper_2510_19608_gb300 as K
    with K.Context(0) as c:
        yield c


@pytest.mark.parametrize("precision", [0, 1])
@pytest.mark.parametrize("n", [5, 31, 32, 33, 64, 65, 97, 130])
def test_largest_error_objective_at_the_block_edges(ctx, n, precision):
    import paper_2510_19608_gb300 as K
    f = fg.make_feeder(n, 900 + n, phase_mode=(0.6, 0.2, 0.2))
    vhat, ihat = O.operating_points(f)
    merges = min(n - 1, 40)
    res = O.reduce(f, vhat, ihat, margin=0.005, max_merges=merges, objective=1)
    ctx.reduce(f, K.default_params(margin=0.005, max_merges=merges, objective=1, precision=precision))
    d = ctx.decisions()
    assert len(d["s"]) == res["n_iter"] and ctx.summary()["candidates"] == res["candidates"]
    assert np.array_equal(d["s"], res["s"]) and np.array_equal(d["r"], res["r"])
    assert np.abs(d["score"] - res["score"]).max(initial=0.0) <= 1e-9
    assert np.abs(d["maxerr"] - res["maxerr"]).max(initial=0.0) <= 1e-9
