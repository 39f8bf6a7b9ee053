"""A feeder searched by a cluster of CTAs gives the run that one CTA gives.

The slot pairs are dealt out to the cluster's CTAs (pair w to CTA w mod 8), so
the sizes are around multiples of 8, with fewer pairs than threads and with
more, and around the sizes from which a cluster is taken.  The sums are exact
integers and the selection exact, so every decision, score, largest error, gap
and candidate count is equal bit for bit, and verify mode finds every carried
score equal to a fresh evaluation.
"""
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
@pytest.mark.parametrize("n,scen,target", [(9, 2, 1.0), (31, 1, 1.0), (32, 2, 1.0), (41, 1, 1.0), (199, 2, 0.9), (200, 3, 0.9), (257, 4, 0.8),
                                           (1025, 1, 0.3), (1499, 2, 0.1), (1500, 2, 0.2), (2100, 4, 0.04)])
def test_cluster_and_one_cta_give_the_same_run(ctx, n, scen, target, precision):
    import paper_2510_19608_gb300 as K
    f = fg.make_feeder(n, 7000 + n, phase_mode=(0.45, 0.15, 0.4), load=("lognormal", 15.0, 1.0), n_scen=scen)
    runs = []
    for records, engine in ((0, 2), (2, 2), (0, 3)):        # records=2: one CTA, its records in shared memory
        try:
            ctx.set_inc_shape(records=records)
            ctx.reduce(f, K.default_params(margin=0.005, target_reduction=target, precision=precision, engine=engine))
        finally:
            ctx.reset_inc_shape()
        s = ctx.summary()
        assert s["inc_mismatches"] == 0
        runs.append((ctx.decisions(), ctx.assignment(), ctx.voltages()[1],
                     [s[k] for k in ("n_iter", "stop_reason", "candidates", "rechecks", "recheck_cands", "smice")]))
    for dec, sup, vred, counts in runs[1:]:
        for k, v in runs[0][0].items():
            assert np.array_equal(v, dec[k]), k
        assert np.array_equal(runs[0][1], sup) and np.array_equal(runs[0][2], vred) and runs[0][3] == counts


@pytest.mark.parametrize("precision", [0, 1])
@pytest.mark.parametrize("sizes", [(700, 520, 90), (640, 499, 500, 501, 30, 9) + (40,) * 40,
                                   (700, 260) + (60,) * 150])
def test_batches_searched_by_clusters_and_single_ctas_give_the_single_runs(ctx, sizes, precision):
    """Clusters of eight where SMs are left, of two for a long chain among many
    (152 feeders on 152 SMs); the other feeders by one CTA each, beside them: every feeder's result is its single run's, bit for bit."""
    import paper_2510_19608_gb300 as K
    feeders = [fg.make_feeder(n, 40 + 7 * i, phase_mode=(0.7, 0.1, 0.2)) for i, n in enumerate(sizes)]
    p = K.default_params(margin=0.005, target_reduction=0.3, precision=precision)
    items, parts, _ = ctx.reduce_batch(feeders, p)
    plan = ctx.batch_plan(feeders, p)
    again, parts2, _ = plan.run()
    plan.close()
    assert again == items and all(np.array_equal(a, b) for a, b in zip(parts, parts2))
    for i in sorted(set([0, 1, 2, 3, 4, 5, len(sizes) - 1]) & set(range(len(sizes)))):
        ctx.reduce(feeders[i], p)
        s = ctx.summary()
        assert items[i]["status"] == 0
        assert [items[i][k] for k in ("n_iter", "stop_reason", "n_kept", "candidates", "smice", "max_error")] == \
            [s[k] for k in ("n_iter", "stop_reason", "n_kept", "candidates", "smice", "max_error")]
        assert np.array_equal(parts[i], ctx.assignment())
