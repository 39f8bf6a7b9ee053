"""The setup's paths at the sizes where they change.

Load flow: one CTA per scenario up to 256 buses, the cooperative grid with its
slices in shared memory up to 2,048, in device memory above; a batch's load
flow in shared memory up to 1,920.  Evaluation: shared memory up to 1,920.  Line
inverses: eight lanes per line, four lines per warp, on every phase mask.  Each
against the FP64 oracle with the tolerances of the parity tests (1e-10 on
voltages, 1e-9 of the largest injection); a batch of one gives a single run's bits.
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


@pytest.mark.parametrize("n,scen", [(2, 1), (5, 4), (255, 2), (256, 3), (257, 2), (1920, 1), (1921, 2), (2048, 2), (2049, 1)])
def test_load_flow_injections_and_batch_at_the_edges(ctx, n, scen):
    import paper_2510_19608_gb300 as K
    f = fg.make_feeder(n, 300 + n, phase_mode=(0.5, 0.2, 0.3), n_scen=scen)
    vhat, ihat = O.operating_points(f)
    v, i, sweeps = ctx.power_flow(f)
    assert 0 < sweeps < 200
    assert np.abs(v - vhat).max() <= 1e-10
    assert np.abs(i - ihat).max() <= 1e-9 * max(1.0, np.abs(ihat).max())
    # the identity assignment: no error, the full voltages
    err, w = ctx.evaluate(f, np.arange(n, dtype=np.int32))
    assert err.max() <= 1e-10 and np.abs(w - vhat).max() <= 1e-10
    p = K.default_params(margin=0.005, max_merges=3)
    ctx.reduce(f, p)
    one, v1 = ctx.summary(), ctx.assignment()
    items, parts, _ = ctx.reduce_batch([f], [p])
    assert items[0]["status"] == 0 and items[0]["smice"] == one["smice"] and items[0]["max_error"] == one["max_error"]
    assert np.array_equal(parts[0], v1)


@pytest.mark.parametrize("bus", [1, 3, 4, 37])
def test_a_singular_line_is_named_whatever_the_load_flow_makes_of_it(ctx, bus):
    import paper_2510_19608_gb300 as K
    from paper_2510_19608_gb300._binding import ESINGULAR
    for n in (40, 300):
        f = fg.make_feeder(n, 11, phase_mode=(0.5, 0.2, 0.3))
        f.z_line[bus] = 0.0
        for call in (lambda: ctx.power_flow(f), lambda: ctx.reduce(f, K.default_params()),
                     lambda: ctx.evaluate(f, np.arange(n, dtype=np.int32))):
            with pytest.raises(K.OkrError) as e:
                call()
            assert e.value.status == ESINGULAR
        with pytest.raises(K.OkrError):            # no network is left behind
            ctx.radialize(np.ones(n, np.uint8))
        items, _, _ = ctx.reduce_batch([f], [K.default_params()])
        assert items[0]["status"] == ESINGULAR
