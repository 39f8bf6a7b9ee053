"""The setup under inputs at the edge of what it takes.

A singular line: its inverse is formed beside the load flow and names it in the
setup's error flag while the load flow runs.  The call returns the singular line
at once (no CTA of the load flow waits for one that left), whatever the size, and
leaves the context as it was.
"""
import time

import numpy as np
import pytest

import feedergen as fg

pytestmark = pytest.mark.gpu

STALL_S = 0.25          # a load flow that waits out its barriers' polls takes longer; a call takes a few ms


@pytest.fixture(scope="module")
def ctx():
    import paper_2510_19608_gb300 as K
    with K.Context(0) as c:
        yield c


@pytest.mark.parametrize("n,scen", [(40, 1), (256, 4), (300, 1), (300, 4), (1000, 2), (2200, 2)])
def test_a_singular_line_beside_the_load_flow_is_reported_at_once(ctx, n, scen):
    import paper_2510_19608_gb300 as K
    from paper_2510_19608_gb300._binding import ESINGULAR
    f = fg.make_feeder(n, 11, phase_mode=(0.5, 0.2, 0.3), n_scen=scen)
    want = ctx.power_flow(f)
    bad = fg.make_feeder(n, 11, phase_mode=(0.5, 0.2, 0.3), n_scen=scen)
    bad.z_line[1:] = 0.0                    # every line: the flag is set by many CTAs, early and late
    one = fg.make_feeder(n, 11, phase_mode=(0.5, 0.2, 0.3), n_scen=scen)
    one.z_line[n // 2] = 0.0
    few = K.default_params(max_merges=2)
    grid = K.default_params(max_merges=2, max_spins=1_000_000)      # the cooperative load flow at every size
    for g in (bad, one):
        for call in (lambda: ctx.power_flow(g), lambda: ctx.reduce(g, few), lambda: ctx.reduce(g, grid),
                     lambda: ctx.evaluate(g, np.arange(n, dtype=np.int32))):
            for rep in range(6):
                t0 = time.perf_counter()
                with pytest.raises(K.OkrError) as e:
                    call()
                dt = time.perf_counter() - t0
                assert e.value.status == ESINGULAR
                assert rep == 0 or dt < STALL_S, dt
    v, i, sweeps = ctx.power_flow(f)
    assert np.array_equal(v, want[0]) and np.array_equal(i, want[1]) and sweeps == want[2]
