"""Where a cluster keeps a large feeder's candidates and sums: in shared memory up to
4,404 buses, in device memory with the records in shared memory up to 9,792; above
that one CTA searches, up to 13,903 with the default shape.  Each against one CTA with
its records in device memory and, by verify mode, against fresh evaluations."""
import numpy as np
import pytest

import feedergen as fg

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("n,scen", [(4404, 1), (4405, 1), (5000, 4), (9792, 1), (9793, 1), (10000, 2), (13903, 4)])
def test_every_placement_gives_the_same_run(n, scen):
    import paper_2510_19608_gb300 as K
    f = fg.make_feeder(n, 9000 + n, phase_mode=(0.45, 0.15, 0.4), load=("lognormal", 15.0, 1.0), n_scen=scen)
    with K.Context(0) as ctx:
        for precision in (0, 1):
            runs = []
            for records, engine in ((0, 0), (1, 2), (0, 3)):
                try:
                    ctx.set_inc_shape(records=records)
                    ctx.reduce(f, K.default_params(margin=0.005, max_merges=4, precision=precision, engine=engine))
                finally:
                    ctx.reset_inc_shape()
                s = ctx.summary()
                assert s["engine"] == 2 and s["inc_mismatches"] == 0 and s["n_iter"] == 4
                runs.append((ctx.decisions(), ctx.assignment(), ctx.voltages()[1]))
            for dec, sup, vred in runs[1:]:
                assert all(np.array_equal(v, dec[k]) for k, v in runs[0][0].items())
                assert np.array_equal(runs[0][1], sup) and np.array_equal(runs[0][2], vred)
