"""A batch's setup in each of its forms gives every feeder the bits it gets alone.

Line inverses: eight lanes per line up to 15,000 lines in the batch or 128 a feeder,
one thread per line above.  Load flows: the voltages in device memory when the
largest feeder leaves room for one CTA on an SM and there are more than two waves of
them; in device memory altogether above 1,920 buses.
"""
import numpy as np
import pytest

import feedergen as fg

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("sizes,scen", [
    ((1300,) + (130,) * 170, 2),                        # one thread per line, voltages in device memory
    ((1921, 1920, 129, 128, 127, 2) + (96,) * 130, 3),  # eight lanes per line, a feeder too large for shared memory
    ((1300,) + (130,) * 100, 1),                        # eight lanes, everything in shared memory
    ((1000,) * 8 + (128,) * 8, 4),
    ((700,) * 25, 4),                                   # one thread per line, everything in shared memory
])
def test_every_form_of_the_setup_gives_the_single_run_s_bits(sizes, scen):
    import paper_2510_19608_gb300 as K
    drawn = {}
    fs = []
    for i, n in enumerate(sizes):
        key = (n, i % 3)
        if key not in drawn:
            drawn[key] = fg.make_feeder(n, 4000 + n + i % 3, phase_mode=(0.4, 0.3, 0.3), n_scen=scen)
        fs.append(drawn[key])
    p = K.default_params(margin=0.005, max_merges=4, precision=0)
    with K.Context(0) as ctx:
        items, parts, _ = ctx.reduce_batch(fs, p)
        alone = {}
        for f, it, sup in zip(fs, items, parts):
            if id(f) not in alone:
                ctx.reduce(f, p)
                s = ctx.summary()
                alone[id(f)] = (s["smice"], s["max_error"], s["n_iter"], ctx.assignment())
            smice, err, k, one = alone[id(f)]
            assert it["status"] == 0 and it["n_iter"] == k
            assert it["smice"] == smice and it["max_error"] == err
            assert np.array_equal(sup, one)
