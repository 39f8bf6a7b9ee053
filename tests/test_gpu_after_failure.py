"""A call that the library refuses for want of memory is over with its status: the
next call on the context runs as if it had not been."""
import ctypes as C

import numpy as np
import pytest

import feedergen as fg
from oracle import mlp as M

pytestmark = pytest.mark.gpu


def test_calls_after_a_refused_allocation_succeed():
    import paper_2510_19608_gb300 as K
    rng = np.random.default_rng(2)
    theta, x = rng.normal(0, 0.12, M.n_params(14)).astype(np.float32), rng.normal(0, 1, (500, 14)).astype(np.float32)
    f = fg.make_feeder(60, 3, n_scen=2)
    p = K.default_params(margin=0.005, max_merges=5)
    ptr = lambda a: a.ctypes.data_as(C.c_void_p)
    with K.Context(0) as ctx:
        ctx.scorer_init(14, theta)
        ctx.reduce(f, p)
        dec, y, ytc = ctx.decisions(), ctx.scorer_predict(x), ctx.scorer_predict_tc(x)

        def refuse():                               # 2e9 samples' work buffers; neither array is read
            loss, t = C.c_double(), np.zeros(1, np.float32)
            assert K.lib().okr_scorer_gradient(ctx._h, ptr(x), ptr(t), C.c_int32(2_000_000_000), None,
                                               C.byref(loss)) == 2          # OKR_ENOMEM

        refuse()
        assert np.array_equal(ctx.scorer_predict(x), y)
        refuse()
        assert np.array_equal(ctx.scorer_predict_tc(x), ytc)
        refuse()
        ctx.reduce(f, p)
        assert all(np.array_equal(dec[k], v) for k, v in ctx.decisions().items())
