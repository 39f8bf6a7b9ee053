"""Feeders of different sizes reduced by threads of one process, each with a context
of its own: every call succeeds and gives what it gives alone.  (The limit of a
kernel's dynamic shared memory is shared by all threads; one set for a small feeder
between another thread's own setting and its launch refused that launch.)"""
import ctypes as C
import threading

import numpy as np
import pytest

import feedergen as fg

pytestmark = pytest.mark.gpu


def test_threads_with_small_and_large_feeders_on_one_kernel():
    import paper_2510_19608_gb300 as K
    from paper_2510_19608_gb300 import _binding as B
    p = K.default_params(margin=0.005, max_merges=1, precision=1)
    faults, done = [], threading.Event()

    def run(n, reps):
        try:
            f = fg.make_feeder(n, 60 + n, n_scen=1)
            hf = B.HostFeeder(f)
            with K.Context(0) as ctx:
                ctx.set_inc_shape(records=1)        # one CTA, records in device memory: the same kernel for all
                ctx.reduce(f, p)
                want = ctx.decisions()
                for _ in range(reps):
                    if K.lib().okr_reduce(ctx._h, C.byref(hf.c), C.byref(p)) != 0:
                        faults.append((n, K.lib().okr_last_error(ctx._h)))
                    if reps > 10_000 and done.is_set():
                        break
                ctx.reduce(f, p)
                got = ctx.decisions()
                assert all(np.array_equal(want[k], got[k]) for k in want)
        except Exception as e:                      # noqa: BLE001 -- reported below, whatever it was
            faults.append((n, repr(e)))

    large = [threading.Thread(target=run, args=(900 + 100 * i, 1200)) for i in range(4)]
    small = [threading.Thread(target=run, args=(4 + i, 10 ** 9)) for i in range(11)]
    for t in large + small:
        t.start()
    for t in large:
        t.join()
    done.set()
    for t in small:
        t.join()
    assert not faults, (len(faults), faults[:3])
