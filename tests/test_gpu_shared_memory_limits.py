"""Kernels around the shared memory that a launch may have without asking for more.

A kernel gets 48 KB in all, its static arrays counted, unless the limit of its
dynamic part was raised; that limit then stays for the process.  So each size runs
in a process of its own, in which no larger one has raised the limit before.
"""
import os
import subprocess
import sys

import pytest

pytestmark = pytest.mark.gpu
ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))

HEAD = """
import numpy as np, feedergen as fg, paper_2510_19608_gb300 as K
from oracle import oracle as O
def feeder(n, scen):
    return fg.make_feeder(n, 50 + n, phase_mode=(0.5, 0.2, 0.3), n_scen=scen)
with K.Context(0) as ctx:
"""


def _run(body):
    src = HEAD + "".join("    " + line + "\n" for line in body.strip().splitlines())
    r = subprocess.run([sys.executable, "-c", src], cwd=ROOT, capture_output=True, text=True, timeout=300)
    assert r.returncode == 0, r.stderr[-2000:]


# (currents, voltages and the tree in shared memory: 96 n + about 10 n bytes)
@pytest.mark.parametrize("n", [460, 461, 462, 463, 464])
def test_evaluation(n):
    _run(f"""
f = feeder({n}, 2)
vhat, _ = O.operating_points(f)
err, w = ctx.evaluate(f, np.arange({n}, dtype=np.int32))
assert err.max() <= 1e-10 and np.abs(w - vhat).max() <= 1e-10
""")


# (a slice and the tree: 16 n + about 10 n bytes)
@pytest.mark.parametrize("n", [1888, 1889, 1890, 1891])
def test_load_flow(n):
    _run(f"""
f = feeder({n}, 2)
vhat, _ = O.operating_points(f)
v, i, _ = ctx.power_flow(f)
assert np.abs(v - vhat).max() <= 1e-10
""")


# (the first evaluation: about 10 n bytes beside 17 KB of static arrays; from 4,405
# buses on a cluster keeps its candidates and sums in device memory)
@pytest.mark.parametrize("precision", [0, 1])
@pytest.mark.parametrize("n", [3124, 3203, 4000, 4915, 4916])
def test_first_evaluation_alone(n, precision):
    _run(f"""
f = feeder({n}, 2)
kw = dict(margin=0.005, max_merges=3, precision={precision})
ctx.reduce(f, K.default_params(engine=3, **kw))
s, d, a = ctx.summary(), ctx.decisions(), ctx.assignment()
assert s["inc_mismatches"] == 0 and s["n_iter"] == 3
ctx.reduce(f, K.default_params(engine=1, **kw))
e = ctx.decisions()
assert np.array_equal(d["s"], e["s"]) and np.array_equal(d["r"], e["r"]) and np.array_equal(a, ctx.assignment())
assert np.allclose(d["score"], e["score"], rtol=0, atol=1e-9)
""")


@pytest.mark.parametrize("precision", [0, 1])
@pytest.mark.parametrize("n", [3125, 4000, 4915])
def test_first_evaluation_of_a_batch(n, precision):
    _run(f"""
fs = [feeder({n}, 2), feeder(90, 1)]
p = K.default_params(margin=0.005, max_merges=3, precision={precision})
items, parts, _ = ctx.reduce_batch(fs, p)
for f, it, sup in zip(fs, items, parts):
    ctx.reduce(f, p)
    one = ctx.summary()
    assert it["status"] == 0 and it["smice"] == one["smice"] and it["max_error"] == one["max_error"]
    assert np.array_equal(sup, ctx.assignment())
""")
