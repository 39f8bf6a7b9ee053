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
