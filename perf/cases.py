"""The work this library is used for, as cases that can be timed and compared.

Each case is a plain dict: its ``kind`` names the entry point, the other keys
its sizes and options.  ``prepare`` makes the inputs from a seed, ``run`` is one
pass through the public entry points, ``work`` counts the bytes and operations
the path cannot do without, ``exact`` gives the same outputs in 64 bits from
plain numpy / torch where that is possible.
"""
from __future__ import annotations

import math

import numpy as np
import torch

import paper_2510_19608_gb300 as K
from paper_2510_19608_gb300 import _binding as B

FEATURES = 14           # features of one candidate row (the search's scorer)
HIDDEN = 128            # units of each hidden layer of the scorer
EXACT_BUSES = 160       # largest feeder whose whole search is repeated in numpy


def listed():
    return [
        # the 40-bus sub-feeder at the library's default parameters (FP64, until nothing is
        # feasible): the smallest call, launches and set-up count
        dict(name="reduce_40", kind="reduce", n=40, scen=2, mix="keep", target=1.0, precision=0, device=False),
        # the 1,000-bus feeder at 50 %, FP32 terms: the library's headline reduction, from host arrays
        dict(name="reduce_1000", kind="reduce", n=1000, scen=2, mix="urban", target=0.5, precision=1, device=False),
        # the 2,200-bus feeder at 90 %, the feeder already in device memory
        dict(name="reduce_2200", kind="reduce", n=2200, scen=2, mix="rural", target=0.9, precision=1, device=True),
        # the 3,100-bus feeder at 80 %, every score in FP64 (the default precision): the largest feeder
        dict(name="reduce_3100", kind="reduce", n=3100, scen=2, mix="rural", target=0.8, precision=0, device=False),
        # the other objective (largest error of the candidate network), an odd size, one scenario
        dict(name="maxerr_501", kind="maxerr", n=501, scen=1, mix="urban", target=0.5, precision=1),
        # a utility's feeders in one launch: 256 of 200 to 2,000 buses, targets 50 / 70 / 90 %
        dict(name="batch_256", kind="batch", count=256, lo=200, hi=2000, scen=2, precision=1),
        # the same small feeders again and again under new loads: a captured batch plan
        dict(name="plan_48", kind="plan", count=48, lo=60, hi=400, scen=1, precision=1),
        # the reduced network of a given kept set: Y_Kron and the buses that make it radial
        dict(name="kron_1000", kind="kron", n=1000, scen=2, mix="urban", kept=0.5),
        # a reduction tested on the 24 hours of a day, four operating points a call
        dict(name="hours_1000", kind="hours", n=1000, hours=24, mix="urban", kept=0.5),
        # training the candidate scorer: one pass over recorded candidates in minibatches
        dict(name="train_64k", kind="train", samples=65536, batch=4096, features=FEATURES),
        # scoring candidates with FP32 activations, a ragged count
        dict(name="predict_300k", kind="predict", samples=300007, features=FEATURES, tc=False),
        # scoring many candidates at once on the tensor cores, a ragged count
        dict(name="predict_tc_3m", kind="predict", samples=3000017, features=FEATURES, tc=True),
    ]


def _log(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def draw(rng):
    kind = rng.choice(["reduce", "reduce", "reduce", "maxerr", "batch", "plan", "kron", "hours", "flow", "train",
                       "gradient", "predict", "predict"])
    mix = rng.choice(["urban", "rural", "keep"])
    if kind == "reduce":
        scen = rng.choice([1, 2, 2, 3, 4])
        n = _log(rng, 24, 3100 if scen <= 2 else 1500)
        return dict(kind=kind, n=n, scen=scen, mix=mix, target=round(rng.uniform(0.3, 0.8), 2),
                    precision=rng.choice([0, 1]), device=rng.choice([False, True]))
    if kind == "maxerr":
        return dict(kind=kind, n=_log(rng, 40, 900), scen=rng.choice([1, 2]), mix=mix,
                    target=round(rng.uniform(0.3, 0.6), 2), precision=rng.choice([0, 1]))
    if kind in ("batch", "plan"):
        lo = _log(rng, 30, 300)
        return dict(kind=kind, count=_log(rng, 3, 160), lo=lo, hi=min(1600, lo * rng.choice([2, 3, 5])),
                    scen=rng.choice([1, 2]), precision=rng.choice([0, 1, 1]))
    if kind == "kron":
        return dict(kind=kind, n=_log(rng, 30, 1800), scen=1, mix=mix, kept=round(rng.uniform(0.15, 0.7), 2))
    if kind == "hours":
        return dict(kind=kind, n=_log(rng, 30, 3000), hours=rng.choice([5, 12, 24]), mix=mix,
                    kept=round(rng.uniform(0.2, 0.8), 2))
    if kind == "flow":
        return dict(kind=kind, n=_log(rng, 30, 4096), scen=rng.choice([1, 2, 3, 4]), mix=mix)
    if kind == "train":
        batch = _log(rng, 500, 8192)
        return dict(kind=kind, samples=batch * rng.randint(1, 12) + rng.randint(0, batch - 1), batch=batch,
                    features=FEATURES)
    if kind == "gradient":
        return dict(kind=kind, samples=_log(rng, 100, 200000), features=rng.choice([FEATURES, FEATURES, 12, 5]))
    return dict(kind="predict", samples=_log(rng, 100, 2000000), features=rng.choice([FEATURES, FEATURES, 16, 3]),
                tc=rng.choice([True, True, False]))


# ---------------------------------------------------------------- inputs
class Feeder:
    """A radial feeder in the form the entry points take."""

    def __init__(self, parent, phases, z_line, s_load, v_slack):
        self.parent, self.phases, self.z_line, self.s_load, self.v_slack = parent, phases, z_line, s_load, v_slack
        self.n_bus, self.n_scen = int(parent.shape[0]), int(s_load.shape[0])


_MIX = {    # kV, probability that a lateral bus drops phases, load in kW per phase
    "keep": (4.16, 0.30, ("uniform", 50.0)),
    "urban": (12.47, 0.12, ("uniform", 100.0)),
    "rural": (12.47, 0.30, ("lognormal", 15.0)),
}


def _levels(parent):
    """Buses by depth.  The tree is drawn breadth first, so levels are ranges."""
    n = parent.shape[0]
    depth = np.zeros(n, np.int64)
    edges = [0, 1]
    while edges[-1] < n:
        lo, hi = edges[-2], edges[-1]
        end = int(np.searchsorted(parent[hi:], hi) + hi)        # children of [lo, hi): parents below hi
        depth[hi:end] = depth[lo] + 1
        edges.append(end)
    return edges


def make_feeder(rng, n, scen, mix, tree=None):
    """Breadth-first tree with 1-3 children per bus, three-phase trunk and laterals that
    lose phases, lognormal line lengths, 30 % unloaded buses; loads scaled so that the
    linear voltage drop stays within 10 %; scenario l carries 0.3^l of the load.
    ``tree``: a generator for the tree and its phases alone (else ``rng`` draws them)."""
    kv, q_drop, load = _MIX[mix]
    tree = tree or rng
    parent = np.concatenate([[-1], np.repeat(np.arange(n), tree.integers(1, 4, n))[:n - 1]]).astype(np.int32)
    edges = _levels(parent)
    size = np.ones(n, np.int64)
    for lo, hi in reversed(list(zip(edges[1:-1], edges[2:]))):
        np.add.at(size, parent[lo:hi], size[lo:hi])
    # phases: a lateral bus (5 % of the buses at most below it) drops to a subset
    has = np.ones((n, 3), bool)
    lateral = size <= max(1, int(0.05 * n)) if mix != "keep" else np.ones(n, bool)
    u, pick = tree.random(n), tree.random((n, 3))
    for lo, hi in zip(edges[1:-1], edges[2:]):
        ph = has[parent[lo:hi]]
        cnt = ph.sum(1)
        drop = (u[lo:hi] < q_drop) & lateral[lo:hi] & (cnt > 1)
        left = np.where(pick[lo:hi, 0] < 0.5, 1, cnt - 1)
        order = np.argsort(np.argsort(np.where(ph, pick[lo:hi], 2.0), axis=1), axis=1)
        has[lo:hi] = ph & (~drop[:, None] | (order < left[:, None]))
    phases = (has * np.array([1, 2, 4])).sum(1).astype(np.uint8)
    # lines
    zr, zx = rng.uniform(0.05, 0.15, (n, 3, 3)), rng.uniform(0.2, 0.5, (n, 3, 3))
    for m in (zr, zx):
        m[:] = np.triu(m, 1) + np.swapaxes(np.triu(m, 1), 1, 2)
    zr[:, range(3), range(3)] = rng.uniform(0.3, 0.6, (n, 3))
    zx[:, range(3), range(3)] = rng.uniform(0.6, 1.4, (n, 3))
    length = np.clip(rng.lognormal(math.log(0.1), 0.7, n), 0.02, 0.5) / (kv * kv)
    z = np.stack([zr, zx], -1) * length[:, None, None, None] * (has[:, :, None] & has[:, None, :])[..., None]
    z[0] = 0.0
    # loads
    p = rng.uniform(0.0, load[1], (n, 3)) if load[0] == "uniform" else rng.lognormal(math.log(load[1]), 1.0, (n, 3))
    s = (p + 1j * p * np.tan(np.arccos(rng.uniform(0.88, 0.98, (n, 3))))) * (3.0 / 1000.0)
    s *= has & (rng.random(n) >= 0.3)[:, None]
    s[0] = 0.0
    down = np.abs(s)
    for lo, hi in reversed(list(zip(edges[1:-1], edges[2:]))):
        np.add.at(down, parent[lo:hi], down[lo:hi])
    fall = np.einsum("npq,nq->np", np.hypot(z[..., 0], z[..., 1]), down)
    for lo, hi in zip(edges[1:-1], edges[2:]):
        fall[lo:hi] += fall[parent[lo:hi]]
    s *= min(1.0, 0.10 / max(float(fall.max()), 1e-12))
    s_load = np.stack([np.stack([(s * 0.3 ** l).real, (s * 0.3 ** l).imag], -1) for l in range(scen)])
    ang = np.array([0.0, -2.0, 2.0]) * math.pi / 3.0
    return Feeder(parent, phases, np.ascontiguousarray(z), np.ascontiguousarray(s_load),
                  np.stack([np.cos(ang), np.sin(ang)], -1))


def _rng(seed):
    return np.random.default_rng(int(seed) % (1 << 63))


def _feeder(case, seed, scen=None):
    # Y_Kron's size is the kept phase-nodes': its network is the same under every seed, with
    # other line impedances and loads
    tree = _rng(case["n"]) if case["kind"] == "kron" else None
    return make_feeder(_rng(seed), case["n"], scen or case["scen"], case["mix"], tree)


def _kept(f, share, seed):
    """A random connected assignment: every bus is kept with the given probability (bus 0
    always) and the others join the nearest kept bus above them."""
    rng, n = _rng(seed + 77), f.n_bus
    keep = rng.random(n) < share
    keep[0] = True
    sup = np.arange(n, dtype=np.int32)
    edges = _levels(f.parent)
    for lo, hi in zip(edges[1:-1], edges[2:]):
        top = sup[f.parent[lo:hi]]
        sup[lo:hi] = np.where(keep[lo:hi], np.arange(lo, hi), top)
    return keep.astype(np.uint8), sup


def _hours(f, hours, seed):
    """Hourly loads [hours, n, 3, 2]: a daily shape, shifted and scaled per bus."""
    rng = _rng(seed + 55)
    h = np.arange(hours)[:, None] + rng.uniform(-2.0, 2.0, f.n_bus)[None, :]
    shape = 0.55 + 0.30 * np.sin(2 * math.pi * (h - 10.0) / 24.0) + 0.15 * np.exp(-((h % 24 - 19.0) ** 2) / 8.0)
    fac = shape * rng.lognormal(0.0, 0.15, (hours, f.n_bus))
    return f.s_load[0][None] * fac[:, :, None, None]


def _theta(features, seed):
    """Scorer parameters: He-normal weights and small biases."""
    rng, H = _rng(seed + 33), HIDDEN
    parts = []
    for a, b, c in ((features, H, 2.0), (H, H, 2.0), (H, H, 2.0), (H, 1, 1.0)):
        parts += [rng.normal(0.0, math.sqrt(c / a), (a, b)), rng.normal(0.0, 0.05, b)]
    return np.concatenate([x.ravel() for x in parts]).astype(np.float32)


def _samples(case, seed):
    """Feature rows as the search records them (scaled logarithms, shares and counts of
    order one) and targets on their log scale."""
    g = torch.Generator().manual_seed(int(seed) % (1 << 62))
    x = torch.randn(case["samples"], case["features"], generator=g, dtype=torch.float32)
    t = (-2.0 + 2.0 * torch.randn(case["samples"], generator=g, dtype=torch.float32)).clamp_(-6.0, 2.0)
    return x.numpy(), t.numpy()


def _batch_inputs(case, seed):
    rng = _rng(seed)
    feeders, params = [], []
    for n in _rng(case["count"]).integers(case["lo"], case["hi"] + 1, case["count"]).tolist():
        feeders.append(make_feeder(rng, n, case["scen"], "urban"))
        params.append(B.default_params(margin=0.005, target_reduction=float(rng.choice([0.5, 0.7, 0.9])),
                                       precision=case["precision"]))
    return feeders, params


def prepare(case, seed):
    kind = case["kind"]
    st = dict(case=case, ctx=K.Context(0))
    if kind in ("reduce", "maxerr"):
        f = _feeder(case, seed)
        st["params"] = B.default_params(margin=0.005, target_reduction=case["target"], precision=case["precision"],
                                        objective=1 if kind == "maxerr" else 0)
        st["feeder"] = f
        if case.get("device"):
            dev = [torch.from_numpy(a).cuda() for a in (f.parent, f.phases, f.z_line, f.s_load)]
            st["keep"] = dev
            st["dfeeder"] = B.device_feeder(f.n_bus, f.n_scen, *[d.data_ptr() for d in dev], f.v_slack)
    elif kind in ("batch", "plan"):
        feeders, params = _batch_inputs(case, seed)
        st["feeders"], st["params"] = feeders, params
        if kind == "plan":
            st["plan"] = st["ctx"].batch_plan(feeders, params)
            st["loads"] = [f.s_load * 0.97 for f in feeders[::4]]
    elif kind == "kron":
        f = _feeder(case, seed)
        st["kept"], _ = _kept(f, case["kept"], case["n"])
        st["ctx"].power_flow(f)
    elif kind == "hours":
        f = _feeder(case, seed, 1)
        _, st["super_of"] = _kept(f, case["kept"], seed)
        h = _hours(f, case["hours"], seed)
        st["feeders"] = [Feeder(f.parent, f.phases, f.z_line, np.ascontiguousarray(h[k:k + 4]), f.v_slack)
                         for k in range(0, case["hours"], 4)]
    elif kind == "flow":
        f = _feeder(case, seed)
        dev = [torch.from_numpy(a).cuda() for a in (f.parent, f.phases, f.z_line, f.s_load)]
        out = [torch.zeros(f.n_scen, f.n_bus, 3, 2, dtype=torch.float64, device="cuda") for _ in range(2)]
        torch.cuda.synchronize()
        st.update(keep=dev, out=out,
                  dfeeder=B.device_feeder(f.n_bus, f.n_scen, *[d.data_ptr() for d in dev], f.v_slack))
    else:
        st["x"], st["t"] = _samples(case, seed)
        st["theta"] = _theta(case["features"], seed)
        st["ctx"].scorer_init(case["features"], st["theta"])
    return st


# ---------------------------------------------------------------- one pass
def run(st):
    case, ctx = st["case"], st["ctx"]
    kind = case["kind"]
    if kind in ("reduce", "maxerr"):
        if "dfeeder" in st:
            ctx.reduce_device(st["dfeeder"], st["params"])
        else:
            ctx.reduce(st["feeder"], st["params"])
        vhat, vred = ctx.voltages()
        return dict(decisions={k: _padded(v, case["n"]) for k, v in ctx.decisions().items()},
                    super_of=ctx.assignment(), vhat=vhat, vred=vred)
    if kind == "batch":
        return _batch_out(*ctx.reduce_batch(st["feeders"], st["params"])[:2])
    if kind == "plan":
        for k, s in enumerate(st["loads"]):
            st["plan"].set_loads(4 * k, s)
        return _batch_out(*st["plan"].run()[:2])
    if kind == "kron":
        y, pn = ctx.kron(st["kept"])
        return dict(y=y, phase_node=pn, critical=ctx.radialize(st["kept"]))
    if kind == "hours":
        got = [ctx.evaluate(f, st["super_of"]) for f in st["feeders"]]
        return dict(error=np.concatenate([e for e, _ in got]), v=[v for _, v in got])
    if kind == "flow":
        sweeps = B.power_flow_static(st["dfeeder"], st["out"][0].data_ptr(), st["out"][1].data_ptr())
        return dict(vhat=st["out"][0], ihat=st["out"][1], sweeps=sweeps)
    if kind == "gradient":
        g, loss = ctx.scorer_gradient(st["x"], st["t"])
        return dict(grad=g, loss=loss)
    if kind == "train":
        ctx.scorer_init(case["features"], st["theta"])
        loss = ctx.scorer_train(st["x"], st["t"], batch=case["batch"], epochs=1, lr=1e-3)
        return dict(theta=ctx.scorer_params(), loss=loss)
    return dict(y=ctx.scorer_predict_tc(st["x"]) if case["tc"] else ctx.scorer_predict(st["x"]))


def _padded(a, n):
    """A decision per merge, at the length of the longest search (it may stop earlier)."""
    out = np.zeros(n, a.dtype)
    out[:a.shape[0]] = a
    return out


def _batch_out(items, parts):
    return dict(super_of=np.concatenate(parts),
                **{k: np.array([it[k] for it in items])
                   for k in ("status", "n_iter", "stop_reason", "n_kept", "candidates", "smice", "max_error")})


# ---------------------------------------------------------------- what a pass cannot do without
def _search_work(n, scen):
    """Inputs and outputs once.  Operations: the first score of every candidate (its
    positions are the buses below it) and the terms the merges change, about 40
    operations per (candidate, phase-node, scenario); about ten load-flow sweeps."""
    items = 2.4 * scen * n * (2.0 * math.log2(n) + 20.0)
    return n * (4 + 1 + 144 + 48 * scen) + n * (40 + 96 * scen), 40.0 * items + 10.0 * 2.4 * scen * n * 40.0


def _mlp_flops(features):
    return 2.0 * (features * HIDDEN + 2 * HIDDEN * HIDDEN + HIDDEN)


def work(case):
    kind = case["kind"]
    if kind in ("reduce", "maxerr"):
        b, f = _search_work(case["n"], case["scen"])
        return dict(bytes=b, flops=f)
    if kind in ("batch", "plan"):
        b, f = _search_work((case["lo"] + case["hi"]) / 2.0, case["scen"])
        return dict(bytes=case["count"] * b, flops=case["count"] * f)
    if kind == "kron":
        k = 2.4 * max(1.0, case["n"] * case["kept"])
        return dict(bytes=16.0 * k * k + 160.0 * case["n"], flops=500.0 * case["n"])
    if kind in ("hours", "flow"):
        points = case["hours"] if kind == "hours" else case["scen"]
        return dict(bytes=case["n"] * (149.0 + points * 48.0 * 2), flops=10.0 * 2.4 * points * case["n"] * 40.0)
    s, f = case["samples"], case["features"]
    if kind == "predict":
        return dict(bytes=4.0 * s * (f + 1), flops=s * _mlp_flops(f))
    return dict(bytes=4.0 * s * (f + 1), flops=3.0 * s * _mlp_flops(f))


# ---------------------------------------------------------------- the same in 64 bits
def _load_flow(f):
    """Voltages [L, n, 3] of every scenario by backward / forward sweeps, in numpy."""
    z = f.z_line[..., 0] + 1j * f.z_line[..., 1]
    s = f.s_load[..., 0] + 1j * f.s_load[..., 1]
    has = (f.phases[:, None] >> np.arange(3) & 1).astype(bool)
    v0 = (f.v_slack[:, 0] + 1j * f.v_slack[:, 1])[None, None, :]
    v = np.where(has[None], np.broadcast_to(v0, s.shape), 0.0)
    edges = _levels(f.parent)
    spans = list(zip(edges[1:-1], edges[2:]))
    for _ in range(300):
        j = np.where(has[None], np.conj(s / np.where(has[None], v, 1.0)), 0.0)
        j[:, 0] = 0.0
        for lo, hi in reversed(spans):
            np.add.at(j, (slice(None), f.parent[lo:hi]), j[:, lo:hi])
        drop = np.einsum("npq,lnq->lnp", z, j)
        new = v.copy()
        for lo, hi in spans:
            new[:, lo:hi] = np.where(has[None, lo:hi], new[:, f.parent[lo:hi]] - drop[:, lo:hi], 0.0)
        done = float(np.abs(new - v).max()) < 1e-15
        v = new
        if done:
            break
    return v


def _path_z(f):
    """Z[i, j] = path impedance of the lowest common ancestor of i and j, [n, n, 3, 3]."""
    n, z = f.n_bus, f.z_line[..., 0] + 1j * f.z_line[..., 1]
    zc = np.zeros((n, 3, 3), complex)
    anc = np.zeros((n, n), bool)
    for i in range(1, n):
        zc[i] = zc[f.parent[i]] + z[i]
        anc[i] = anc[f.parent[i]]
        anc[i, i] = True
    out = np.zeros((n, n, 3, 3), complex)
    for a in range(1, n):
        below = np.nonzero(anc[:, a])[0]
        out[np.ix_(below, below)] += z[a]
    return out


def _injections(f, v):
    """Ihat = Y vhat per bus, and Y's line blocks."""
    n, z = f.n_bus, f.z_line[..., 0] + 1j * f.z_line[..., 1]
    i = np.zeros_like(v)
    for k in range(1, n):
        p = [q for q in range(3) if f.phases[k] >> q & 1]
        y = np.linalg.inv(z[k][np.ix_(p, p)])
        c = (v[:, k][:, p] - v[:, f.parent[k]][:, p]) @ y.T
        i[:, k, p] += c
        i[:, f.parent[k], p] -= c
    return i


def _greedy(f, v, target, margin=0.005, tau=1e-9):
    """The exhaustive search on a small feeder: candidates, scores, ties and stop rule as
    the method states them, every candidate from scratch."""
    n, has = f.n_bus, (f.phases[:, None] >> np.arange(3) & 1).astype(bool)
    Z, inj, mag = _path_z(f), _injections(f, v), np.abs(v)
    cur, sup = v.copy(), np.arange(n)
    dec = []

    def smice(vc, s):
        e = np.where(has[None], np.abs(mag - np.abs(vc[:, s])), 0.0).max(2)       # [L, n]
        m = np.zeros_like(e)
        for l in range(e.shape[0]):
            np.maximum.at(m[l], s, e[l])
        return m.sum(), e.max()

    for _ in range(min(n - 1, math.ceil(target * n - 1e-12))):
        found = []
        for i in range(1, n):
            a, b = sup[f.parent[i]], sup[i]
            if a == b:
                continue
            for s, r in ((a, b), (b, a)):
                if r == 0 or (f.phases[r] & f.phases[s]) != f.phases[r]:
                    continue
                vc = cur + np.einsum("npq,lq->lnp", Z[:, s] - Z[:, r], inj[:, r])
                sc, me = smice(vc, np.where(sup == r, s, sup))
                found.append((sc, me, int(r), int(s), vc))
        ok = [c for c in found if c[1] <= margin]
        if not ok:
            break
        m = min(c[0] for c in ok)
        sc, me, r, s, cur = min((c for c in ok if c[0] <= m + tau), key=lambda c: (c[2], c[3]))
        inj[:, s] += inj[:, r]
        inj[:, r] = 0.0
        sup = np.where(sup == r, s, sup)
        dec.append((s, r, sc, me))
    return dec, cur, sup


def _mlp64(theta, features, x):
    """Forward pass in 64 bits at the bfloat16 weights the products use."""
    H, o, out = HIDDEN, 0, []
    th = torch.from_numpy(theta).cuda()
    for a, b in ((features, H), (H, H), (H, H), (H, 1)):
        w = th[o:o + a * b].bfloat16().double().reshape(a, b)
        out.append((w, th[o + a * b:o + a * b + b].double()))
        o += a * b + b
    return out


def exact(case, seed):
    kind = case["kind"]
    if kind == "reduce" or kind == "maxerr":
        f = _feeder(case, seed)
        v = _load_flow(f)
        dec, vred, sup = None, None, None
        if kind == "reduce" and f.n_bus <= EXACT_BUSES and f.n_scen <= 2:
            got, cur, s = _greedy(f, v, case["target"])
            dec = dict(gap=None, maxerr=_padded(np.array([d[3] for d in got]), f.n_bus), ncand=None, r=None,
                       s=None, score=_padded(np.array([d[2] for d in got]), f.n_bus))
            has = (f.phases[:, None] >> np.arange(3) & 1).astype(bool)
            vred = np.where(has[None], cur[:, s], 0.0)
        return dict(decisions=dec, super_of=sup, vhat=v, vred=vred)
    if kind == "kron":
        f = _feeder(case, seed)
        kept, _ = _kept(f, case["kept"], case["n"])
        has = (f.phases[:, None] >> np.arange(3) & 1).astype(bool)
        row = np.cumsum(has.ravel()).reshape(-1, 3) - 1
        N = int(has.sum())
        if N > 5200:
            return None
        z = f.z_line[..., 0] + 1j * f.z_line[..., 1]
        Y = torch.zeros(N, N, dtype=torch.complex128)
        for k in range(1, f.n_bus):
            p = np.nonzero(has[k])[0]
            y = torch.from_numpy(np.linalg.inv(z[k][np.ix_(p, p)]))
            a, b = torch.from_numpy(row[k, p]), torch.from_numpy(row[f.parent[k], p])
            for i, j, sgn in ((a, a, 1), (b, b, 1), (a, b, -1), (b, a, -1)):
                Y[i[:, None], j[None, :]] += sgn * y
        kf = torch.from_numpy(np.repeat(kept.astype(bool), 3)[has.ravel()])
        Y = Y.cuda()
        kf = kf.cuda()
        kk, kr, rk, rr = Y[kf][:, kf], Y[kf][:, ~kf], Y[~kf][:, kf], Y[~kf][:, ~kf]
        out = kk - kr @ torch.linalg.solve(rr, rk) if rr.numel() else kk
        return dict(critical=None, phase_node=None, y=out.cpu().numpy())
    if kind == "flow":
        f = _feeder(case, seed)
        v = _load_flow(f)
        v2 = np.stack([v.real, v.imag], -1)
        return dict(ihat=None, sweeps=None, vhat=v2)
    if kind == "predict":
        x, _ = _samples(case, seed)
        w = _mlp64(_theta(case["features"], seed), case["features"], x)
        ys = []
        for c in torch.from_numpy(x).split(1 << 18):
            h = c.cuda().double()
            for a, b in w[:3]:
                h = torch.relu(h @ a + b)
            ys.append((h @ w[3][0] + w[3][1]).squeeze(1).cpu())
        return dict(y=torch.cat(ys).numpy())
    if kind == "gradient":
        x, t = _samples(case, seed)
        w = [(a.requires_grad_(), b.requires_grad_())
             for a, b in _mlp64(_theta(case["features"], seed), case["features"], x)]
        h = torch.from_numpy(x).cuda().double()
        for a, b in w[:3]:
            h = torch.relu(h @ a + b)
        y = (h @ w[3][0] + w[3][1]).squeeze(1)
        loss = (y - torch.from_numpy(t).cuda().double()).square().mean()
        loss.backward()
        g = torch.cat([p.grad.ravel() for a, b in w for p in (a, b)])
        return dict(grad=g.cpu().numpy(), loss=float(loss))
    # batches, plans and hours return what a search or an evaluation gives for many feeders;
    # training rounds its weights to bfloat16 at every step, which no 64-bit run repeats
    return None
