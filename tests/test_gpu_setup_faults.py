"""The setup under inputs at the edge of what it takes.

A singular line: its inverse is formed beside the load flow and names it in the
setup's error flag while the load flow runs.  The call returns the singular line
at once (no CTA of the load flow waits for one that left), whatever the size, and
leaves the context as it was.

A device array of doubles at an odd multiple of 8 bytes is a double's array like
any other for the entry point that reads the caller's memory.
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


@pytest.mark.parametrize("n,scen", [(5, 1), (256, 2), (300, 3)])
def test_static_load_flow_reads_arrays_at_any_double_s_address(n, scen):
    import torch
    import paper_2510_19608_gb300 as K
    f = fg.make_feeder(n, 21, phase_mode=(0.5, 0.2, 0.3), n_scen=scen)
    par, ph = torch.from_numpy(f.parent).cuda(), torch.from_numpy(f.phases).cuda()
    runs = []
    for shift in (0, 1):                    # doubles from a 16-byte boundary
        z = torch.zeros(f.z_line.size + 2, dtype=torch.float64, device="cuda")
        s = torch.zeros(f.s_load.size + 2, dtype=torch.float64, device="cuda")
        z[shift:shift + f.z_line.size] = torch.from_numpy(f.z_line.reshape(-1)).cuda()
        s[shift:shift + f.s_load.size] = torch.from_numpy(f.s_load.reshape(-1)).cuda()
        v = torch.full((scen * n * 6 + 2,), float("nan"), dtype=torch.float64, device="cuda")
        i = torch.full((scen * n * 6 + 2,), float("nan"), dtype=torch.float64, device="cuda")
        assert z.data_ptr() % 16 == 0 and v.data_ptr() % 16 == 0
        at = 8 * shift
        df = K.device_feeder(n, scen, par.data_ptr(), ph.data_ptr(), z.data_ptr() + at, s.data_ptr() + at, f.v_slack)
        torch.cuda.synchronize()
        sw = K.power_flow_static(df, v.data_ptr() + at, i.data_ptr() + at, torch.cuda.current_stream().cuda_stream)
        k = scen * n * 6
        runs.append((sw, v[shift:shift + k].cpu().numpy(), i[shift:shift + k].cpu().numpy()))
    assert runs[0][0] == runs[1][0]
    assert np.isfinite(runs[0][1]).all()
    assert np.array_equal(runs[0][1], runs[1][1]) and np.array_equal(runs[0][2], runs[1][2])
