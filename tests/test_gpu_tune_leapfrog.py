"""The leapfrog tuner times what wave_step runs: its figure for 16 FP32 steps is
that of a wave_step call of 16 steps (2000^2: 43 us; 16 single launches 104 us),
and every shape gives the same steps.
"""
import math

import pytest
import torch

import eb_inputs as ei

pytestmark = pytest.mark.gpu


def test_tuner_times_the_path_of_wave_step():
    import __graft_entry__ as ge
    import paper_2204_06083_gb300 as eb
    ge.build()
    grid = ei.box_grid(2, 2000)
    h = eb.EB(grid, ei.random_star(1))
    dt = 0.9 * grid.h / math.sqrt(2.0)
    gen = torch.Generator(device="cuda").manual_seed(1)
    base = [torch.randn(h.shape(), generator=gen, device="cuda") for _ in range(2)]
    f = [t.clone() for t in base]
    h.wave_step(f[0], f[1], dt, 16)
    want = [t.clone() for t in f]
    res = h.autotune(eb.EB_F32, reps=20, op=eb.EB_TUNE_LEAPFROG)
    g = [t.clone() for t in base]
    h.wave_step(g[0], g[1], dt, 16)
    cp = (h.classes() & eb.CODE_CP) != 0  # which nodes off the CPs are cleared depends on the tiles
    assert torch.equal(g[0][cp], want[0][cp]) and torch.equal(g[1][cp], want[1][cp])
    times = []
    for _ in range(5):
        a, b = torch.cuda.Event(enable_timing=True), torch.cuda.Event(enable_timing=True)
        a.record()
        for _ in range(20):
            h.wave_step(f[0], f[1], 1e-12, 16)
        b.record()
        torch.cuda.synchronize()
        times.append(1000.0 * a.elapsed_time(b) / 20)
    assert min(res.us) <= 1.5 * min(times), (res.us, times)
