"""Double-float solves around the sizes where the list kernels' CTAs change.

The kernels of the double-float iteration change from CTAs of 64 threads to 256
at 64 pairs per SM, the others at 256.  Solutions on both sides of 64 pairs per
SM by the oracle's residual; and an iteration just below 256 pairs per SM takes no
longer than just above (a fifth longer while the double-float kernels changed there
too: four times the partials, a quarter of the threads to sum them).
"""
import statistics

import numpy as np
import pytest
import torch

import eb_inputs as ei
from oracle import eb as oeb

pytestmark = pytest.mark.gpu


def _sides(eb, per_sm, n):
    """((handle, n) just below, (handle, n) just above) per_sm CP pairs per SM"""
    def pairs(h):
        return int(((h.classes().view(-1, 2) & eb.CODE_CP) != 0).any(dim=1).sum())

    line = per_sm * torch.cuda.get_device_properties(0).multi_processor_count
    last = None
    while True:
        h = eb.EB(*ei.circle_k1(n))
        if pairs(h) >= line:
            break
        last, n = h, n + 2
    assert pairs(last) < line <= pairs(h) and pairs(h) - pairs(last) < line // 25
    return (last, n - 2), (h, n)


@pytest.fixture(scope="module")
def eb():
    import __graft_entry__ as ge
    import paper_2204_06083_gb300 as eb
    ge.build()
    return eb


@pytest.fixture(scope="module")
def small(eb):
    return [(h, oeb.build(*ei.circle_k1(n))) for h, n in _sides(eb, 64, 200)]


@pytest.mark.parametrize("side", [0, 1])
@pytest.mark.parametrize("vprec", ["EB_F32", "EB_BF16"])
@pytest.mark.parametrize("sigma", [0.0, 50.0])
def test_solve(eb, small, side, vprec, sigma):
    h, ref = small[side]
    amg = eb.AMG(h, sigma, vcycle_prec=getattr(eb, vprec))
    b = np.random.default_rng(side).standard_normal(ref.num_cp)
    for use_graph in (1, 0, 2):
        x, st = amg.solve(torch.tensor(ref.to_grid(b), device="cuda"), rtol=1e-11, outer=eb.EB_DF64,
                          use_graph=use_graph)
        v = ref.from_grid(x.cpu().numpy())
        assert st.converged
        assert np.linalg.norm(b - ref.A @ v - sigma * v) <= 2e-11 * np.linalg.norm(b)


def test_time_of_an_iteration(eb):
    solvers = []
    for h, n in _sides(eb, 256, 400):
        b = torch.randn((n, n), generator=torch.Generator(device="cuda").manual_seed(1), device="cuda",
                        dtype=torch.float64)
        solvers.append((eb.AMG(h, vcycle_prec=eb.EB_F32), b.contiguous()))
    times = [[], []]
    for rep in range(12):
        for k, (amg, b) in enumerate(solvers):
            x = torch.zeros_like(b)
            torch.cuda.synchronize()
            e0, e1 = torch.cuda.Event(enable_timing=True), torch.cuda.Event(enable_timing=True)
            e0.record()
            st = amg.solve(b, x=x, rtol=1e-11, outer=eb.EB_DF64)[1]
            e1.record()
            torch.cuda.synchronize()
            if rep >= 3:
                times[k].append(e0.elapsed_time(e1) / st.iterations)
    below, above = (statistics.median(t) for t in times)
    assert below <= 1.06 * above, (below, above)
