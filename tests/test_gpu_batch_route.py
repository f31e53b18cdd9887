"""batch_set_level0_tma takes effect on a batch that has solved before: the
kernels of the next solve's level-0 steps, as the profiler lists them, are those
of the route in force, in captured iterations too.
"""
import pytest
import torch

import eb_inputs as ei

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("host_loop", [False, True])
def test_level0_route_after_a_solve(host_loop):
    import __graft_entry__ as ge
    import paper_2204_06083_gb300 as eb
    from torch.profiler import ProfilerActivity, profile
    ge.build()
    grids = [ei.box_grid(2, n) for n in (96, 128)]
    B = eb.Batch(grids, [ei.random_star(k) for k in (41, 42)])
    B.heat_setup([g.h for g in grids], vcycle_prec=eb.EB_F32)
    B.set_profile(host_loop)
    gen = torch.Generator(device="cuda").manual_seed(1)
    b1 = torch.randn(B.num_nodes, generator=gen, device="cuda", dtype=torch.float64)

    def kernels():
        u = B.zeros()
        with profile(activities=[ProfilerActivity.CUDA]) as p:
            B.heat_step(u, b1, rtol=1e-10)
            torch.cuda.synchronize()
        return [e.name for e in p.events()]

    kernels()  # the first profile of a process may miss kernels
    for on in (False, True, False):
        B.set_level0_tma(on)
        names = kernels()
        if not any("k_g_cheb_first" in n for n in names):
            pytest.skip("the profiler records no kernels here")
        copies = sum("k_g_cheb_step_tma" in n for n in names)
        sweeps = sum("k_g_cheb_step<2, float, float, 0>" in n for n in names)
        assert (copies == 0 and sweeps > 0) if not on else (copies > 0 and sweeps == 0), (on, copies, sweeps)
