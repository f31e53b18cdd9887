"""Solves of right-hand sides of extreme size: b and s b give x and s x.

At s = 1e-146 the products r'z of the last iterations lie below FP64's normal
range, where their reciprocals are infinite; some ten digits of them are left,
so the solution scales to 1e-8.  s is a power of two times that, so that nothing
else rounds differently.
"""
import math

import pytest
import torch

import eb_inputs as ei

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("precond", ["EB_PC_AMG", "EB_PC_JACOBI"])
@pytest.mark.parametrize("use_graph,check_every", [(1, 1), (0, 1)])
@pytest.mark.parametrize("exponent", [-485, -300, 300, 480])
def test_solution_scales_with_the_right_hand_side(precond, use_graph, check_every, exponent):
    import __graft_entry__ as ge
    import paper_2204_06083_gb300 as eb
    ge.build()
    grid, ls = ei.circle_k1(64)
    h = eb.EB(grid, ls)
    amg = eb.AMG(h, coarse_max=30)
    gen = torch.Generator(device="cuda").manual_seed(2)
    b = torch.randn(h.shape(), generator=gen, device="cuda", dtype=torch.float64)
    kw = dict(rtol=1e-10, precond=getattr(eb, precond), use_graph=use_graph, check_every=check_every)
    x, st = amg.solve(b, **kw)
    s = math.ldexp(1.0, exponent)
    y, st2 = amg.solve(b * s, **kw)
    assert st.converged and st2.converged
    assert abs(st2.iterations - st.iterations) <= 1
    assert torch.linalg.norm(y / s - x) <= 1e-8 * torch.linalg.norm(x)
