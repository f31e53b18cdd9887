"""Solves with the learned stage after the network's handle changed under a
hierarchy that has captured its iteration.

The captured iteration holds the network's workspace and forward path; a solve
after the workspace grew (a larger batch in between), after nn_set_fused, or
with another network (which may live at the address of a destroyed one) takes
them as they are then.  Direct launches (use_graph = 0) give the values; the
two agree bit for bit, as on a fresh handle.
"""
import numpy as np
import pytest
import torch

import eb_inputs as ei

pytestmark = pytest.mark.gpu


def _setup():
    import __graft_entry__ as ge
    import paper_2204_06083_gb300 as eb
    from paper_2204_06083_gb300 import learned
    ge.build()
    grid, ls = ei.circle_k1(64)
    h = eb.EB(grid, ls)
    amg = eb.AMG(h, vcycle_prec=eb.EB_F32, coarse_max=30)
    bs = [torch.from_numpy(np.random.default_rng(k).standard_normal(h.shape())).cuda() for k in range(4)]
    return eb, learned, h, amg, bs


def _both(eb, amg, net, b, check_every):
    # check_every 1: the loop on the device; 2: captured runs of two iterations
    use = 1 if check_every == 1 else 2
    kw = dict(rtol=1e-10, maxit=200, mode=eb.EB_NN_ENERGY, check_every=check_every)
    x, st = eb.solve_nn(amg, net, b, use_graph=use, **kw)
    y, sd = eb.solve_nn(amg, net, b, use_graph=0, **kw)
    assert st.converged and sd.converged
    assert torch.equal(x, y)
    return st


@pytest.mark.parametrize("check_every", [1, 2])
def test_workspace_grows_between_solves(check_every):
    eb, learned, h, amg, bs = _setup()
    net = eb.Net(learned.init_params(3))
    _both(eb, amg, net, bs[0], check_every)
    inp = torch.randn((3, 70, 90, 2), device="cuda")
    net.backward(inp, torch.randn((3, 70, 90), device="cuda"))  # more pixels than the grid has nodes
    _both(eb, amg, net, bs[1], check_every)


@pytest.mark.parametrize("check_every", [1, 2])
def test_forward_path_changes_between_solves(check_every):
    eb, learned, h, amg, bs = _setup()
    net = eb.Net(learned.init_params(3))
    _both(eb, amg, net, bs[0], check_every)
    net.set_fused(False)
    layered = _both(eb, amg, net, bs[1], check_every)
    fresh = eb.AMG(h, vcycle_prec=eb.EB_F32, coarse_max=30)
    want = _both(eb, fresh, net, bs[1], check_every)
    assert layered.iterations == want.iterations and layered.launches == want.launches


@pytest.mark.parametrize("check_every", [1, 2])
def test_networks_that_follow_one_another(check_every):
    eb, learned, h, amg, bs = _setup()
    for k in range(4):
        net = eb.Net(learned.init_params(k, last_scale=0.1 * k))
        _both(eb, amg, net, bs[k], check_every)
        net.close()
