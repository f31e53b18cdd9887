"""Reduced-precision V-cycles with merged transfers against the FP64 V-cycle.

FP32 V-cycles prolongate with the first post-smoothing step in one launch and
restrict without waiting for the residual; FP64 V-cycles take them one by one.
The two agree to the FP32 rounding of some 30 operations on O(1) numbers per
level, 1e-5 of the result's norm (the bound of the larger FP32 parity test), on
hierarchies of several levels, V- and W-cycles, every smoother degree (degree 1
has no merged level 0), both coarsenings, a variable coefficient and a shift.
"""
import numpy as np
import pytest
import torch

import eb_inputs as ei

pytestmark = pytest.mark.gpu

CASES = [(2, 66, dict()), (2, 130, dict(cheb_degree=1)), (2, 130, dict(cheb_degree=3)), (2, 200, dict(cycle=2)),
         (2, 130, dict(coarsening=1)), (2, 130, dict(coarsening=1, cycle=2)), (3, 28, dict()),
         (3, 40, dict(cheb_degree=3)), (2, 160, dict(beta=True)), (2, 160, dict(shift=400.0))]


@pytest.mark.parametrize("dim,n,opts", CASES)
def test_fp32_cycle_with_merged_transfers(dim, n, opts):
    import __graft_entry__ as ge
    import paper_2204_06083_gb300 as eb
    ge.build()
    opts = dict(opts)
    beta, shift = opts.pop("beta", False), opts.pop("shift", 0.0)
    grid, ls = ei.circle_k1(n) if dim == 2 else ei.ellipsoid_k3(n)
    h = eb.EB(grid, ls)
    if beta:
        h.set_beta(ei.beta_half_points(grid, ei.beta_bone))
    a64 = eb.AMG(h, shift, coarse_max=12, **opts)
    a32 = eb.AMG(h, shift, coarse_max=12, vcycle_prec=eb.EB_F32, **opts)
    assert a64.num_levels == a32.num_levels and (a64.num_levels > 2 or n < 40)
    gen = torch.Generator(device="cuda").manual_seed(n)
    cp = (h.classes() & eb.CODE_CP) != 0
    r = torch.randn(h.shape(), generator=gen, device="cuda", dtype=torch.float64) * cp
    z64, z32 = a64.vcycle(r), a32.vcycle(r)
    err = float(torch.linalg.norm(z32 - z64) / torch.linalg.norm(z64))
    assert err <= 1e-5, err
    assert torch.equal(z32[~cp], torch.zeros_like(z32[~cp]))
