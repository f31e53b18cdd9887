"""BF16 V-cycles with merged transfers against the FP64 V-cycle.

The products A P of the merged launches are rounded once more to BF16, and the
restriction forms P'b - (A P)'x, a difference, with them.  The cycle stays within
the 3e-2 of the FP64 one that the whole-cycle comparison allows, on hierarchies of
several levels, V- and W-cycles, every smoother degree, both coarsenings, a
variable coefficient and a shift, for noise and for a smooth right-hand side,
whose differences cancel most; and solves take at most 2 iterations more than
twice those of the FP64 cycle.
"""
import pytest
import torch

import eb_inputs as ei

pytestmark = pytest.mark.gpu

CASES = [(2, 66, dict()), (2, 130, dict(cheb_degree=1)), (2, 130, dict(cheb_degree=3)), (2, 200, dict(cycle=2)),
         (2, 130, dict(coarsening=1)), (2, 130, dict(coarsening=1, cycle=2)), (3, 40, dict(cheb_degree=3)),
         (3, 64, dict()), (2, 160, dict(beta=True)), (2, 160, dict(shift=400.0)), (2, 514, dict())]


@pytest.mark.parametrize("dim,n,opts", CASES)
def test_bf16_cycle_with_merged_transfers(dim, n, opts):
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
    a16 = eb.AMG(h, shift, coarse_max=12, vcycle_prec=eb.EB_BF16, **opts)
    assert a64.num_levels == a16.num_levels
    gen = torch.Generator(device="cuda").manual_seed(n)
    cp = (h.classes() & eb.CODE_CP) != 0
    noise = torch.randn(h.shape(), generator=gen, device="cuda", dtype=torch.float64) * cp
    for r in (noise, cp.double()):
        z64, z16 = a64.vcycle(r), a16.vcycle(r)
        err = float(torch.linalg.norm(z16 - z64) / torch.linalg.norm(z64))
        assert err <= 3e-2, err
        assert torch.equal(z16[~cp], torch.zeros_like(z16[~cp]))
        x64, s64 = a64.solve(r, rtol=1e-10)
        x16, s16 = a16.solve(r, rtol=1e-10)
        assert s16.converged and s16.iterations <= 2 * s64.iterations + 2
