"""Solves that alternate between solution vectors, and grids around the sizes
where the list kernels change their CTA size.

The captured iteration takes the solution vector's address from the solver's
scalars, so one capture serves every vector: solving into several buffers in
turn gives the same values as a fresh solver, on FP64 and double-float outer
iterations, single and batched.  Solutions are checked against the residual of
the oracle's matrix at every size (128: CTAs of 64 threads; 400: 256)."""
import numpy as np
import pytest
import torch

import eb_inputs as ei
from oracle import eb as oeb

pytestmark = pytest.mark.gpu


def _pkg():
    import __graft_entry__ as ge
    import paper_2204_06083_gb300 as eb
    ge.build()
    return eb


@pytest.mark.parametrize("n", [24, 128, 400])
@pytest.mark.parametrize("vprec,outer", [("EB_F64", "EB_F64"), ("EB_F32", "EB_F64"), ("EB_F32", "EB_DF64")])
def test_solves_into_alternating_vectors(n, vprec, outer):
    eb = _pkg()
    grid, ls = ei.circle_k1(n)
    ref = oeb.build(grid, ls)
    h = eb.EB(grid, ls)
    amg = eb.AMG(h, vcycle_prec=getattr(eb, vprec), coarse_max=30)
    rng = np.random.default_rng(n)
    bs = [torch.tensor(ref.to_grid(rng.standard_normal(ref.num_cp)), device="cuda") for _ in range(2)]
    bufs = [torch.zeros_like(bs[0]) for _ in range(3)]
    for k in range(6):
        b, x = bs[k % 2], bufs[k % 3]
        x.zero_()
        amg.solve(b, x, rtol=1e-11, outer=getattr(eb, outer))
        fresh = eb.AMG(h, vcycle_prec=getattr(eb, vprec), coarse_max=30)
        want, _ = fresh.solve(b, rtol=1e-11, outer=getattr(eb, outer))
        assert torch.equal(x, want)
        r = ref.from_grid(b.cpu().numpy()) - ref.A @ ref.from_grid(x.cpu().numpy())
        assert np.linalg.norm(r) <= 2e-11 * np.linalg.norm(ref.from_grid(b.cpu().numpy()))


@pytest.mark.parametrize("outer", ["EB_F64", "EB_DF64"])
def test_batched_steps_into_alternating_vectors(outer):
    eb = _pkg()
    sizes = [(n, ei.random_star(n)) for n in (64, 130, 200)]
    grids = [ei.box_grid(2, n) for n, _ in sizes]
    b = eb.Batch(grids, [l for _, l in sizes])
    b.heat_setup([g.h for g in grids], vcycle_prec=eb.EB_F32, coarse_max=30)
    b.set_outer(getattr(eb, outer))
    gen = torch.Generator(device="cuda").manual_seed(1)
    b1 = torch.randn(b.num_nodes, generator=gen, device="cuda", dtype=torch.float64)
    want = None
    for _ in range(2):
        us = [b.zeros() for _ in range(2)]
        for u in us:
            b.heat_step(u, b1, rtol=1e-11)
            want = u.clone() if want is None else want
            assert torch.equal(u, want)
