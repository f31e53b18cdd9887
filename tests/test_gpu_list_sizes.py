"""Applies and solves on grids just below and just above the size where the
kernels over the list of CP pairs change from CTAs of 64 threads to CTAs of 256.

The line lies at 256 pairs per SM; the grid sizes are searched for on the
device at hand and the side each lies on is asserted.  Applies against the
oracle's matrix (FP64 to 1e-14 of |A||x|, FP32 to 4e-7), solutions by its residual.
"""
import numpy as np
import pytest
import torch

import eb_inputs as ei
from oracle import eb as oeb

pytestmark = pytest.mark.gpu


def _pairs(eb, h):
    cp = (h.classes().view(-1, 2) & eb.CODE_CP) != 0
    return int(cp.any(dim=1).sum())


@pytest.fixture(scope="module")
def sides():
    """[(handle, oracle) just below the line, (handle, oracle) just above]"""
    import __graft_entry__ as ge
    import paper_2204_06083_gb300 as eb
    ge.build()
    line = 256 * torch.cuda.get_device_properties(0).multi_processor_count
    n, last = 400, None
    while True:
        h = eb.EB(*ei.circle_k1(n))
        if _pairs(eb, h) >= line:
            break
        last, n = h, n + 2
    below, above = _pairs(eb, last), _pairs(eb, h)
    assert below < line <= above and above - below < line // 50
    return eb, [(last, oeb.build(*ei.circle_k1(n - 2))), (h, oeb.build(*ei.circle_k1(n)))]


@pytest.mark.parametrize("side", [0, 1])
def test_apply(sides, side):
    eb, hs = sides
    h, ref = hs[side]
    v = np.random.default_rng(side).standard_normal(ref.num_cp)
    want, scale = ref.A @ v, abs(ref.A) @ abs(v)
    x = torch.tensor(ref.to_grid(v), device="cuda")
    got = ref.from_grid(h.apply(x).cpu().numpy())
    assert (np.abs(got - want) <= 1e-14 * scale).all()
    got = ref.from_grid(h.apply(x.float()).double().cpu().numpy())
    assert (np.abs(got - want) <= 4e-7 * scale).all()


@pytest.mark.parametrize("side", [0, 1])
@pytest.mark.parametrize("vprec,outer", [("EB_F64", "EB_F64"), ("EB_F32", "EB_F64"), ("EB_F32", "EB_DF64"),
                                         ("EB_BF16", "EB_DF64")])
def test_solve(sides, side, vprec, outer):
    eb, hs = sides
    h, ref = hs[side]
    amg = eb.AMG(h, vcycle_prec=getattr(eb, vprec))
    b = np.random.default_rng(side).standard_normal(ref.num_cp)
    for use_graph in (1, 0):
        x, st = amg.solve(torch.tensor(ref.to_grid(b), device="cuda"), rtol=1e-11, outer=getattr(eb, outer),
                          use_graph=use_graph)
        assert st.converged
        r = b - ref.A @ ref.from_grid(x.cpu().numpy())
        assert np.linalg.norm(r) <= 2e-11 * np.linalg.norm(b)


@pytest.mark.parametrize("side", [0, 1])
def test_jacobi_solve_of_the_shifted_operator(sides, side):
    eb, hs = sides
    h, ref = hs[side]
    sigma = 4000.0
    amg = eb.AMG(h, sigma)
    b = np.random.default_rng(side).standard_normal(ref.num_cp)
    x, st = amg.solve(torch.tensor(ref.to_grid(b), device="cuda"), rtol=1e-11, precond=eb.EB_PC_JACOBI)
    v = ref.from_grid(x.cpu().numpy())
    assert st.converged
    assert np.linalg.norm(b - ref.A @ v - sigma * v) <= 2e-11 * np.linalg.norm(b)
