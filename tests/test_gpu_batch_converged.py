"""Batches whose geometries converge many iterations apart, in double-float.

A nearly explicit step (dt = 1e-7), an ordinary one and a steady problem (dt
infinite) in one batch, at smoother degrees 1 to 6 with FP32 and BF16 V-cycles:
the iterations that only the last one needs leave the others as they are, and
each takes the iterations of the FP64 outer iteration (within one, the bound of
the existing comparison of the two).  Solutions to rtol 1e-11 against a sparse LU
of the oracle's matrices: kappa of the steady problem is some 1e3, so 1e-8.
"""
import numpy as np
import pytest
import scipy.sparse.linalg as spla
import torch

import eb_inputs as ei
from oracle import eb as oeb

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("vprec", ["EB_F32", "EB_BF16"])
@pytest.mark.parametrize("degree", [1, 2, 3, 6])
def test_early_converged_geometries(vprec, degree):
    import __graft_entry__ as ge
    import paper_2204_06083_gb300 as eb
    ge.build()
    sizes, dts = (96, 64, 130), (1e-7, 0.01, float("inf"))
    grids, lss = [ei.box_grid(2, n) for n in sizes], [ei.random_star(40 + n) for n in sizes]
    B = eb.Batch(grids, lss)
    B.heat_setup(dts, theta=1.0, vcycle_prec=getattr(eb, vprec), cheb_degree=degree, coarse_max=30)
    gen = torch.Generator(device="cuda").manual_seed(degree)
    b1 = torch.randn(B.num_nodes, generator=gen, device="cuda", dtype=torch.float64)
    its = {}
    for outer in (eb.EB_F64, eb.EB_DF64):
        B.set_outer(outer)
        for _ in range(2):  # the second step starts from buffers that a finished solve left
            u = B.zeros()
            st = B.heat_step(u, b1, rtol=1e-11)
            assert all(s.converged for s in st)
            its[outer] = [s.iterations for s in st]
            assert torch.isfinite(u).all()
    assert all(abs(a - b) <= 1 for a, b in zip(its[eb.EB_F64], its[eb.EB_DF64])), its
    it = its[eb.EB_DF64]
    assert it[0] < it[1] < it[2] and it[0] + 5 <= it[2], it
    for g, (gr, ls) in enumerate(zip(grids, lss)):
        r = oeb.build(gr, ls)
        A = oeb.assemble_unit(r, 0.0 if np.isinf(dts[g]) else gr.h ** 2 / dts[g]).tocsc()
        want = spla.spsolve(A, gr.h ** 2 * r.from_grid(B.view(b1, g).cpu().numpy()))
        got = r.from_grid(B.view(u, g).cpu().numpy())
        assert np.linalg.norm(got - want) <= 1e-8 * np.linalg.norm(want)
