"""GPU parity of the coarsest level's explicit inverse (symmetric block sweeps).

With one level the V-cycle is the inverse itself, so V r is compared with a
dense FP64 solve of the level's own matrix, at row counts around the block size
of 32: part of a block, a whole one, a few rows past one, many blocks with a
ragged last one.  Both
sides solve an SPD system backward stably, so they differ by at most
c n eps kappa with kappa <= 4 dim / lambda_min <= 1100 on these grids and c n
of order 10: 1e-11 holds with room.
"""
import numpy as np
import pytest
import torch

import eb_inputs as ei

pytestmark = pytest.mark.gpu


def _grid(dim, n, radius):
    return ei.box_grid(dim, n), ei.sphere((0.013, 0.007, 0.003)[:dim], radius)


# (dim, nodes per axis, radius in units of h) -> rows
CASES = [(2, 8, 1.7), (2, 12, 2.6), (2, 16, 3.3), (2, 16, 4.2), (2, 16, 4.6), (2, 20, 5.4), (2, 32, 10.3),
         (2, 40, 17.6), (3, 12, 3.7), (3, 16, 6.4)]


@pytest.mark.parametrize("dim,n,rh", CASES)
@pytest.mark.parametrize("shift", [0.0, 37.5])
def test_coarse_inverse_matches_dense_solve(dim, n, rh, shift):
    import __graft_entry__ as ge
    import paper_2204_06083_gb300 as eb
    ge.build()
    grid, ls = _grid(dim, n, rh * 2.0 / (n - 1))
    h = eb.EB(grid, ls)
    amg = eb.AMG(h, shift, max_levels=1)
    assert amg.num_levels == 1 and amg.rows[0] == h.info.num_cp
    rows = amg.rows[0]
    rp, ci, v = (t.cpu().numpy() for t in amg.level(0, 0))
    A = np.zeros((rows, rows))
    for i in range(rows):
        A[i, ci[rp[i]:rp[i + 1]]] = v[rp[i]:rp[i + 1]]
    nodes = h.cp_data()[0].cpu().numpy()
    rng = np.random.default_rng(rows)
    rc = rng.standard_normal(rows)
    r = np.zeros(grid.num_nodes)
    r[nodes] = rc
    z = amg.vcycle(torch.tensor(r, device="cuda").view(h.shape())).cpu().numpy().ravel()[nodes]
    ref = np.linalg.solve(A, rc)
    assert np.linalg.norm(z - ref) <= 1e-11 * np.linalg.norm(ref)
