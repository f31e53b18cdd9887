"""Sparse products of the hierarchy whose rows span few and many columns.

The products keep a bitmap of a row's column range in shared memory: a small one
(16,384 columns) while every row fits, a large one otherwise.  Long thin ellipses
take rows across the line.  Every coarse matrix equals P' (A P) of the level's own
matrices: the same structure, values to 1e-13 of the row's largest (a few ulp).
"""
import numpy as np
import pytest
import scipy.sparse as sp

import eb_inputs as ei

pytestmark = pytest.mark.gpu


def _csr(arrays, n, m):
    rp, ci, v = (t.cpu().numpy() for t in arrays)
    return sp.csr_matrix((v, ci, rp), shape=(n, m))


@pytest.mark.parametrize("n0,n1,large", [(9000, 60, False), (16000, 60, True)])
def test_products_of_a_long_domain(n0, n1, large):
    import __graft_entry__ as ge
    import paper_2204_06083_gb300 as eb
    ge.build()
    h = 2.0 / (n0 - 1)
    grid = ei.Grid(dim=2, n=(n0, n1, 1), lo=(-1.0, -0.5 * h * (n1 - 1), 0.0), h=h)
    ls = ei.ellipsoid((0.0, 0.0), (0.98, 0.47 * h * (n1 - 1)), np.eye(3))
    amg = eb.AMG(eb.EB(grid, ls))
    assert amg.num_levels > 2
    widest = 0
    for l in range(amg.num_levels - 1):
        n, m = amg.rows[l], amg.rows[l + 1]
        A, P, C = _csr(amg.level(l, 0), n, n), _csr(amg.level(l, 1), n, m), _csr(amg.level(l + 1, 0), m, m)
        R = (P.T.tocsr() @ (A @ P)).tocsr()
        R.sort_indices()
        assert np.array_equal(C.indptr, R.indptr) and np.array_equal(C.indices, R.indices)
        scale = np.repeat(np.maximum.reduceat(np.abs(R.data), R.indptr[:-1]), np.diff(R.indptr))
        assert np.all(np.abs(C.data - R.data) <= 1e-13 * scale)
        widest = max(widest, int((R.indices[R.indptr[1:] - 1] - R.indices[R.indptr[:-1]] + 1).max()))
    assert (widest > 16384) == large
