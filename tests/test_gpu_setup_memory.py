"""Peak device memory of a hierarchy's set-up.

The products A_l P_l are the largest matrices of a set-up and most are needed
for one Galerkin product only.  Above what the finished hierarchy holds, the
peak (the memory pool's high-water mark) is at most the largest such product, or
with a reduced-precision V-cycle the sum of those that merged transfers are made
of, if that is larger: level 0's is not among them in 3D.
"""
import ctypes as C

import pytest
import scipy.sparse as sp
import torch

import eb_inputs as ei

pytestmark = pytest.mark.gpu

USED_CURRENT, USED_HIGH = 7, 8  # CUmemPool_attribute


def _pool():
    cu = C.CDLL("libcuda.so.1")
    pool = C.c_void_p()
    assert cu.cuDeviceGetDefaultMemPool(C.byref(pool), torch.cuda.current_device()) == 0

    def get(attr):
        v = C.c_uint64()
        assert cu.cuMemPoolGetAttribute(pool, attr, C.byref(v)) == 0
        return v.value

    def reset():
        torch.cuda.synchronize()
        zero = C.c_uint64(0)
        assert cu.cuMemPoolSetAttribute(pool, USED_HIGH, C.byref(zero)) == 0

    return get, reset


@pytest.mark.parametrize("vprec", ["EB_F64", "EB_F32", "EB_BF16"])
def test_products_are_not_kept(vprec):
    import __graft_entry__ as ge
    import paper_2204_06083_gb300 as eb
    ge.build()
    grid, ls = ei.ellipsoid_k3(160)
    h = eb.EB(grid, ls)
    get, reset = _pool()
    torch.cuda.synchronize()
    before = get(USED_CURRENT)
    reset()
    amg = eb.AMG(h, vcycle_prec=getattr(eb, vprec), coarse_max=200)
    torch.cuda.synchronize()
    held, peak = get(USED_CURRENT) - before, get(USED_HIGH) - before

    def csr(level, which, cols):
        rp, ci, _ = (t.cpu().numpy() for t in amg.level(level, which))
        return sp.csr_matrix(([1] * len(ci), ci, rp), shape=(len(rp) - 1, cols))

    products = []  # bytes of A_l P_l: row pointers, column indices, FP64 values
    for l in range(amg.num_levels - 1):
        A, P = csr(l, 0, amg.rows[l]), csr(l, 1, amg.rows[l + 1])
        products.append(12 * (A @ P).nnz + 4 * (A.shape[0] + 1))
    assert len(products) >= 2 and sum(products[1:]) > 2 ** 21
    kept = 0 if vprec == "EB_F64" else sum(products[1:])
    slack = 2 ** 20  # allocation granularity, the flags and counters of a level
    assert peak - held <= max(max(products), kept) + slack, (peak, held, products)
