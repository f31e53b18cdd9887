"""FP32 leapfrog steps taken several per launch, on handles that have their plan,
against one step per launch: equal fields (a zero's sign may differ).

Every number of steps per launch on small grids, and grids whose tasks are long
(20 and 40 rows, the most a task takes) and more than the warps of a launch, so
that a warp's rings start anew over another task's rows; widths that are and are
not multiples of 4.  A handle's first short calls, which have no plan, agree too.
"""
import ctypes as C
import math

import pytest
import torch

import eb_inputs as ei

pytestmark = pytest.mark.gpu


def _handle(n0, n1, radius):
    import __graft_entry__ as ge
    import paper_2204_06083_gb300 as eb
    ge.build()
    g = ei.box_grid(2, n0)
    grid = ei.Grid(dim=2, n=(n0, n1, 1), lo=(-1.0, -0.5 * g.h * (n1 - 1), 0.0), h=g.h)
    return eb, eb.EB(grid, ei.sphere((0.0, 0.0), radius)), 0.9 * grid.h / math.sqrt(2.0)


def _compare(eb, h, dt, nsteps, seed):
    gen = torch.Generator(device="cuda").manual_seed(seed)
    a = [torch.randn(h.shape(), generator=gen, device="cuda") for _ in range(2)]
    b = [t.clone() for t in a]
    h.wave_step(a[0], a[1], dt, nsteps)
    stream = C.c_void_p(torch.cuda.current_stream().cuda_stream)
    rc = eb.load().wave_step_noalloc(h.handle, eb.EB_F32, C.c_double(dt), C.c_void_p(b[0].data_ptr()),
                                     C.c_void_p(b[1].data_ptr()), nsteps, stream)
    assert rc == eb.EB_OK
    torch.cuda.synchronize()
    assert torch.isfinite(a[1]).all()
    assert torch.equal(a[0], b[0]) and torch.equal(a[1], b[1])


SMALL = [(16, 16, 0.5), (114, 112, 0.6), (130, 127, 0.7), (340, 337, 0.7), (66, 66, 0.965), (128, 128, 0.98)]
LARGE = [(2050, 2041, 0.9), (5800, 5790, 0.95), (5802, 5799, 0.95)]


@pytest.mark.parametrize("n0,n1,radius", SMALL)
def test_every_number_of_steps(n0, n1, radius):
    eb, h, dt = _handle(n0, n1, radius)
    _compare(eb, h, dt, 64, 1)
    for nsteps in list(range(1, 18)) + [23, 24, 25]:
        _compare(eb, h, dt, nsteps, nsteps)


@pytest.mark.parametrize("n0,n1,radius", LARGE)
def test_long_tasks(n0, n1, radius):
    eb, h, dt = _handle(n0, n1, radius)
    for nsteps in (33, 3, 9, 16):
        _compare(eb, h, dt, nsteps, nsteps)


def test_first_calls_of_a_handle():
    eb, h, dt = _handle(340, 337, 0.7)
    for nsteps in (5, 8, 8, 8, 8, 8, 5):  # the fifth brings the plan
        _compare(eb, h, dt, nsteps, nsteps)
