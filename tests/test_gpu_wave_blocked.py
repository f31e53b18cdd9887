"""FP32 leapfrog steps taken several per launch, against one step per launch.

wave_step runs 2D FP32 steps eight per launch; wave_step_noalloc takes them one
by one with the same arithmetic per node, so the fields agree exactly (equal
values; a zero's sign may differ).  Sizes around the strips (112 written
columns, 8 halo columns) and rows beyond the grid's edges, widths that are and
are not multiples of 4, every number of steps per launch, domains that touch
several strips or lie in one, and values off the CPs that must be ignored.
"""
import math

import pytest
import torch

import eb_inputs as ei

pytestmark = pytest.mark.gpu


def _grid(n0, n1):
    g = ei.box_grid(2, n0)
    return ei.Grid(dim=2, n=(n0, n1, 1), lo=(-1.0, -0.5 * g.h * (n1 - 1), 0.0), h=g.h)


# the last two: a domain that reaches the second-outermost nodes (clamped rows and columns)
CASES = [(16, 16, 0.5), (64, 61, 0.5), (114, 112, 0.6), (130, 127, 0.7), (228, 225, 0.7), (340, 337, 0.7), (386, 381, 0.6),
         (66, 66, 0.965), (128, 128, 0.98)]


@pytest.mark.parametrize("n0,n1,radius", CASES)
@pytest.mark.parametrize("nsteps", [2, 3, 5, 7, 9, 11, 13, 15, 16, 17, 40])
def test_blocked_steps_match_single_steps(n0, n1, radius, nsteps):
    import __graft_entry__ as ge
    import ctypes as C
    import paper_2204_06083_gb300 as eb
    ge.build()
    grid = _grid(n0, n1)
    h = eb.EB(grid, ei.sphere((0.0, 0.0), radius))
    gen = torch.Generator(device="cuda").manual_seed(n0 + nsteps)
    u0 = torch.randn(h.shape(), generator=gen, device="cuda")
    u1 = torch.randn(h.shape(), generator=gen, device="cuda")
    a0, a1, b0, b1 = u0.clone(), u1.clone(), u0.clone(), u1.clone()
    dt = 0.9 * grid.h / math.sqrt(2.0)
    h.wave_step(a0, a1, dt, nsteps)
    stream = C.c_void_p(torch.cuda.current_stream().cuda_stream)
    rc = eb.load().wave_step_noalloc(h.handle, eb.EB_F32, C.c_double(dt), C.c_void_p(b0.data_ptr()),
                                     C.c_void_p(b1.data_ptr()), nsteps, stream)
    assert rc == eb.EB_OK
    torch.cuda.synchronize()
    assert torch.isfinite(a1).all()
    assert torch.equal(a0, b0) and torch.equal(a1, b1)


def test_blocked_steps_on_two_streams_and_in_a_captured_graph():
    import __graft_entry__ as ge
    import paper_2204_06083_gb300 as eb
    ge.build()
    grid = _grid(386, 381)
    h = eb.EB(grid, ei.sphere((0.0, 0.0), 0.6))
    dt = 0.9 * grid.h / math.sqrt(2.0)
    cp = ((h.classes() & eb.CODE_CP) != 0).float()
    base = [torch.randn(h.shape(), device="cuda") * cp for _ in range(4)]
    want = [t.clone() for t in base]
    h.wave_step(want[0], want[1], dt, 24)
    h.wave_step(want[2], want[3], dt, 24)
    torch.cuda.synchronize()
    got = [t.clone() for t in base]
    s1, s2 = torch.cuda.Stream(), torch.cuda.Stream()
    torch.cuda.synchronize()
    for _ in range(3):  # both pairs in flight on streams of their own, the handle shared
        h.wave_step(got[0], got[1], dt, 8, stream=s1)
        h.wave_step(got[2], got[3], dt, 8, stream=s2)
    torch.cuda.synchronize()
    assert all(torch.equal(a, b) for a, b in zip(got, want))
    # during capture the steps are single launches, as before
    cap = [t.clone() for t in base[:2]]
    g = torch.cuda.CUDAGraph()
    side = torch.cuda.Stream()
    with torch.cuda.graph(g, stream=side):
        h.wave_step(cap[0], cap[1], dt, 12, stream=side)
    g.replay()
    g.replay()
    torch.cuda.synchronize()
    assert torch.equal(cap[0], want[0]) and torch.equal(cap[1], want[1])
