"""FP32 leapfrog calls of one handle on several streams, and of several handles
from several threads: none waits for another, and the results are those of the
same calls one after another.
"""
import math
import threading

import pytest
import torch

import eb_inputs as ei

pytestmark = pytest.mark.gpu


def _handle(n):
    import __graft_entry__ as ge
    import paper_2204_06083_gb300 as eb
    ge.build()
    grid = ei.box_grid(2, n)
    h = eb.EB(grid, ei.sphere((0.0, 0.0), 0.6))
    cp = ((h.classes() & eb.CODE_CP) != 0).float()
    return h, 0.9 * grid.h / math.sqrt(2.0), cp


def _fields(h, cp, seed):
    gen = torch.Generator(device="cuda").manual_seed(seed)
    return [torch.randn(h.shape(), generator=gen, device="cuda") * cp for _ in range(2)]


LONG = 40000  # steps: thousands of launches, milliseconds of work behind the call's return


def test_short_run_does_not_wait_for_a_long_one_on_another_stream():
    h, dt, cp = _handle(514)
    a, b, c = (_fields(h, cp, s) for s in (1, 2, 3))
    want = [t.clone() for t in b]
    h.wave_step(c[0], c[1], dt, 64)  # the plan is there
    h.wave_step(want[0], want[1], dt, 40)
    torch.cuda.synchronize()
    s1, s2 = torch.cuda.Stream(), torch.cuda.Stream()
    long_done = torch.cuda.Event()
    h.wave_step(a[0], a[1], dt, LONG, stream=s1)
    long_done.record(s1)
    h.wave_step(b[0], b[1], dt, 40, stream=s2)
    s2.synchronize()
    assert not long_done.query()
    torch.cuda.synchronize()
    assert torch.equal(b[0], want[0]) and torch.equal(b[1], want[1])


def test_calls_of_two_handles_from_two_threads():
    h1, dt, cp = _handle(514)
    h2, _, _ = _handle(514)
    a, b, c = (_fields(h1, cp, s) for s in (1, 2, 3))
    for h in (h1, h2):
        h.wave_step(c[0], c[1], dt, 64)
    torch.cuda.synchronize()
    s1, s2 = torch.cuda.Stream(), torch.cuda.Stream()
    started = threading.Event()

    def long_run():
        started.set()
        h1.wave_step(a[0], a[1], dt, 10 * LONG, stream=s1)

    t = threading.Thread(target=long_run)
    t.start()
    started.wait()
    h2.wave_step(b[0], b[1], dt, 8, stream=s2)
    s2.synchronize()
    assert t.is_alive()  # the long run is still being enqueued
    t.join()
    torch.cuda.synchronize()


def test_one_handle_from_two_threads():
    h, dt, cp = _handle(386)
    base = [_fields(h, cp, s) for s in (1, 2)]
    want = [[t.clone() for t in f] for f in base]
    for f in want:
        for _ in range(30):
            h.wave_step(f[0], f[1], dt, 8)
    got = [[t.clone() for t in f] for f in base]
    streams = [torch.cuda.Stream() for _ in got]
    torch.cuda.synchronize()

    def runs(k):
        for _ in range(30):
            h.wave_step(got[k][0], got[k][1], dt, 8, stream=streams[k])

    ts = [threading.Thread(target=runs, args=(k,)) for k in range(2)]
    for t in ts:
        t.start()
    for t in ts:
        t.join()
    torch.cuda.synchronize()
    for f, w in zip(got, want):
        assert torch.equal(f[0], w[0]) and torch.equal(f[1], w[1])
