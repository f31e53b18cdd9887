"""Cut points of stars with few and many cuts and 1 to 8 harmonics.

Up to 16 cuts per multiprocessor eight lanes share a root's harmonics, up to 32
four; beyond that a lane does a root alone.  The boundary point of every cut satisfies psi = 0 to
1e-13: the iteration ends on steps of 1e-15 h, the slope of psi is below 4, and an
evaluation of O(1) terms rounds to a few 1e-16.
"""
import numpy as np
import pytest

import eb_inputs as ei

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("nk", [1, 2, 3, 4, 5, 8])
@pytest.mark.parametrize("n,most", [(66, 16), (514, 16), (1800, 32), (3600, 1000)])
def test_star_roots(n, most, nk):
    import torch
    import __graft_entry__ as ge
    import paper_2204_06083_gb300 as eb
    ge.build()
    rng = np.random.default_rng(100 + nk)
    ks = list(range(2, 2 + nk))
    amps, ph = rng.uniform(0.0, 0.03, nk), rng.uniform(0.0, 6.0, nk)
    c = (0.02, 0.01)
    h = eb.EB(ei.box_grid(2, n), ei.star(c, 0.5, ks, list(amps), list(ph)))
    sms = torch.cuda.get_device_properties(0).multi_processor_count
    least = {16: 0, 32: 16, 1000: 32}[most]
    assert least * sms < h.info.num_cut <= most * sms
    xg = h.cuts()[3].cpu().numpy().reshape(-1, 2)
    phi = np.arctan2(xg[:, 1] - c[1], xg[:, 0] - c[0])
    r = 0.5 + sum(a * np.sin(k * phi + p) for k, a, p in zip(ks, amps, ph))
    assert np.abs(np.hypot(xg[:, 0] - c[0], xg[:, 1] - c[1]) - r).max() <= 1e-13
