"""The one-launch network forward where a thread block walks several work units.

More units (strips x row runs x images) than multiprocessors: the accumulator
slots, the activation rings and the barriers go on from one unit to the next.
Odd and even numbers of steps per unit (layer 1 takes steps in pairs), one and
two strips, ragged widths.  Bit-identical to the layer-by-layer launches, which
do the same arithmetic in the same order.
"""
import numpy as np
import pytest
import torch

from oracle import cnn as ocnn

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("shape", [(200, 5, 120), (330, 4, 30), (500, 1, 116), (170, 8, 117), (310, 3, 233)])
def test_units_in_turn(shape):
    import __graft_entry__ as ge
    import paper_2204_06083_gb300 as eb
    ge.build()
    rng = np.random.default_rng(sum(shape))
    s = rng.standard_normal(shape)
    m = (rng.random(shape) < 0.6).astype(np.float64)
    inp = torch.from_numpy(np.stack([s, m], axis=-1).astype(np.float32)).cuda()
    layers = [(W, rng.uniform(-0.05, 0.05, size=b.shape)) for W, b in ocnn.unpack(ocnn.init_params(7))]
    net = eb.Net(ocnn.pack(layers))
    net.set_fused(True)
    fused = net.forward(inp).clone()
    net.status()
    net.set_fused(False)
    assert torch.equal(fused, net.forward(inp))
