"""GPU parity of the gradient kernels at the edges of their tiles.

* against the oracle storing the same values in bf16, per layer, at shapes
  around the tiles (4-row x 128-pixel jobs of the 32 -> 32 layers, 32-pixel
  segments and 128-pixel runs of layers 1 and 6): rel-L2 <= 2e-2, the bound of
  the larger parity test (what remains is FP32 against FP64 sums flipping a
  bf16 rounding);
* the gradient of a stack large enough for every CTA to empty its tensor-core
  accumulators several times equals the sum of its images' gradients: both are
  FP32 sums of the same products in another grouping, with chains of at most
  some 10^3 terms, so they agree to about 10^3 x 2^-24 = 6e-5 of the sums'
  norms (1e-4 asserted).
"""
import numpy as np
import pytest
import torch

from oracle import cnn as ocnn

pytestmark = pytest.mark.gpu


def _net(seed):
    import __graft_entry__ as ge
    import paper_2204_06083_gb300 as eb
    ge.build()
    rng = np.random.default_rng(seed + 1000)
    theta = ocnn.pack([(W, rng.uniform(-0.05, 0.05, size=b.shape)) for W, b in ocnn.unpack(ocnn.init_params(seed))])
    return eb.Net(theta), theta.astype(np.float32).astype(np.float64)


def _layers(g):
    offs = np.cumsum([0] + [w + b for w, b in ocnn.layer_sizes()])
    return [g[offs[l]:offs[l + 1]] for l in range(6)]


@pytest.mark.parametrize("shape", [(1, 1, 1), (3, 2, 3), (1, 4, 128), (1, 5, 129), (2, 7, 33), (2, 9, 127),
                                   (1, 3, 260)])
def test_gradient_at_tile_edges(shape):
    net, theta = _net(11)
    nimg, H, W = shape
    rng = np.random.default_rng(H * 1000 + W)
    s = rng.standard_normal((nimg, H, W)).astype(np.float32)
    m = (rng.random((nimg, H, W)) < 0.7).astype(np.float32)
    m[0, 0, 0] = 1.0
    dout = rng.standard_normal((nimg, H, W)).astype(np.float32)
    net.backward(torch.from_numpy(np.stack([s, m], axis=-1)).cuda(), torch.from_numpy(dout).cuda())
    net.status()
    g = net.params()[1].astype(np.float64)
    ref = np.zeros(ocnn.NPARAM)
    for k in range(nimg):
        _, cache = ocnn.forward(theta, s[k].astype(np.float64), m[k].astype(np.float64), storage="bf16")
        ref += ocnn.backward(theta, cache, dout[k].astype(np.float64))
    for l, (a, b) in enumerate(zip(_layers(g), _layers(ref))):
        assert np.linalg.norm(a - b) <= 2e-2 * np.linalg.norm(b), (l, np.linalg.norm(a - b), np.linalg.norm(b))


def test_gradient_of_a_stack_is_the_sum_of_its_images():
    net, _ = _net(12)
    n, H, W = 20, 301, 290  # 20 x 76 x 3 jobs: some 30 per CTA
    gen = torch.Generator(device="cuda").manual_seed(3)
    inp = torch.randn((n, H, W, 2), generator=gen, device="cuda")
    inp[..., 1] = (inp[..., 1] > -0.5).float()
    dout = torch.randn((n, H, W), generator=gen, device="cuda")
    net.backward(inp, dout)
    net.status()
    whole = net.params()[1].astype(np.float64)
    parts = np.zeros_like(whole)
    for k in range(n):
        net.backward(inp[k:k + 1].contiguous(), dout[k:k + 1].contiguous())
        parts += net.params()[1]
    net.status()
    for l, (a, b) in enumerate(zip(_layers(whole), _layers(parts))):
        assert np.linalg.norm(a - b) <= 1e-4 * np.linalg.norm(b), (l, np.linalg.norm(a - b), np.linalg.norm(b))
