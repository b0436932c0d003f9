"""The fused forward's two forms and two ways to load its input.

Up to one tile of 128 rows per SM a CTA runs 16 warps, beyond that two CTAs of 8 share
an SM; input rows are loaded 16 bytes at a time where each starts on a 16-byte
boundary. No output bit may depend on either.
"""
import time

import numpy as np
import pytest

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("nin,hidden,nhidden,nout", [(4, 64, 2, 24), (8, 256, 2, 160), (256, 112, 1, 37), (20, 16, 3, 5)])
def test_alignment_and_tiles(nin, hidden, nhidden, nout):
    import torch

    from paper_0712_2247_gb300.mlp import MLP

    n = 128 * 153
    net = MLP(nin, hidden, nhidden, nout, max_batch=n, seed=3)
    g = torch.Generator(device="cuda").manual_seed(nin)
    flat = torch.randn(n * nin + 1, device="cuda", generator=g)
    X = flat[:n * nin].reshape(n, nin)
    Y = net.forward(X)
    # the same values one element on, where no row is aligned
    shifted = torch.empty(n * nin + 1, device="cuda")
    shifted[1:] = flat[:n * nin]
    assert torch.equal(net.forward(shifted[1:].reshape(n, nin)), Y)
    # fewer tiles: one per SM and less
    for a, b in ((0, 128 * 152), (0, 128 * 152 - 127), (128 * 152, n), (5, 6), (300, 433)):
        assert torch.equal(net.forward(X[a:b].contiguous()), Y[a:b])
    net.close()


def test_wide_inputs_cost_little_more():
    """512 rows, 256 inputs against 4 (one layer's weights more, 1.25 allowed): read
    four bytes at a time they took 1.36 times as long."""
    import torch

    from paper_0712_2247_gb300.mlp import MLP

    def us(nin):
        net = MLP(nin, 256, 3, 160, max_batch=512)
        X = torch.randn(512, nin, device="cuda")
        took = []
        for _ in range(40):
            t = time.perf_counter()
            net.forward(X)
            took.append(time.perf_counter() - t)
        net.close()
        return np.median(took) * 1e6

    assert us(256) < 1.25 * us(4)
