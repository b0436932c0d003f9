"""The fused forward equals the layer-by-layer products of a training call.

Inference runs all layers of 128 rows in one CTA, training one product per
launch with the same operands in the same order, so the loss computed from the
training forward and from the fused outputs must agree to rounding, and the
outputs match the FP64 oracle with the same bfloat16 operands. Edges: one row,
a ragged last tile, more tiles than resident CTAs, widths that fill less than a
weight chunk, one to five hidden layers, misaligned output rows.
"""
import numpy as np
import pytest

from oracle import mlp as omlp

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("nin,hidden,nhidden,nout", [
    (4, 256, 3, 160), (1, 16, 1, 1), (17, 48, 2, 37), (40, 112, 5, 130), (256, 240, 1, 256), (33, 256, 1, 16)])
@pytest.mark.parametrize("batch", [1, 31, 33, 128, 129, 640])
def test_fused_forward(nin, hidden, nhidden, nout, batch):
    from paper_0712_2247_gb300.mlp import MLP

    rng = np.random.default_rng(nin + batch)
    net = MLP(nin, hidden, nhidden, nout, max_batch=batch, seed=3)
    p = net.get_params()
    p += (0.05 * rng.standard_normal(p.size)).astype(np.float32)
    net.set_params(p)
    X = rng.standard_normal((batch, nin)).astype(np.float32)
    Y = net.forward(X)
    shapes = omlp.layer_shapes(nin, hidden, nhidden, nout)
    Yo, _ = omlp.forward(p.astype(np.float64), X, shapes, bf16=True)
    # activations that round to neighbouring bfloat16 values, one contribution per layer
    tol = 2e-3 * max(1.0, (nhidden + 1) / 4.0)
    assert np.abs(Y - Yo).max() <= tol * np.abs(Yo).max()
    T = np.zeros((batch, nout), np.float32)
    M = np.ones((batch, nout), np.float32)
    loss, _ = net.gradients(X, T, M)
    assert abs(loss - (Y.astype(np.float64) ** 2).mean()) <= 1e-6 * loss
    net.close()


def test_many_tiles():
    """More row tiles than CTAs run at once: every tile equals the rows alone."""
    from paper_0712_2247_gb300.mlp import MLP

    rng = np.random.default_rng(0)
    n = 128 * 700 + 5
    net = MLP(4, 64, 2, 24, max_batch=n, seed=3)
    X = rng.standard_normal((n, 4)).astype(np.float32)
    Y = net.forward(X)
    for a in (0, 128 * 303, 128 * 304, 128 * 650, n - 133):
        assert np.array_equal(net.forward(X[a:a + 133]), Y[a:a + 133])
    net.close()
