"""Weight and bias gradients whose batch is split into parts.

The weight products of all layers run side by side, batches above 4096 rows in
parts (chunks rounded up to 64 rows) that are added in order; bias gradients,
mask and loss are block sums. Checked against the FP64 oracle with the same bfloat16
operand rounding at the edges of a part and of a ragged last one, for a network
of two layers and one of ten (more than one launch of the products holds).
Tolerances: those of the four-layer network (loss 1e-4, every block 5e-3 of its
largest element; FP32 accumulation and activations that round to neighbouring
bfloat16 values, one contribution per layer), scaled with the layers beyond four.
"""
import numpy as np
import pytest

from oracle import mlp as omlp

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("nhidden", [1, 9])
@pytest.mark.parametrize("batch", [1, 17, 129, 300, 4096, 4097, 8300])
def test_split_gradients(batch, nhidden):
    from paper_0712_2247_gb300.mlp import MLP

    nin, hidden, nout = 7, 48, 37
    rng = np.random.default_rng(batch)
    net = MLP(nin, hidden, nhidden, nout, max_batch=batch, seed=2)
    X = rng.standard_normal((batch, nin)).astype(np.float32)
    T = rng.standard_normal((batch, nout)).astype(np.float32)
    M = (rng.random((batch, nout)) < 0.7).astype(np.float32)
    p = net.get_params().astype(np.float64)
    shapes = omlp.layer_shapes(nin, hidden, nhidden, nout)
    ol, og = omlp.loss_and_grads(p, X, T, M, shapes, bf16=True)
    loss, g = net.gradients(X, T, M)
    depth = max(1.0, (nhidden + 1) / 4.0)
    assert abs(loss - ol) <= 1e-4 * depth * abs(ol)
    at = 0
    for o, i in shapes:
        for n in (o * i, o):
            d = np.abs(g[at:at + n] - og[at:at + n]).max()
            assert d <= 5e-3 * depth * np.abs(og[at:at + n]).max(), (n, d)
            at += n
    # the training step uses the same gradients: Adam's first step from them
    want, _, _ = omlp.adam_step(p, g.astype(np.float64), np.zeros(len(p)), np.zeros(len(p)), 1, 1e-3)
    net.train_step(X, T, M, lr=1e-3)
    assert np.abs(net.get_params() - want).max() <= 1e-6
    net.close()
