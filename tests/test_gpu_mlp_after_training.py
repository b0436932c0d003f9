"""The copies of the weights after training.

Inference reads packed bfloat16 weights, the training products two other layouts of
them; Adam's kernel updates all three beside the FP32 parameters. After some steps
a second network that is given the trained parameters must predict, and compute
gradients, with the same bits. Ragged widths (chunks of the packed copy that end
short, an output layer that is no multiple of 16) and more layers than one launch
of the update holds.
"""
import numpy as np
import pytest

from oracle import mlp as omlp

pytestmark = pytest.mark.gpu

WIDTHS = [(4, 256, 3, 160), (1, 16, 1, 1), (17, 48, 2, 37), (40, 112, 5, 130), (256, 240, 1, 256), (7, 48, 9, 37)]


def data(nin, nout, batch, seed):
    rng = np.random.default_rng(seed)
    X = rng.standard_normal((batch, nin)).astype(np.float32)
    T = rng.standard_normal((batch, nout)).astype(np.float32)
    M = (rng.random((batch, nout)) < 0.8).astype(np.float32)
    return X, T, M


@pytest.mark.parametrize("nin,hidden,nhidden,nout", WIDTHS)
@pytest.mark.parametrize("batch", [33, 300])
def test_trained_network_equals_its_parameters(nin, hidden, nhidden, nout, batch):
    from paper_0712_2247_gb300.mlp import MLP

    a = MLP(nin, hidden, nhidden, nout, max_batch=batch, seed=1)
    for k in range(5):
        a.train_step(*data(nin, nout, batch, k), lr=2e-3)
    p = a.get_params()
    b = MLP(nin, hidden, nhidden, nout, max_batch=batch, seed=2)
    assert not np.array_equal(p, b.get_params())
    b.set_params(p)
    X, T, M = data(nin, nout, batch, 99)
    assert np.array_equal(a.forward(X), b.forward(X))
    (la, ga), (lb, gb) = a.gradients(X, T, M), b.gradients(X, T, M)
    assert la == lb and np.array_equal(ga, gb)
    a.close()
    b.close()


@pytest.mark.parametrize("nin,hidden,nhidden,nout", WIDTHS)
def test_three_adam_steps(nin, hidden, nhidden, nout):
    """Against FP64 Adam fed with the device's gradients. Per step the parameter is
    rounded once (2^-24 of it) and the update, lr times a ratio below 3, carries
    about ten FP32 roundings."""
    from paper_0712_2247_gb300.mlp import MLP

    lr, batch = 1e-3, 65
    net = MLP(nin, hidden, nhidden, nout, max_batch=batch, seed=4)
    p = net.get_params().astype(np.float64)
    m, v = np.zeros_like(p), np.zeros_like(p)
    b1, b2 = float(np.float32(0.9)), float(np.float32(0.999))
    tol = 0.0
    for t in (1, 2, 3):
        X, T, M = data(nin, nout, batch, 10 + t)
        _, g = net.gradients(X, T, M)
        net.train_step(X, T, M, lr=lr)
        p, m, v = omlp.adam_step(p, g.astype(np.float64), m, v, t, float(np.float32(lr)), b1, b2,
                                 float(np.float32(1e-8)))
        tol += 2.0 ** -24 * np.abs(p).max() + lr * 3 * 10 * 2.0 ** -24
        assert np.abs(net.get_params() - p).max() <= tol
    net.close()
