"""A network on a non-blocking stream of the caller's.

Creation fills its buffers with zeros on the default stream, which such a stream does
not wait for; the parameters written right after it must survive.
"""
import numpy as np
import pytest

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("batch", [64, 200000])
def test_parameters_survive_creation(batch):
    import torch

    from paper_0712_2247_gb300.mlp import MLP

    rng = np.random.default_rng(0)
    X = rng.standard_normal((64, 4)).astype(np.float32)
    T, M = np.zeros((64, 160), np.float32), np.ones((64, 160), np.float32)
    a = MLP(max_batch=64, seed=7)
    for _ in range(3):
        s = torch.cuda.Stream()
        b = MLP(max_batch=batch, seed=7, stream=s.cuda_stream)
        assert np.array_equal(a.get_params(), b.get_params())
        assert np.array_equal(a.forward(X), b.forward(X))
        assert np.array_equal(a.gradients(X, T, M)[1], b.gradients(X, T, M)[1])
        b.close()
    a.close()
