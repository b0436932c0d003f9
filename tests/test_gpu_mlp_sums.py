"""Range and bits of the training call's sums: mask, loss and bias gradients.

They are FP64 sums of FP32 values (the loss of FP64 squares). With all parameters
zero the outputs are exactly zero, so the output error is d = 2 mask (0 - T) /
sum(mask), known on the host, and the last layer's bias gradient its column sum.
"""
import math

import numpy as np
import pytest

pytestmark = pytest.mark.gpu

NIN, HIDDEN, NOUT = 3, 16, 5


def network(batch):
    from paper_0712_2247_gb300.mlp import MLP

    net = MLP(NIN, HIDDEN, 1, NOUT, max_batch=batch)
    net.set_params(np.zeros(net.num_params, np.float32))
    return net


def call(T, M):
    net = network(len(T))
    loss, g = net.gradients(np.ones((len(T), NIN), np.float32), T, M)
    net.close()
    return loss, g[-NOUT:]


@pytest.mark.parametrize("batch", [1, 40, 700])
@pytest.mark.parametrize("size", [1e-30, 1e-18, 3.0, 1e19, 1e25])
def test_loss_range(size, batch):
    """Squares below and above the range of FP32: the error of a sum of n
    positive FP64 terms, each rounded once, stays below (n + 1) 2^-53."""
    rng = np.random.default_rng(batch)
    T = (size * rng.standard_normal((batch, NOUT))).astype(np.float32)
    M = np.ones_like(T)
    loss, gb = call(T, M)
    n = T.size
    want = math.fsum(float(t) ** 2 for t in T.ravel()) / n
    assert abs(loss - want) <= (n + 2) * 2.0 ** -53 * want
    d = (-2.0 * T.astype(np.float64) / n).astype(np.float32).astype(np.float64)
    for c in range(NOUT):
        s, a = math.fsum(d[:, c]), math.fsum(abs(d[:, c]))
        assert abs(gb[c] - s) <= 2.0 ** -24 * abs(s) + (batch + 2) * 2.0 ** -53 * a


def test_infinite_error_gives_an_infinite_loss():
    T = np.ones((100, NOUT), np.float32)
    T[37, 2] = np.inf
    loss, gb = call(T, np.ones_like(T))
    assert loss == np.inf
    assert gb[2] == -np.inf and np.isfinite(np.delete(gb, 2)).all()


def test_column_sum_keeps_fp64_bits():
    """Rows that one thread adds: 1, 1.5 2^-25, sixteen times 2^-51, then the
    first two again with the other sign. Every partial sum is an FP64 number."""
    d = np.zeros((1024, NOUT), np.float32)
    rows = 7 + 32 * np.arange(20)
    v = np.array([1.0, 1.5 * 2.0 ** -25] + [2.0 ** -51] * 16 + [-1.5 * 2.0 ** -25, -1.0])
    d[rows, 3] = v
    M = np.zeros_like(d)
    M[rows, 3] = 1.0
    M[rows[:12] + 1, 0] = 1.0  # mask sum 32, a power of two: T is exact
    loss, gb = call((-d * 16.0).astype(np.float32), M)
    assert gb[3] == 2.0 ** -47
    assert gb[0] == 0.0


def test_mask_sum_keeps_fp64_bits_and_range():
    """The same values as weights of one thread's elements (16,384 apart), and
    weights whose sum only FP64 holds."""
    step = 64 * 256
    batch = -(-20 * step // NOUT)
    v = [1.0, 1.5 * 2.0 ** -25] + [2.0 ** -51] * 16
    for w in (v, [3e38] * 18):
        M = np.zeros(batch * NOUT, np.float32)
        M[11 + step * np.arange(18)] = w
        M = M.reshape(batch, NOUT)
        T = np.zeros_like(M)
        k = 11 // NOUT, 11 % NOUT
        T[k] = 0.5
        loss, _ = call(T, M)
        e = 0.5 * float(M[k])
        want = e * e / math.fsum(float(x) for x in np.float32(w))
        assert abs(loss - want) <= 2.0 ** -52 * want


def test_error_scale_below_fp32_range():
    """2 / sum(mask) is no FP32 number with all its bits; the errors are."""
    T = np.full((64, NOUT), 2.0, np.float32)
    M = np.full_like(T, 2.0 ** 126)
    net = network(64)
    loss, g = net.gradients(np.ones((64, NIN), np.float32), T, M)
    net.close()
    d = np.float32(-2.0 * 2.0 * 2.0 ** 126 / (T.size * 2.0 ** 126))
    want = 64.0 * float(d)
    assert np.abs(g[-NOUT:] - want).max() <= 2.0 ** -24 * abs(want)
