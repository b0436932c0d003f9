"""Thin grids, whose padded fields are many times their nodes, step without overlap.

Kernels that come up early take places on the SMs that their predecessor still needs:
a step took up to 2.5 times the sum of its kernels' times there. Steps in a row may take
1.2 times that sum (measured with events between the launches).
"""
import time

import numpy as np
import pytest

pytestmark = pytest.mark.gpu


def kernels_us(g):
    return min(sum(g.step_profiled(20)[0].values()) for _ in range(5)) / 20 * 1e3


@pytest.mark.parametrize("n,sigma", [((1, 1, 20000), 4), ((1, 5, 4000), 8), ((1, 300, 100), 12), ((9, 190, 39), 10)])
def test_slit(n, sigma):
    from paper_0712_2247_gb300 import lbif

    with lbif.Slit(*n, sigma, 0.15, 0.9) as g:
        g.step(20)
        took = []
        for _ in range(5):
            g.status()
            t = time.perf_counter()
            g.step(100)
            g.status()
            took.append((time.perf_counter() - t) / 100 * 1e6)
        assert min(took) < 1.2 * kernels_us(g)


def test_ensemble():
    from paper_0712_2247_gb300 import lbif

    m = 400
    H = np.random.default_rng(3).integers(4, 80, m)
    one = np.ones(m)
    with lbif.Ensemble(H, 0.15 * one, 1e-6 * one, 0.9 * one, 4, 1, 1, storage=0) as e:
        took = []
        for _ in range(5):
            t = time.perf_counter()
            e.run(tol=1e-30, max_steps=200, check_every=100)
            took.append((time.perf_counter() - t) / 200 * 1e6)
        assert min(took[1:]) < 1.2 * kernels_us(e)
