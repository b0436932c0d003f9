"""Further chains of overlapping kernels: without the ball between force and pull
pass, FP32 in place, and steps replayed from a captured graph, each against
steps that the host waits for one by one.
"""
import numpy as np
import pytest

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def L():
    from paper_0712_2247_gb300 import build, lbif

    build.build()
    return lbif


@pytest.mark.parametrize("kw", [dict(hs=False), dict(hs=False, inplace=True), dict(inplace=True),
                                dict(hs=False, tail=True, eps=0.02), dict(shifted=True, inplace=True, storage=1)])
@pytest.mark.parametrize("n,sigma", [((4, 4, 8), 4), ((16, 16, 32), 4), ((32, 32, 70), 6), ((33, 9, 40), 14)])
def test_chains(L, n, sigma, kw):
    from paper_0712_2247_gb300 import inputs

    rho, u = inputs.random_fields(n[::-1], 6 * 0.2 / (np.pi * sigma ** 3), seed=sum(n))
    got = []
    for calls, steps in ((1, 48), (48, 1)):
        with L.Slit(*n, sigma, 0.2, 0.85, body=(1e-5, -2e-6, 0.0), **kw) as s:
            s.set_fields(rho, u)
            for _ in range(calls):
                s.step(steps)
                if calls > 1:
                    s.status()
            assert s.status() == 0
            got.append((*s.moments(), s.forces()))
    for a, b in zip(*got):
        assert np.array_equal(a, b)


@pytest.mark.parametrize("inplace,storage", [(True, 0), (True, 1), (False, 0)])
@pytest.mark.parametrize("nx,ny", [(4, 4), (16, 9), (32, 16)])
def test_graph_replay(L, nx, ny, inplace, storage):
    H = [9, 16, 12, 8]
    args = (H, [0.2, 0.15, 0.22, 0.18], [1e-6, 2e-6, 1e-6, 3e-6], [0.8, 1.0, 0.7, 0.9], 4, nx, ny)
    with L.Ensemble(*args, storage=storage, inplace=inplace, seed=5) as a, \
            L.Ensemble(*args, storage=storage, inplace=inplace, seed=5) as b:
        a.run(tol=1e-30, max_steps=60, check_every=20)
        for _ in range(a.t):
            b.step(1)
            b.status()
        assert a.t == b.t >= 60
        for x, y in zip(a.moments(), b.moments()):
            assert np.array_equal(x, y)
