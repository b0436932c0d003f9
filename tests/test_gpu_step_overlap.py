"""Steps whose kernels come up while their predecessors still run.

Small grids launch the step's kernels with programmatic dependent launch, larger
ones without. A kernel that read before its predecessor's end would give other
bits: many steps in one call are therefore compared with steps that the host waits
for one by one, on grids on both sides of the line, for FP32 and FP16 storage, in
place, and with the fluid-fluid tail between the overlapping kernels.
"""
import numpy as np
import pytest

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def L():
    from paper_0712_2247_gb300 import build, lbif

    build.build()
    return lbif


@pytest.mark.parametrize("kw", [{}, dict(storage=1), dict(storage=1, inplace=True), dict(tail=True, eps=0.3)])
@pytest.mark.parametrize("n,sigma", [((4, 4, 8), 4), ((9, 7, 21), 4), ((16, 16, 32), 4), ((24, 24, 48), 6),
                                     ((32, 32, 76), 8), ((32, 32, 77), 8), ((48, 48, 48), 4)])
def test_steps_in_a_row_equal_steps_one_by_one(L, n, sigma, kw):
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
