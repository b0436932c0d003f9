"""Narrow grids whose padded rows would be 128 bytes.

A warp spans several of their rows, which would all start in the same banks. Columns
are added there; a wider grid, whose rows are longer anyway, is the measure (1.4 of its
ball time per node; 2.0 without the columns), and results equal those
of a grid that holds copies.
"""
import numpy as np
import pytest

pytestmark = pytest.mark.gpu


def test_no_slower_than_a_wider_grid():
    from paper_0712_2247_gb300 import lbif

    def us(nx):
        with lbif.Slit(nx, 256, 211, 10, 0.15, 0.9) as g:
            g.step(2)
            return min(g.step_profiled(6)[0]["ball_g2"] for _ in range(5)) / nx

    assert us(5) < 1.4 * us(12)


@pytest.mark.parametrize("nx,ny,sigma,kw", [(8, 9, 12, {}), (6, 7, 10, dict(storage=1, inplace=True)),
                                            (14, 5, 8, dict(tail=True, eps=0.05)), (5, 4, 12, dict(inplace=True))])
def test_same_as_copies(nx, ny, sigma, kw):
    from paper_0712_2247_gb300 import inputs, lbif

    nz, k, m = 21, 4, 3
    rho, u = inputs.random_fields((nz, ny, nx), 6 * 0.15 / (np.pi * sigma ** 3), seed=nx)
    with lbif.Slit(nx, ny, nz, sigma, 0.15, 0.9, **kw) as s, lbif.Slit(k * nx, m * ny, nz, sigma, 0.15, 0.9, **kw) as b:
        s.set_fields(rho, u)
        b.set_fields(np.ascontiguousarray(np.tile(rho, (1, m, k))), np.ascontiguousarray(np.tile(u, (1, 1, m, k))))
        s.step(6)
        b.step(6)
        (r0, u0), (r1, u1) = s.moments(), b.moments()
        assert np.array_equal(np.tile(r0, (1, m, k)), r1) and np.array_equal(np.tile(u0, (1, 1, m, k)), u1)
