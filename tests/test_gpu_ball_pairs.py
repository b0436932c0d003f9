"""The ball average's tiles (two x nodes a thread) against the direct sums.

The direct kernel runs on grids below half a tile; a state of period (nx, ny) on a
larger grid must give the same forces and pressure bit for bit. Odd extents (a
pair with one node inside), rows and tiles that end early, every specialised
radius up to 6, z chunks of 2 R, R and R / 2 planes and explicit CTA targets, both
stagings.
"""
import numpy as np
import pytest

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("nx,ny,k,m", [(7, 5, 5, 4), (15, 7, 3, 3), (5, 3, 7, 7), (13, 6, 5, 3)])
@pytest.mark.parametrize("sigma,nz,zper", [(2, 9, False), (4, 17, True), (6, 40, False), (8, 13, False), (10, 25, True),
                                           (12, 31, False)])
def test_ball_pairs_equal_direct(nx, ny, k, m, sigma, nz, zper):
    from paper_0712_2247_gb300 import inputs, lbif

    rho, u = inputs.random_fields((nz, ny, nx), 6 * 0.2 / (np.pi * sigma ** 3), seed=nx + nz)
    s = lbif.Slit(nx, ny, nz, sigma, 0.2, 0.8, periodic_z=zper)
    b = lbif.Slit(k * nx, m * ny, nz, sigma, 0.2, 0.8, periodic_z=zper)
    s.set_fields(rho, u)
    p = np.tile(s.pressure(), (1, m, k))
    for ctas in (0, 1, 500, 4000):
        for staging in ("tma", "loads"):
            b.set_shapes(ball_ctas=ctas, ball_staging=staging)
            b.set_fields(np.ascontiguousarray(np.tile(rho, (1, m, k))), np.ascontiguousarray(np.tile(u, (1, 1, m, k))))
            assert np.array_equal(b.pressure(), p), (ctas, staging)
