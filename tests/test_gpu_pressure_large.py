"""Pressure on both sides of the vectorised kernel's line (1024 nodes per SM).

A state of period (nx, ny) on a grid of m ny rows runs the vectorised kernel, the state
itself the per-node one; both against the FP64 oracle (1e-6 of its largest value, as
the existing comparison) for every vectorised diameter, wide, ragged, narrow and
few-column grids.
"""
import numpy as np
import pytest

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("sigma", [4, 6, 8, 10, 12])
@pytest.mark.parametrize("nx,ny,nz,m,zper", [(128, 3, 26, 16, False), (131, 2, 25, 24, True), (30, 5, 27, 39, False),
                                             (3, 2, 26, 998, False), (203, 4, 24, 8, True)])
def test_pressure(sigma, nx, ny, nz, m, zper):
    import oracle
    from paper_0712_2247_gb300 import inputs, lbif

    assert nx * ny * m * nz >= 1024 * 152 > nx * ny * nz
    rho, u = inputs.random_fields((nz, ny, nx), 6 * 0.2 / (np.pi * sigma ** 3), seed=nx)
    o = oracle.Oracle(nx, ny, nz, sigma, 0.2, 0.8, zper=zper)
    o.init_fields(rho.astype(np.float64), u.astype(np.float64))
    p = o.moments(pressure=True)[2]
    for k in (1, m):
        with lbif.Slit(nx, k * ny, nz, sigma, 0.2, 0.8, periodic_z=zper) as g:
            g.set_fields(np.ascontiguousarray(np.tile(rho, (1, k, 1))), np.ascontiguousarray(np.tile(u, (1, 1, k, 1))))
            assert np.abs(g.pressure() - np.tile(p, (1, k, 1))).max() <= 1e-6 * np.abs(p).max()


def test_stack():
    from paper_0712_2247_gb300 import lbif

    H = [90, 120]
    e = lbif.Ensemble(H, [0.1, 0.2], [0.0, 0.0], [0.8, 0.9], 4, 33, 24, storage=0, noise=1e-3, seed=2)
    assert e.N >= 1024 * 152
    p = np.full(e.shape, 7.0, np.float32)
    e._check(e._lib.lbif_moments(e._h, None, None, p.ctypes.data, 0))
    gap = np.ones(e.shape[0], bool)
    for z, h in zip(e.zlo, H):
        gap[z:z + h] = False
    assert (p[gap] == 0).all() and (p[~gap] > 0).all()
