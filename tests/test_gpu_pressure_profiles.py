"""Pressure (four nodes a thread) and profile sums at the edges of their blocks.

Pressure against the FP64 oracle (1e-6 of its largest value, as the existing
comparison) for every vectorised diameter, wide, ragged, narrow and one-column
grids, an ideal fluid and gap planes of a stack. Plane averages against
math.fsum of the same FP32 fields: 1e-12 of the field's magnitude for the
averages and the totals, rows that end inside a thread batch, and a flow whose average
cancels.
"""
import math

import numpy as np
import pytest

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("sigma", [4, 6, 8, 10, 12])
@pytest.mark.parametrize("nx,ny,nz,zper", [(128, 3, 26, False), (131, 2, 25, True), (30, 5, 27, False), (3, 2, 26, False)])
def test_pressure(sigma, nx, ny, nz, zper):
    import oracle
    from paper_0712_2247_gb300 import inputs, lbif

    rho, u = inputs.random_fields((nz, ny, nx), 6 * 0.2 / (np.pi * sigma ** 3), seed=nx)
    g = lbif.Slit(nx, ny, nz, sigma, 0.2, 0.8, periodic_z=zper)
    g.set_fields(rho, u)
    o = oracle.Oracle(nx, ny, nz, sigma, 0.2, 0.8, zper=zper)
    o.init_fields(rho.astype(np.float64), u.astype(np.float64))
    p = o.moments(pressure=True)[2]
    assert np.abs(g.pressure() - p).max() <= 1e-6 * np.abs(p).max()


def test_pressure_of_a_stack_and_without_force():
    from paper_0712_2247_gb300 import lbif

    e = lbif.Ensemble([9, 12], [0.1, 0.2], [0.0, 0.0], [0.8, 0.9], 4, 33, 5, storage=0, noise=1e-3, seed=2)
    p = np.full(e.shape, 7.0, np.float32)
    e._check(e._lib.lbif_moments(e._h, None, None, p.ctypes.data, 0))
    r, _ = e.moments()
    gap = np.ones(e.shape[0], bool)
    for z, h in zip(e.zlo, e.H):
        gap[z:z + h] = False
    assert (p[gap] == 0).all() and (p[~gap] > 0).all()
    g = lbif.Slit(37, 4, 9, 4, 0.2, 0.8, hs=False, seed=3)
    r, _ = g.moments()
    assert np.abs(g.pressure() - r / 3).max() <= 1e-6 * r.max()


@pytest.mark.parametrize("nx,ny,nz", [(1, 1, 5), (3, 7, 4), (256, 40, 3), (201, 33, 9), (1024, 70, 2), (5, 300, 3)])
def test_profiles(nx, ny, nz):
    from paper_0712_2247_gb300 import lbif

    rng = np.random.default_rng(nx)
    g = lbif.Slit(nx, ny, nz, 2, 0.2, 0.8)
    rho = (g.n0 * (1 + 0.1 * rng.standard_normal((nz, ny, nx)))).astype(np.float32)
    u = (0.05 * rng.standard_normal((3, nz, ny, nx))).astype(np.float32)
    u[0] -= u[0].mean((1, 2), keepdims=True)
    g.set_fields(rho, u)
    n, ux, tot = g.profiles()
    r, v = g.moments()
    n0 = float(np.float32(g.n0))
    d = np.float32(rho) / np.float32(g.n0) - np.float32(1)
    A = nx * ny
    for z in range(nz):
        assert abs(ux[z] - math.fsum(v[0, z].ravel().astype(float)) / A) <= 1e-12 * 0.05
        assert abs(n[z] - n0 * (1 + math.fsum(d[z].ravel().astype(float)) / A)) <= 1e-12 * n0
    m = [math.fsum(((1 + d.astype(float)) * v[a].astype(float)).ravel()) * n0 for a in range(3)]
    assert np.abs(tot[1:] - m).max() <= 1e-12 * n0 * 0.05 * A * nz
