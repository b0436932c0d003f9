"""Narrow grids: the same step, bit for bit, as on a grid that holds copies.

A state of period (nx, ny) on a grid of (k nx, m ny) nodes steps like the nx x ny
grid itself (periodic in x and y). The large grid runs the one-plane tiles; the
small one whole planes per CTA (cross-sections of at most 64 nodes) or paired
planes on tiles 32, 16 or 8 columns wide. Walls, periodic z, FP16, in place,
planes that do not fill a CTA, one-node cross-sections, halos wider and
narrower than the grid, and a stack of thin slits against separate ones.
"""
import numpy as np
import pytest

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def L():
    from paper_0712_2247_gb300 import build, lbif

    build.build()
    return lbif


@pytest.mark.parametrize("nx,ny", [(1, 1), (4, 4), (5, 3), (64, 1), (8, 8), (3, 21), (13, 5), (16, 16), (20, 7), (7, 30)])
@pytest.mark.parametrize("nz,zper,sigma,kw", [
    (13, False, 4, {}), (9, True, 4, dict(storage=1)), (12, False, 6, dict(inplace=True, storage=1)),
    (310, False, 4, dict(shifted=True)), (1, True, 4, dict(inplace=True))])
def test_narrow_equals_copies(L, nx, ny, nz, zper, sigma, kw):
    from paper_0712_2247_gb300 import inputs

    k, m = -(-32 // nx), max(1, -(-4 // ny))
    a = dict(periodic_z=zper, body=(1e-5, -2e-6, 0.0), **kw)
    rho, u = inputs.random_fields((nz, ny, nx), 6 * 0.2 / (np.pi * sigma ** 3), seed=nx + nz)
    s = L.Slit(nx, ny, nz, sigma, 0.2, 0.85, **a)
    b = L.Slit(k * nx, m * ny, nz, sigma, 0.2, 0.85, **a)
    b.set_shapes(pull_gathers="prefetch")
    s.set_fields(rho, u)
    b.set_fields(np.ascontiguousarray(np.tile(rho, (1, m, k))), np.ascontiguousarray(np.tile(u, (1, 1, m, k))))
    for g in (s, b):
        g.step(7)
    (r0, u0), (r1, u1) = s.moments(), b.moments()
    assert s.status() == 0 and b.status() == 0
    assert np.array_equal(np.tile(r0, (1, m, k)), r1) and np.array_equal(np.tile(u0, (1, 1, m, k)), u1)
    # the halo too: the next force reads it
    assert np.array_equal(np.tile(s.forces(), (1, 1, m, k)), b.forces())


@pytest.mark.parametrize("nx,ny", [(4, 4), (1, 1), (9, 9)])
def test_thin_stack_equals_separate(L, nx, ny):
    H = [8, 33, 1, 12, 80]
    n = len(H)
    eta, F, tau = np.linspace(0.1, 0.22, n), np.geomspace(1e-6, 1e-5, n), np.linspace(0.7, 1.1, n)
    e = L.Ensemble(H, eta, F, tau, 4, nx, ny, storage=0, noise=0.0)
    e.step(11)
    r, u = e.moments()
    for i, h in enumerate(H):
        g = L.Slit(nx, ny, h, 4, eta[i], tau[i], body=(F[i], 0, 0), noise=0.0)
        g.step(11)
        r1, u1 = g.moments()
        z = e.zlo[i]
        assert np.array_equal(r[z:z + h], r1) and np.array_equal(u[:, z:z + h], u1), i
