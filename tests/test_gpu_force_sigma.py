"""The vectorised shell force at sigma 6 and 10 against the FP64 oracle.

Window alignments differ from those of sigma 4, 8 and 12 (corner offsets 4, 2
and 7, 3). Grids: a full tile row, ragged ones (one node into the next tile,
rows that end inside a four-node block), narrow grids and rows shorter than
one block; walls and periodic z; the energy source. Tolerance 1e-5 normwise, as
for every force comparison with FP32 fields of unit scale.
"""
import numpy as np
import pytest

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("sigma", [6, 10])
@pytest.mark.parametrize("nx,ny,nz,zper", [
    (128, 5, 14, False), (129, 4, 12, True), (134, 3, 13, False), (45, 6, 15, False), (5, 4, 12, True), (3, 2, 16, False)])
def test_force(sigma, nx, ny, nz, zper):
    import oracle
    from paper_0712_2247_gb300 import inputs, lbif

    n0 = 6 * 0.2 / (np.pi * sigma ** 3)
    rho, u = inputs.random_fields((nz, ny, nx), n0, seed=nx + sigma)
    g = lbif.Slit(nx, ny, nz, sigma, 0.2, 0.8, periodic_z=zper, body=(1e-4, 0, 0))
    g.set_fields(rho, u)
    o = oracle.Oracle(nx, ny, nz, sigma, 0.2, 0.8, zper=zper, body=(1e-4, 0, 0))
    o.init_fields(rho.astype(np.float64), u.astype(np.float64))
    F = o.forces()
    F = np.asarray(F[0] if isinstance(F, tuple) else F) / n0
    assert np.abs(g.forces() - F).max() <= 1e-5 * np.abs(F).max()


@pytest.mark.parametrize("sigma", [6, 10])
@pytest.mark.parametrize("nx,ny", [(130, 3), (9, 4)])
def test_energy_source(sigma, nx, ny):
    import oracle
    from paper_0712_2247_gb300 import lbif

    nz = 18
    g = lbif.Slit(nx, ny, nz, sigma, 0.2, 0.8, c2=True, seed=4)
    o = oracle.Oracle(nx, ny, nz, sigma, 0.2, 0.8, c2=True, seed=4)
    g.step(3)
    o.step(3)
    for a, b in zip(g.moments(), o.moments()):
        assert np.abs(a - b).max() <= 1e-5 * np.abs(b).max()
