"""The spectral tail against the FP64 oracle at the edges of its kernels.

The z sum keeps 64 planes per CTA and four per thread and slides windows of the
kernel's even and odd parts; lines are transformed 4096 or 1024 elements per
CTA, or 256-point ones in registers. Heights at and beside multiples of 4 and 64,
reaches from 2 to beyond the height, periodic wrap with the reach above nz,
lengths 2 to 512, both x and y. Tolerance 1e-5 of the largest force.
"""
import numpy as np
import pytest

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("nx,ny,nz,sigma,rcut,zper", [
    (16, 8, 3, 2, 1.0, False), (16, 8, 64, 2, 2.5, False), (8, 8, 65, 4, 2.0, False), (8, 16, 63, 4, 2.5, True),
    (32, 2, 12, 4, 2.5, True), (2, 32, 13, 4, 2.5, False), (512, 2, 9, 2, 2.0, False), (2, 512, 9, 2, 2.0, True),
    (256, 2, 11, 4, 1.5, True), (8, 8, 130, 8, 2.5, False), (4, 8, 7, 8, 2.5, True)])
def test_spectral_tail(nx, ny, nz, sigma, rcut, zper):
    import oracle
    from paper_0712_2247_gb300 import inputs, lbif

    n0 = 6 * 0.2 / (np.pi * sigma ** 3)
    rho, u = inputs.random_fields((nz, ny, nx), n0, seed=nx + nz)
    kw = dict(tail=True, eps=0.3, rcut=rcut, hs=False)
    g = lbif.Slit(nx, ny, nz, sigma, 0.2, 0.8, periodic_z=zper, **kw)
    g.set_fields(rho, u)
    o = oracle.Oracle(nx, ny, nz, sigma, 0.2, 0.8, zper=zper, **kw)
    o.init_fields(rho.astype(np.float64), u.astype(np.float64))
    F = o.forces()
    F = np.asarray(F[0] if isinstance(F, tuple) else F) / n0
    assert np.abs(g.forces() - F).max() <= 1e-5 * np.abs(F).max()
