"""The direct tail sum against the FP64 oracle at the edges of its blocks.

Four x nodes a thread, displacements four at a time, a half space of rows dealt
to eight warps: rows that end inside a block, extents below one block and below
the kernel's reach (several images of a node), reaches that are and are not
multiples of four, a cut-off just above sigma (few terms per row), walls and
periodic z. Tolerance 1e-5 of the largest force, as for all force comparisons.
"""
import numpy as np
import pytest

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("nx,ny,nz,sigma,rcut,zper", [
    (27, 6, 12, 4, 2.5, False), (60, 5, 11, 4, 2.5, False), (5, 3, 14, 4, 2.5, True), (3, 1, 9, 2, 4.0, False),
    (33, 4, 13, 4, 2.0, True), (24, 7, 10, 6, 1.0, False), (45, 5, 12, 6, 1.7, False), (12, 24, 24, 8, 2.5, False),
    (1, 1, 30, 4, 2.5, False)])
def test_direct_tail(nx, ny, nz, sigma, rcut, zper):
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
    G = g.forces()
    assert np.abs(G - F).max() <= 1e-5 * np.abs(F).max()
    # a uniform periodic state has no force at all
    if zper:
        g.set_fields(np.full_like(rho, np.float32(n0)), np.zeros_like(u))
        assert not g.forces().any()
