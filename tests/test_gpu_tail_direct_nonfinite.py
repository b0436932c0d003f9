"""The direct tail sum takes part only of what lies in the shell.

Displacements go four at a time, so a thread also loads neighbours inside the core
and beyond the cut-off, whose coefficients are zero. An infinite density must reach
exactly the nodes whose shell sigma <= |d| <= rcut sigma holds it (with all its
periodic images); every other node keeps the bits it has without it.
"""
import numpy as np
import pytest

pytestmark = pytest.mark.gpu


def reached(shape, sigma, rcut, zper, at):
    """Nodes of the shell around ``at``, with periodic images."""
    nz, ny, nx = shape
    R = int(np.ceil(rcut * sigma))
    out = np.zeros(shape, bool)
    d = np.arange(-R, R + 1)
    dz, dy, dx = np.meshgrid(d, d, d, indexing="ij")
    r2 = dz * dz + dy * dy + dx * dx
    on = (r2 >= sigma * sigma) & (r2 <= (rcut * sigma) ** 2)
    z, y, x = at[0] + dz[on], (at[1] + dy[on]) % ny, (at[2] + dx[on]) % nx
    if zper:
        z %= nz
    ok = (z >= 0) & (z < nz)
    out[z[ok], y[ok], x[ok]] = True
    return out


@pytest.mark.parametrize("bad", [np.inf, np.nan])
@pytest.mark.parametrize("nx,ny,nz,sigma,rcut,zper,at", [
    (27, 26, 30, 4, 2.5, False, (3, 5, 0)), (27, 26, 30, 4, 2.5, False, (29, 25, 26)),
    (45, 23, 24, 4, 2.5, True, (0, 0, 22)), (33, 24, 20, 6, 1.0, False, (9, 12, 13)),
    (30, 31, 28, 6, 1.7, True, (27, 1, 29)), (7, 3, 40, 2, 4.0, False, (20, 1, 3))])
def test_infinite_density_stays_in_its_shell(nx, ny, nz, sigma, rcut, zper, at, bad):
    from paper_0712_2247_gb300 import inputs, lbif

    n0 = 6 * 0.2 / (np.pi * sigma ** 3)
    rho, u = inputs.random_fields((nz, ny, nx), n0, seed=nx + nz)
    F = []
    for v in (rho[at], bad):
        rho[at] = v
        with lbif.Slit(nx, ny, nz, sigma, 0.2, 0.8, periodic_z=zper, tail=True, eps=0.3, rcut=rcut, hs=False) as g:
            g.set_fields(rho, u)
            F.append(g.forces())
    hit = reached(rho.shape, sigma, rcut, zper, at)
    hit[at] = True
    assert np.isfinite(F[0]).all() and not hit.all()
    for a, b in zip(*F):
        assert np.array_equal(a[~hit], b[~hit])
        assert not np.isfinite(b[hit]).any()
