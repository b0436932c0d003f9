"""Cross-sections just above 64 nodes that fill few nodes of a marched tile.

They run whole planes per CTA like the smaller ones. The results equal those of a
grid that holds copies of the state, which runs marched tiles, bit for bit.
"""
import numpy as np
import pytest

pytestmark = pytest.mark.gpu

THIN = [(65, 1), (1, 65), (33, 2), (2, 33), (22, 3), (17, 4), (11, 11), (13, 6), (1, 128), (128, 1), (127, 1), (3, 41)]


@pytest.fixture(scope="module")
def L():
    from paper_0712_2247_gb300 import build, lbif

    build.build()
    return lbif


@pytest.mark.parametrize("nx,ny", THIN + [(16, 8), (43, 3)])
@pytest.mark.parametrize("nz,zper,kw", [(13, False, {}), (9, True, dict(storage=1)), (311, False, dict(inplace=True)),
                                        (1, True, dict(inplace=True, storage=1))])
def test_thin_equals_copies(L, nx, ny, nz, zper, kw):
    from paper_0712_2247_gb300 import inputs

    k, m = -(-32 // nx), max(1, -(-4 // ny))
    if nx * ny * k * m <= 128:
        k *= 2
    a = dict(periodic_z=zper, body=(1e-5, -2e-6, 0.0), **kw)
    rho, u = inputs.random_fields((nz, ny, nx), 6 * 0.2 / (np.pi * 4 ** 3), seed=nx + nz)
    s = L.Slit(nx, ny, nz, 4, 0.2, 0.85, **a)
    b = L.Slit(k * nx, m * ny, nz, 4, 0.2, 0.85, **a)
    b.set_shapes(pull_gathers="prefetch")
    s.set_fields(rho, u)
    b.set_fields(np.ascontiguousarray(np.tile(rho, (1, m, k))), np.ascontiguousarray(np.tile(u, (1, 1, m, k))))
    for g in (s, b):
        g.step(7)
    (r0, u0), (r1, u1) = s.moments(), b.moments()
    assert s.status() == 0 and b.status() == 0
    assert np.array_equal(np.tile(r0, (1, m, k)), r1) and np.array_equal(np.tile(u0, (1, 1, m, k)), u1)
    assert np.array_equal(np.tile(s.forces(), (1, 1, m, k)), b.forces())


@pytest.mark.parametrize("nx,ny", [(65, 1), (1, 65), (33, 2)])
def test_thin_costs_less_than_full_tiles(L, nx, ny):
    """Against a cross-section that fills the marched tiles which this one would
    occupy: with idle tiles both took about as long; 0.7 of its time is allowed."""
    def pull_ms(x, y):
        with L.Slit(x, y, 6000, 4, 0.2, 0.9) as g:
            g.step(2)
            return min(g.step_profiled(6)[0]["collide_stream"] for _ in range(6))

    assert pull_ms(nx, ny) < 0.7 * pull_ms(*((nx, 4) if nx > 1 else (8, ny)))
