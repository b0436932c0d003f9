"""Wide slits of few planes.

Their pull pass steps one plane a round. Same bits as the prefetched form and as a
smaller grid's state repeated (which runs the pair form), for both storages and
layouts, walls and periodic z, on both sides of the rule's line; and the pass takes at
most 1.12 of the prefetched form's time (with pairs 1.27 to 1.33).
"""
import numpy as np
import pytest

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("kw", [{}, dict(storage=1), dict(inplace=True), dict(storage=1, inplace=True),
                                dict(periodic_z=True), dict(shifted=True)])
@pytest.mark.parametrize("nz", [1, 2, 7, 8, 9])
def test_same_bits(nz, kw):
    from paper_0712_2247_gb300 import inputs, lbif

    nx, ny, k, m = 67, 32, 4, 8  # 268 x 256: 576 tiles of 32 x 4
    a = dict(body=(1e-5, -2e-6, 0.0), **kw)
    rho, u = inputs.random_fields((nz, ny, nx), 6 * 0.15 / (np.pi * 4 ** 3), seed=nz)
    big = np.ascontiguousarray(np.tile(rho, (1, m, k))), np.ascontiguousarray(np.tile(u, (1, 1, m, k)))
    with lbif.Slit(nx, ny, nz, 4, 0.15, 0.9, **a) as s, lbif.Slit(k * nx, m * ny, nz, 4, 0.15, 0.9, **a) as b, \
            lbif.Slit(k * nx, m * ny, nz, 4, 0.15, 0.9, **a) as c:
        c.set_shapes(pull_gathers="prefetch")
        s.set_fields(rho, u)
        b.set_fields(*big)
        c.set_fields(*big)
        for g in (s, b, c):
            g.step(7)
            assert g.status() == 0
        (r0, u0), (r1, u1), (r2, u2) = s.moments(), b.moments(), c.moments()
    assert np.array_equal(r1, r2) and np.array_equal(u1, u2)
    assert np.array_equal(np.tile(r0, (1, m, k)), r1) and np.array_equal(np.tile(u0, (1, 1, m, k)), u1)


@pytest.mark.parametrize("n,kw", [((300, 300, 4), {}), ((300, 300, 5), dict(inplace=True))])
def test_as_fast_as_one_plane_a_round(n, kw):
    from paper_0712_2247_gb300 import lbif

    def pull_ms(gathers):
        with lbif.Slit(*n, 2, 0.15, 0.9, **kw) as g:
            g.set_shapes(pull_gathers=gathers)
            g.step(2)
            return min(g.step_profiled(6)[0]["collide_stream"] for _ in range(5))

    assert pull_ms("loads") < 1.12 * pull_ms("prefetch")
