"""The tail sum pair by pair, used for shells of few pairs on grids that fill the chip.

Against the FP64 oracle (tolerance 1e-5 of the largest force, as for all force
comparisons) with walls and periodic z, odd extents and extents below the reach, on
both sides of the rule's line; a density that is not finite stays in its shell; a
stack of slits has the bits of lone ones; and a cut-off at sigma costs a small part of
a wider one (by rows 0.37 of it).
"""
import numpy as np
import pytest

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("nx,ny,nz,sigma,rcut,zper", [
    (17, 17, 17, 4, 1.0, False), (17, 17, 15, 4, 1.0, False), (7, 3, 220, 8, 1.0, True), (31, 29, 26, 6, 1.0, True),
    (45, 41, 40, 2, 1.5, False), (45, 41, 38, 2, 1.5, True)])
def test_against_oracle(nx, ny, nz, sigma, rcut, zper):
    import oracle
    from paper_0712_2247_gb300 import inputs, lbif

    n0 = 6 * 0.2 / (np.pi * sigma ** 3)
    rho, u = inputs.random_fields((nz, ny, nx), n0, seed=nx + nz)
    kw = dict(tail=True, eps=0.3, rcut=rcut, hs=False)
    o = oracle.Oracle(nx, ny, nz, sigma, 0.2, 0.8, zper=zper, **kw)
    o.init_fields(rho.astype(np.float64), u.astype(np.float64))
    F = o.forces()
    F = np.asarray(F[0] if isinstance(F, tuple) else F) / n0
    with lbif.Slit(nx, ny, nz, sigma, 0.2, 0.8, periodic_z=zper, **kw) as g:
        g.set_fields(rho, u)
        assert np.abs(g.forces() - F).max() <= 1e-5 * np.abs(F).max()
        if zper:  # a uniform periodic state has no force at all
            g.set_fields(np.full_like(rho, np.float32(n0)), np.zeros_like(u))
            assert not g.forces().any()


def test_infinite_density_stays_in_its_shell():
    from test_gpu_tail_direct_nonfinite import reached

    from paper_0712_2247_gb300 import inputs, lbif

    nx, ny, nz, sigma, at = 31, 29, 26, 6, (3, 28, 0)
    rho, u = inputs.random_fields((nz, ny, nx), 6 * 0.2 / (np.pi * sigma ** 3), seed=1)
    F = []
    for v in (rho[at], np.inf):
        rho[at] = v
        with lbif.Slit(nx, ny, nz, sigma, 0.2, 0.8, tail=True, eps=0.3, rcut=1.0, hs=False) as g:
            g.set_fields(rho, u)
            F.append(g.forces())
    hit = reached(rho.shape, sigma, 1.0, False, at)
    hit[at] = True
    for a, b in zip(*F):
        assert np.array_equal(a[~hit], b[~hit]) and not np.isfinite(b[hit]).any()


def test_stack_equals_lone_slits():
    from test_gpu_tail_direct_stack import stack

    from paper_0712_2247_gb300 import lbif

    H, nx, ny = [30, 14, 25], 23, 21
    with stack(H, nx, ny, rcut=1.0) as e:
        e.step(9)
        r, u = e.moments()
        for h, z in zip(H, e.zlo):
            with lbif.Slit(nx, ny, h, 4, 0.2, 0.9, body=(1e-6, 0, 0), tail=True, eps=0.2, rcut=1.0, noise=0.0) as g:
                g.step(9)
                r1, u1 = g.moments()
                assert np.array_equal(r[z:z + h], r1) and np.array_equal(u[:, z:z + h], u1)


def test_cut_off_at_sigma_is_cheap():
    from paper_0712_2247_gb300 import lbif

    def tail_ms(rcut):
        with lbif.Slit(100, 100, 60, 4, 0.15, 0.9, tail=True, eps=0.02, rcut=rcut) as g:
            g.step(2)
            return min(g.step_profiled(4)[0]["tail"] for _ in range(5))

    assert tail_ms(1.0) < 0.25 * tail_ms(1.25)
