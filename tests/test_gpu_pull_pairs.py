"""The pull pass with two planes per round equals the one-plane form bit for bit.

A thread of the default form steps the nodes of two planes; rounds that touch
a wall, end on a single plane, or join two slits take its one-node path. Edges:
segments of one, odd and all planes, odd heights, ragged tiles, single-plane
slits, periodic z, both storage types and layouts, velocity-shifted forcing, a
stack of slits whose pairs straddle gaps, and frozen slits beside active ones.
"""
import numpy as np
import pytest

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def L():
    from paper_0712_2247_gb300 import build, lbif

    build.build()
    return lbif


def state(g):
    r, u = g.moments()
    assert g.status() == 0
    return r, u


@pytest.mark.parametrize("nx,ny,nz,zper,kw", [
    (32, 4, 9, False, {}),
    (45, 7, 14, False, dict(storage=1)),
    (33, 5, 11, True, {}),
    (64, 8, 2, True, dict(storage=1)),
    (40, 6, 1, True, {}),
    (40, 6, 13, False, dict(inplace=True)),
    (37, 9, 8, True, dict(inplace=True, storage=1)),
    (36, 4, 12, False, dict(shifted=True)),
    (36, 4, 12, False, dict(c2=True)),
])
def test_pairs_equal_single_planes(L, nx, ny, nz, zper, kw):
    a = dict(periodic_z=zper, body=(1e-5, -2e-6, 0.0), seed=5, **kw)
    ref = L.Slit(nx, ny, nz, 4, 0.2, 0.85, **a)
    ref.set_shapes(pull_gathers="prefetch")
    ref.step(17)
    r0, u0 = state(ref)
    for lz in (0, 1, 2, 3, 6, nz, 64):
        g = L.Slit(nx, ny, nz, 4, 0.2, 0.85, **a)
        g.set_shapes(pull_lz=lz)
        g.step(17)
        r, u = state(g)
        assert np.array_equal(r, r0) and np.array_equal(u, u0), lz


@pytest.mark.parametrize("storage,inplace", [(0, False), (0, True), (1, False), (1, True)])
def test_pairs_in_a_stack_of_slits(L, storage, inplace):
    H = [9, 8, 1, 2, 15, 10]
    n = len(H)
    a = (H, np.linspace(0.1, 0.22, n), np.geomspace(1e-6, 1e-5, n), np.linspace(0.7, 1.1, n), 4, 33, 6)
    out = []
    for shapes in (dict(pull_gathers="prefetch"), dict(pull_lz=0), dict(pull_lz=3), dict(pull_lz=10)):
        e = L.Ensemble(*a, storage=storage, inplace=inplace, seed=2)
        e.set_shapes(**shapes)
        # slits freeze at different checks, so frozen ones lie beside active ones
        out.append((e.run(tol=1e-3, max_steps=60, check_every=10),) + e.moments())
    for taken, r, u in out[1:]:
        assert np.array_equal(taken, out[0][0])
        assert np.array_equal(r, out[0][1]) and np.array_equal(u, out[0][2])
