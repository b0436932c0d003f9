"""Stacks of slits with the direct tail sum.

Gap planes between the slits (twelve each at sigma 4, cut 2.5) take no part: a stack
of single-plane slits costs a fraction of a grid as high, and every slit has the
bits of a lone one. Through the C ABI, which takes the tail for stacks.
"""
import ctypes

import numpy as np
import pytest

pytestmark = pytest.mark.gpu


def stack(H, nx, ny, sigma=4, rcut=2.5):
    """An Ensemble with the tail on (its constructor leaves it off)."""
    from paper_0712_2247_gb300 import lbif

    class Stack(lbif.Ensemble):
        def __init__(self):
            self._lib = lbif.load_library()
            n = len(H)
            f = lbif.Force((ctypes.c_double * 3)(), 1, 1, 1, 0, 1, 0.2, rcut, 0, 0)
            o = lbif.Opts(0, 3, 0.0, None, 1)
            Hc = np.asarray(H, np.int32)
            a = [np.full(n, v) for v in (0.2, 1e-6, 0.9)]
            pd = lambda v: v.ctypes.data_as(ctypes.POINTER(ctypes.c_double))
            self._h = lbif._vp()
            self._check(self._lib.lbif_batch_create(
                ctypes.byref(self._h), n, Hc.ctypes.data_as(ctypes.POINTER(ctypes.c_int32)), *map(pd, a),
                float(sigma), nx, ny, ctypes.byref(f), ctypes.byref(o)))
            self.zlo = np.zeros(n, np.int32)
            self._check(self._lib.lbif_batch_info(self._h, None, self.zlo.ctypes.data_as(ctypes.POINTER(ctypes.c_int32)),
                                                  None))
            self.nslits, self.shape = n, (int(self.zlo[-1]) + int(Hc[-1]), ny, nx)

    return Stack()


def test_stack_equals_lone_slits():
    from paper_0712_2247_gb300 import lbif

    H, nx, ny = [9, 14, 1, 30], 13, 7
    with stack(H, nx, ny) as e:
        e.step(9)
        r, u = e.moments()
        F = e.forces()
        for h, z in zip(H, e.zlo):
            with lbif.Slit(nx, ny, h, 4, 0.2, 0.9, body=(1e-6, 0, 0), tail=True, eps=0.2, noise=0.0) as g:
                g.step(9)
                r1, u1 = g.moments()
                assert np.array_equal(r[z:z + h], r1) and np.array_equal(u[:, z:z + h], u1)
                assert np.array_equal(F[:, z:z + h], g.forces())


def test_gap_planes_take_no_part():
    """13 planes of 14 lie in gaps; half of the whole grid's time is allowed."""
    from paper_0712_2247_gb300 import lbif

    def tail_ms(g):
        g.step(2)
        return min(g.step_profiled(4)[0]["tail"] for _ in range(5))

    nx, ny = 60, 44
    with stack([1] * 24, nx, ny) as e, lbif.Slit(nx, ny, e.shape[0], 4, 0.2, 0.9, tail=True, eps=0.2) as g:
        assert tail_ms(e) < 0.5 * tail_ms(g)
