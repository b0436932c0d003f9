"""Direct ball sums of a large radius on a small grid.

Their blocks of 256 threads share the rows they read in L1. A node's sum takes as
long on a grid that fills few SMs as on one that fills them all; with blocks of 64
threads on the small one it took 1.13 times that (174 us against 154).
"""
import pytest

pytestmark = pytest.mark.gpu


def test_small_grid_costs_no_more_than_a_large_one():
    from paper_0712_2247_gb300 import lbif

    def ball_ms(h):
        with lbif.Slit(97, 3, h, 18, 0.15, 0.9) as g:
            g.step(2)
            return min(g.step_profiled(6)[0]["ball_g2"] for _ in range(6))

    assert ball_ms(3) < 1.07 * ball_ms(155)
