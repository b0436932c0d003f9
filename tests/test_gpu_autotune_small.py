"""The autotuner on grids whose own segment length is below its candidates'.

The library cuts small grids into segments of two planes or so; forcing eight on them
leaves most SMs idle. The tuned pull pass may cost 1.25 times the default one (it
takes about 2 times with eight planes), and the default length stays a candidate.
"""
import pytest

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("n", [(32, 4, 64), (32, 32, 64), (40, 40, 64)])
@pytest.mark.parametrize("storage", [0, 1])
def test_tuned_is_not_slower(n, storage):
    from paper_0712_2247_gb300 import lbif

    def pull_ms(g):
        return min(g.step_profiled(10)[0]["collide_stream"] for _ in range(8))

    with lbif.Slit(*n, 4, 0.2, 0.9, storage=storage) as g:
        g.step(4)
        before = pull_ms(g)
        g.autotune(5)
        assert pull_ms(g) < 1.25 * before, g.shapes()
