"""GPU path: the host's copy of the grid and counter, and blocks kept between
stages of different shapes (requires a GB300)."""
import numpy as np
import pytest

from paper_1503_06182_gb300 import vegas as v
from paper_1503_06182_gb300.workloads import DY_PARAMS

pytestmark = pytest.mark.gpu
UNIFORM = np.tile(np.arange(51) / 50, (4, 1))


def make(**kw):
    return v.Vegas(4, 50, 7, precision="fp32", **kw)


@pytest.mark.parametrize("graph", [0, 1])
def test_grid_follows_stages_and_uploads(graph):
    a, b = make(), make()
    try:
        for g in (a, b):
            g.set(v.VEGAS_OPT_GRAPH, graph)
        a.iterate(30_000, 3, v.VEGAS_DY, DY_PARAMS)
        b.launch(30_000, 3, v.VEGAS_DY, DY_PARAMS)
        assert np.array_equal(a.grid, b.grid) and not np.array_equal(a.grid, UNIFORM)
        saved = a.state()
        assert saved == b.state()
        # an upload right behind a stage that nobody waited for
        b.fetch(3)
        b.launch(30_000, 2, v.VEGAS_DY, DY_PARAMS)
        b.grid = UNIFORM
        assert np.array_equal(b.grid, UNIFORM)
        # a frozen stage keeps the grid
        b.set(v.VEGAS_OPT_ADAPT, 0)
        b.iterate(30_000, 1, v.VEGAS_DY, DY_PARAMS)
        assert np.array_equal(b.grid, UNIFORM)
        # a restored state continues alike, with captured stages kept
        a.iterate(30_000, 2, v.VEGAS_DY, DY_PARAMS)
        want, want_grid = a.iterate(30_000, 2, v.VEGAS_DY, DY_PARAMS)[3], a.grid
        for g in (a, b):
            g.restore(saved)
            g.iterate(30_000, 2, v.VEGAS_DY, DY_PARAMS)
            assert np.array_equal(g.iterate(30_000, 2, v.VEGAS_DY, DY_PARAMS)[3], want)
            assert np.array_equal(g.grid, want_grid)
    finally:
        a.close()
        b.close()


def test_grid_without_the_result_block():
    """More iterations than the mapped records hold: the grid still comes back."""
    a, b = make(), make()
    try:
        a.iterate(2000, 70, v.VEGAS_DY, DY_PARAMS)
        for _ in range(70):
            b.iterate(2000, 1, v.VEGAS_DY, DY_PARAMS)
        assert np.array_equal(a.grid, b.grid)
    finally:
        a.close()
        b.close()


def test_stratified_stages_of_alternating_sizes():
    """Stages of different call counts share one block: each starts from the
    uniform allocation and equals the stage of a fresh context."""
    a = make()
    try:
        a.set(v.VEGAS_OPT_STRAT, 1)
        for n in (40_000, 100_000, 40_000, 3_000, 100_000):
            state = a.state()
            got = a.iterate(n, 2, v.VEGAS_DY, DY_PARAMS)[3]
            s, counts, var = a.strat()
            b = make()
            try:
                b.set(v.VEGAS_OPT_STRAT, 1)
                b.restore(state)
                assert np.array_equal(b.iterate(n, 2, v.VEGAS_DY, DY_PARAMS)[3], got)
                s2, counts2, var2 = b.strat()
                assert s == s2 and np.array_equal(counts, counts2) and np.array_equal(var, var2)
            finally:
                b.close()
    finally:
        a.close()
