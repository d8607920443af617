"""GPU path: stages that a caller captured in a CUDA graph of its own and
replays, and grids set between them (requires a GB300)."""
import numpy as np
import pytest

from paper_1503_06182_gb300 import vegas as v
from paper_1503_06182_gb300.workloads import DY_PARAMS

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu
UNIFORM = np.tile(np.arange(51) / 50, (4, 1))


def make(stream, **kw):
    g = v.Vegas(4, 50, 7, precision="fp32", stream=stream, **kw)
    g.set(v.VEGAS_OPT_GRAPH, 0)
    g.set(v.VEGAS_OPT_EPT, 4)
    return g


@pytest.mark.parametrize("ncall,replays", [(5_000, 2), (50_000, 3)])
def test_the_counter_and_the_grid_follow_replays(ncall, replays):
    """After r replays of a captured stage the state is that of r stages, and a
    grid set right behind a replay is the one that stays."""
    s = torch.cuda.Stream()
    a, b = make(s.cuda_stream), make(None)
    try:
        for g in (a, b):
            g.iterate(ncall, 2, v.VEGAS_DY, DY_PARAMS)
        graph = torch.cuda.CUDAGraph()
        with torch.cuda.graph(graph, stream=s, capture_error_mode="thread_local"):
            a.launch(ncall, 2, v.VEGAS_DY, DY_PARAMS)
        with torch.cuda.stream(s):
            for _ in range(replays):
                graph.replay()
        for _ in range(replays):
            per = b.iterate(ncall, 2, v.VEGAS_DY, DY_PARAMS)[3]
        s.synchronize()
        assert a.state() == b.state()
        assert np.array_equal(a.fetch(2)[3], per)
        for _ in range(5):
            with torch.cuda.stream(s):
                graph.replay()
            a.grid = UNIFORM
            assert np.array_equal(a.grid, UNIFORM)
        s.synchronize()
        assert np.array_equal(a.grid, UNIFORM)
        b.restore(a.state())
        for g in (a, b):
            g.set(v.VEGAS_OPT_ADAPT, 0)
        assert np.array_equal(a.iterate(ncall, 1, v.VEGAS_DY, DY_PARAMS)[3],
                              b.iterate(ncall, 1, v.VEGAS_DY, DY_PARAMS)[3])
    finally:
        a.close()
        b.close()


def test_grids_follow_one_another():
    """Grids set in a row, on the legacy stream and across a change of stream: the
    events see the last one."""
    s = torch.cuda.Stream()
    r = np.random.default_rng(3)
    grids = [np.concatenate([np.zeros((4, 1)), np.sort(r.random((4, 49))), np.ones((4, 1))], axis=1)
             for _ in range(6)]
    a, b = make(0), make(None)
    try:
        for k, e in enumerate(grids):
            for f in (UNIFORM, grids[k - 1], e):
                a.grid = f
            if k % 2:
                v.vegas_set_stream(a.h, s.cuda_stream if k % 4 == 1 else 0)
            b.grid = e
            ev = np.arange(500)
            assert np.array_equal(a.grid, e)
            wa, wb = (g.eval_events(v.VEGAS_DY, DY_PARAMS, k, ev)[0] for g in (a, b))
            assert np.array_equal(wa, wb)
    finally:
        a.close()
        b.close()
