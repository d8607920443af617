"""GPU path: the tile's limb sums at the edges of their windows (requires a
GB300).  Weights over hundreds of binades take several windows per tile, and
the number of bins chooses the row length (9, 7 or 5 limbs)."""
import math
from fractions import Fraction

import numpy as np
import pytest

from paper_1503_06182_gb300 import vegas as v

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("precision", ["fp64", "fp32"])
@pytest.mark.parametrize("ndim,nbins,ncall,sigma", [
    (2, 7, 3000, 0.028),     # nine limbs, weights down to 2^-460
    (1, 2, 1025, 0.02),      # two bins, two events past a tile
    (4, 256, 1024, 0.05),    # 1024 bins: the last shape of nine limbs
    (3, 342, 1023, 0.034),   # 1026 bins: seven limbs
    (4, 1024, 1500, 0.05),   # five limbs
    (5, 50, 2049, 0.1),      # bins in shared memory
    (16, 256, 1100, 0.3),    # the largest shape
])
def test_sums_equal_the_exact_sums_of_the_weights(ndim, nbins, ncall, sigma, precision):
    """The sums against exact rational sums of the events' own weights (which
    vegas_eval_events returns in full).  A sum is rounded once to FP64 (2^-53);
    before that a tile drops at most 2^-62 of each square and 2^-66 of a bin's
    sum, and the weights' sum at most 2^-96 of the tile's largest weight."""
    g = v.Vegas(ndim, nbins, 11, precision=precision)
    try:
        w, bins = g.eval_events(v.VEGAS_GAUSS, (sigma,), 0, np.arange(ncall))
        g.iterate(ncall, 1, v.VEGAS_GAUSS, (sigma,))
        sums = g.last_sums()
    finally:
        g.close()
    exact = [Fraction(x) for x in w]
    squares = [x * x for x in exact]
    want = np.zeros(2 + ndim * nbins)
    want[0], want[1] = float(sum(exact)), float(sum(squares))
    rows = [Fraction(0)] * (ndim * nbins)
    for e, row in enumerate(bins):
        for a, b in enumerate(row):
            rows[a * nbins + b] += squares[e]
    want[2:] = [float(r) for r in rows]
    assert np.array_equal(sums == 0, want == 0)
    assert np.all(np.abs(sums - want) <= 2.0 ** -52 * want)


def test_wide_weights_identical_across_launch_shapes():
    """Several windows per tile: the same bits for every block size and in a
    batch."""
    params, ncall = (0.028,), 3000
    outs = []
    for ept in (1, 2, 4, 8):
        g = v.Vegas(2, 50, 11, precision="fp32")
        try:
            g.set(v.VEGAS_OPT_EPT, ept)
            outs.append((g.iterate(ncall, 3, v.VEGAS_GAUSS, params)[3], g.grid))
        finally:
            g.close()
    B = v.VegasBatch([(2, ncall, v.VEGAS_GAUSS, params)], 50, 11, precision="fp32")
    try:
        outs.append((B.iterate(3)[3][0], B.grid(0)))
    finally:
        B.close()
    for per, grid in outs[1:]:
        assert np.array_equal(per, outs[0][0]) and np.array_equal(grid, outs[0][1])


@pytest.mark.parametrize("precision", ["fp64", "fp32"])
@pytest.mark.parametrize("ncall", [2, 127, 128, 129, 19456, 19457, 38913, 77824, 100_001])
def test_sums_at_the_edges_of_the_tile_sizes(ncall, precision):
    """Every tile size and its last, partly filled tile: the sums against sums
    of the events' own weights, rounded once (math.fsum; the squares' own
    roundings add 2^-53), and the same bits for every block size."""
    p = (0.1, 0.1)  # weights of both signs
    sums = []
    for ept in (1, 2, 4, 8):
        g = v.Vegas(3, 40, 11, precision=precision)
        try:
            g.set(v.VEGAS_OPT_EPT, ept)
            g.iterate(ncall, 1, v.VEGAS_GAUSS, p)
            sums.append(g.last_sums())
            if ept == 8:
                g.grid = np.tile(np.arange(41) / 40, (3, 1))
                w, bins = g.eval_events(v.VEGAS_GAUSS, p, 0, np.arange(ncall))
        finally:
            g.close()
    assert all(np.array_equal(s, sums[0]) for s in sums[1:])
    w2 = w * w
    scale = math.fsum(np.abs(w))
    assert abs(sums[0][0] - math.fsum(w)) <= 2.0 ** -52 * scale
    assert abs(sums[0][1] - math.fsum(w2)) <= 2.0 ** -51 * sums[0][1]
    for a in range(3):
        for b in range(40):
            want = math.fsum(w2[bins[:, a] == b])
            assert abs(sums[0][2 + 40 * a + b] - want) <= 2.0 ** -51 * want
