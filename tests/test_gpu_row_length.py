"""GPU path: a tile's sums do not depend on how many limbs its rows have
(requires a GB300).  A plain fill of up to 512 bins has 13, one with a histogram
9: the same events take one window of limbs in one and several in the other."""
import numpy as np
import pytest

from paper_1503_06182_gb300 import vegas as v

pytestmark = pytest.mark.gpu


def grid(wide, narrow):
    """Two axes of eight bins, seven of them of about the given width."""
    e = np.zeros((2, 9))
    for a, w in enumerate((wide, narrow)):
        e[a, 1:8] = np.cumsum(w * (1 + 0.09 * np.arange(7)))
        e[a, 8] = 1.0
    return e


@pytest.mark.parametrize("precision", ["fp64", "fp32"])
@pytest.mark.parametrize("wide,narrow", [
    # the squares' lowest digits: 12% of a bin's events at 2^-50 of the tile's
    # largest weight, the others 2^-21 below those, one limb under nine limbs' window
    (1.2 * 2.0 ** -50, 1.3 * 2.0 ** -22), (1.1 * 2.0 ** -50, 2.0 ** -20),
    (1.5 * 2.0 ** -48, 2.0 ** -24), (1.3 * 2.0 ** -52, 2.0 ** -18),
])
def test_a_histogram_leaves_the_sums_unchanged(wide, narrow, precision):
    """Bit for bit, over many samples: a carry out of the digits that a bin drops
    moves its sum by some 2^-64, which one rounding in about 2000 shows."""
    ctx = []
    for hist in (0, 5):
        g = v.Vegas(2, 8, 3, precision=precision)
        g.set(v.VEGAS_OPT_ADAPT, 0)
        g.grid = grid(wide, narrow)
        if hist:
            g.hist_set(hist, 0.0, 1.0)
        ctx.append(g)
    differ = 0
    try:
        for _ in range(3000):  # a Gaussian so wide that the weight is the Jacobian
            sums = []
            for g in ctx:
                g.iterate(100_000, 1, v.VEGAS_GAUSS, (1e6,))
                sums.append(g.last_sums()[:18])
            differ += not np.array_equal(*sums)
    finally:
        for g in ctx:
            g.close()
    assert differ == 0
