"""GPU path: edges that the shapes of other tests miss (requires a GB300): the
reduce's 256 and 257 tiles (stratified stages alone reach them) and plain
stages on either side, the bins at which rows get shorter, and a histogram's
bins one by one, with one copy of their limbs and with four, over several
windows and both signs."""
import math
from fractions import Fraction

import numpy as np
import pytest

import oracle
from paper_1503_06182_gb300 import vegas as v

pytestmark = pytest.mark.gpu


def calls_for(tiles):
    """The most calls of a stratified stage on two axes with that many tiles."""
    n = tiles * 1024
    while -(-(n + 2 * oracle.plus_nstrat(2, n) ** 2) // 1024) > tiles:
        n -= 1
    return n


@pytest.mark.parametrize("precision", ["fp64", "fp32"])
@pytest.mark.parametrize("tiles", [255, 256, 257])
def test_stratified_stages_around_256_tiles(tiles, precision):
    """One iteration against the oracle: the estimate and the grid to 1e-12 in
    FP64 (the same weights to some 2^-50, in sums of one sign); in FP32 the
    weights carry 2^-21, a bin's share half of that twice over, and an edge a
    like part of a bin."""
    ncall, p = calls_for(tiles), (0.2,)
    tol = 1e-12 if precision == "fp64" else 1e-5
    g = v.Vegas(2, 30, 5, precision=precision)
    try:
        g.set(v.VEGAS_OPT_STRAT, 1)
        per = g.iterate(ncall, 1, v.VEGAS_GAUSS, p)[3]
        grid = g.grid
    finally:
        g.close()
    ref = oracle.iterate_plus(2, 30, 5, ncall, 1, v.VEGAS_GAUSS, p)
    assert abs(per[0, 0] - ref.per_iter[0, 0]) <= tol * ref.per_iter[0, 0]
    assert np.max(np.abs(grid - ref.edges)) <= tol


@pytest.mark.parametrize("precision", ["fp64", "fp32"])
@pytest.mark.parametrize("ndim,nbins,ncall,sigma", [
    (1, 7, 155_648, 0.02), (1, 7, 155_649, 0.02),  # 152 tiles, and the next count
    (2, 256, 3001, 0.03),   # 512 bins: the last shape of 13 limbs
    (3, 171, 3001, 0.04),   # 513 bins: nine
    (1, 1024, 3001, 0.02),  # 1024 bins: the last of nine
    (5, 205, 2050, 0.1),    # 1025: seven
    (2, 1024, 3001, 0.03),  # 2048: the last of seven, and of the 64-bit significands
    (3, 683, 3001, 0.04),   # 2049: five, the FP64 pipe
])
def test_sums_where_the_rows_get_shorter(ndim, nbins, ncall, sigma, precision):
    """Against exact rational sums of the events' own weights: rounded once
    (2^-53), and a bin's digits below the kept ones (2^-66 of its largest square
    per event)."""
    g = v.Vegas(ndim, nbins, 11, precision=precision)
    try:
        w, bins = g.eval_events(v.VEGAS_GAUSS, (sigma,), 0, np.arange(ncall))
        g.iterate(ncall, 1, v.VEGAS_GAUSS, (sigma,))
        sums = g.last_sums()
    finally:
        g.close()
    if ncall <= 5000:
        exact = [Fraction(x) for x in w]
        squares = [x * x for x in exact]
        rows = [Fraction(0)] * (ndim * nbins)
        for e, row in enumerate(bins):
            for a, b in enumerate(row):
                rows[a * nbins + b] += squares[e]
        want = np.array([float(sum(exact)), float(sum(squares))] + [float(r) for r in rows])
        tol = 2.0 ** -52
    else:
        w2 = w * w  # (each rounded: 2^-53 more)
        want = np.array([math.fsum(w), math.fsum(w2)] +
                        [math.fsum(w2[bins[:, a] == b]) for a in range(ndim) for b in range(nbins)])
        tol = 2.0 ** -51
    assert np.array_equal(sums == 0, want == 0)
    assert np.all(np.abs(sums - want) <= tol * want)


@pytest.mark.parametrize("precision", ["fp64", "fp32"])
@pytest.mark.parametrize("shift", [0.0, 2.0 ** -40, 0.3])
@pytest.mark.parametrize("nh", [2, 16, 64, 128, 256, 512])
def test_every_histogram_bin(nh, shift, precision):
    """A histogram of x_0 that divides it as the uniform grid does (powers of two:
    the same bin for the same event, exactly), each bin's sums of w and w^2 against
    exact sums.  Of w a bin drops less than two units of 2^-63 of its largest |w|
    per event; its sum of w^2 is the grid bin's, bit for bit."""
    ncall, p = 3001, (0.02, shift)
    g = v.Vegas(1, nh, 11, precision=precision)
    try:
        g.hist_set(nh, 0.0, 1.0)
        w, bins = g.eval_events(v.VEGAS_GAUSS, p, 0, np.arange(ncall))
        g.iterate(ncall, 1, v.VEGAS_GAUSS, p)
        got = np.array(g.hist()[2])
        rows = g.last_sums()[2:2 + nh]
    finally:
        g.close()
    exact = [Fraction(x) for x in w]
    assert got[0, 0] == got[0, -1] == 0.0
    for b in range(nh):
        mine = [exact[e] for e in np.flatnonzero(bins[:, 0] == b)]
        s1, s2 = sum(mine, Fraction(0)), sum((x * x for x in mine), Fraction(0))
        top = max((abs(x) for x in mine), default=Fraction(0))
        lost = 2 * len(mine) * top * Fraction(2) ** -63
        assert abs(Fraction(got[0, b + 1]) - s1) <= abs(s1) * Fraction(2) ** -52 + lost
        assert abs(Fraction(got[1, b + 1]) - s2) <= s2 * Fraction(2) ** -52
        assert got[1, b + 1] == rows[b]
