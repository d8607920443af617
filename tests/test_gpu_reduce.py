"""GPU path: the reduce over the tiles at the edges of its forms (requires a
GB300): one warp's lanes, the clusters' 256 tiles, the 128-bit sums' 2048, and
runs of more than 2048 tiles per thread."""
import math

import numpy as np
import pytest

from paper_1503_06182_gb300 import vegas as v

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("ncall", [
    2, 31 * 128, 32 * 128 + 1,                   # a warp's lanes
    255 * 1024, 256 * 1024, 256 * 1024 + 1,      # clusters, then a CTA per slot
    512 * 1024, 2048 * 1024, 2048 * 1024 + 1,    # 128-bit sums, then 192-bit
])
@pytest.mark.parametrize("ndim,nbins,sigma", [(1, 3, 0.02), (2, 40, 0.05)])
def test_sums_at_the_edges_of_the_forms(ncall, ndim, nbins, sigma):
    """Against sums of the events' own weights, rounded once (math.fsum; the
    squares' own roundings add 2^-53).  Weights over many binades: a bin's
    exponent differs from tile to tile."""
    g = v.Vegas(ndim, nbins, 11, precision="fp32")
    try:
        w, bins = g.eval_events(v.VEGAS_GAUSS, (sigma,), 0, np.arange(ncall))
        g.iterate(ncall, 1, v.VEGAS_GAUSS, (sigma,))
        sums = g.last_sums()
    finally:
        g.close()
    w2 = w * w
    want = [math.fsum(w), math.fsum(w2)]
    for a in range(ndim):
        order = np.argsort(bins[:, a], kind="stable")
        cut = np.searchsorted(bins[order, a], np.arange(nbins + 1))
        want += [math.fsum(w2[order[cut[b]:cut[b + 1]]]) for b in range(nbins)]
    want = np.array(want)
    assert np.all(np.abs(sums - want) <= 2.0 ** -52 * want)


def test_more_than_2048_tiles_per_thread():
    """6e8 events in 585938 tiles: each axis' bins add up to the sum of the
    squares (roundings: 2^-53 per value), which the integral's error also
    follows from."""
    ncall = 600_000_000
    g = v.Vegas(2, 2, 11, precision="fp32")
    try:
        I, s = g.iterate(ncall, 1, v.VEGAS_GAUSS, (0.2,))[:2]
        sums = g.last_sums()
    finally:
        g.close()
    rows = sums[2:].reshape(2, 2).sum(axis=1)
    assert np.all(np.abs(rows - sums[1]) <= 2.0 ** -51 * sums[1])
    # the integral of exp(-|x - 1/2|^2 / (2 sigma^2)) over the unit square
    exact = 2 * math.pi * 0.2 ** 2 * math.erf(0.5 / (0.2 * math.sqrt(2.0))) ** 2
    assert abs(I - exact) < 6 * s and s < 1e-3
