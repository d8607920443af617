"""GPU path: the grid refinement at the edges of its range of bins (requires a
GB300): each iteration's new edges against the oracle's refinement of the
GPU's own sums."""
import numpy as np
import pytest

import oracle
from paper_1503_06182_gb300 import vegas as v

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("alpha", [1.5, 0.0, 0.5, 1.0, 2.0, 0.7])
@pytest.mark.parametrize("ndim,nbins", [(1, 2), (2, 3), (3, 31), (2, 64), (2, 65), (5, 224),
                                        (3, 225), (2, 256), (2, 257), (2, 449), (1, 1024)])
def test_new_edges_equal_the_oracles(ndim, nbins, alpha):
    """The compressed shares agree to 2^-45 or better on either side, and a new
    edge moves by that fraction of its bin: below 1e-12."""
    g = v.Vegas(ndim, nbins, 3, alpha=alpha)
    try:
        for sigma in (0.1, 0.02):
            for _ in range(2):
                old = g.grid
                g.iterate(5000, 1, v.VEGAS_GAUSS, (sigma,))
                d = g.last_sums()[2:].reshape(ndim, nbins)
                want = oracle.refine(d, old, alpha)
                assert np.max(np.abs(g.grid - want)) < 1e-12
    finally:
        g.close()
