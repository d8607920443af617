"""GPU path: the histogram's limbs with and without their copies (requires a
GB300)."""
import numpy as np
import pytest

from paper_1503_06182_gb300 import vegas as v
from paper_1503_06182_gb300.workloads import DY_PARAMS

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("precision", ["fp32", "fp64"])
@pytest.mark.parametrize("nh", [1, 6, 7, 100, 160, 161, 250, 1000])
@pytest.mark.parametrize("ndim,nbins,ncall", [(4, 100, 50_001), (4, 50, 777), (16, 60, 20_000)])
def test_histogram_sums_add_up(ndim, nbins, ncall, nh, precision):
    """Every event falls into one of the nh + 2 bins: their sums of w and of w^2
    add up to the iteration's (all weights are positive; at most 1002 values,
    each rounded once: 1002 x 2^-53 = 1.2e-13), the same for every block size."""
    outs = []
    for ept in (2, 4):
        g = v.Vegas(ndim, nbins, 5, precision=precision)
        try:
            g.set(v.VEGAS_OPT_EPT, ept)
            g.hist_set(nh, 70.0, 110.0)
            g.iterate(ncall, 2, v.VEGAS_DY, DY_PARAMS)
            last = np.array(g.hist()[2])
            sums = g.last_sums()
        finally:
            g.close()
        assert last.shape == (2, nh + 2)
        assert np.all(np.abs(last.sum(axis=1) - sums[:2]) <= 1.2e-13 * sums[:2])
        outs.append(last)
    assert np.array_equal(outs[0], outs[1])
