"""GPU path: numbers of bins whose refinement takes close to 48 KB of shared
memory, where a kernel has to ask for more (requires a GB300)."""
import numpy as np
import pytest

import oracle
from paper_1503_06182_gb300 import vegas as v
from paper_1503_06182_gb300.workloads import DY_PARAMS

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("nbins", [430, 450, 519, 525, 600, 608, 611, 613, 614, 615, 700, 1024])
def test_every_reduce_launches(nbins):
    """A stage of few tiles (clusters), one of more (a CTA per slot) and a batch
    (tile ranges): one iteration's estimate and grid against the oracle to 1e-12,
    and a gradient stage of more than 2048 tiles against the plain estimate."""
    for ncall in (3_000, 300_000):
        ref = oracle.iterate(2, nbins, 5, ncall, 1, oracle.GAUSS, (0.2,))
        g = v.Vegas(2, nbins, 5)
        B = v.VegasBatch([(2, ncall, v.VEGAS_GAUSS, (0.2,))], nbins, 5)
        try:
            per = g.iterate(ncall, 1, v.VEGAS_GAUSS, (0.2,))[3]
            bper = B.iterate(1)[3]
            assert np.allclose(per, ref.per_iter, rtol=1e-12, atol=0)
            assert np.max(np.abs(g.grid - ref.edges)) < 1e-12
            assert np.array_equal(np.asarray(bper).reshape(-1), per.reshape(-1))
            assert np.array_equal(B.grid(0), g.grid)
        finally:
            g.close()
            B.close()
    n = 2049 * 1024
    g = v.Vegas(4, nbins, 5, precision="fp32")
    try:
        g.set(v.VEGAS_OPT_ADAPT, 0)
        s = g.state()
        I = g.iterate(n, 1, v.VEGAS_DY, DY_PARAMS)[0]
        g.restore(s)
        assert abs(g.adjoint(n, 1, DY_PARAMS)[2] - I) <= 1e-12 * I
    finally:
        g.close()
