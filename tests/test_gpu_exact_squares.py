"""GPU path: the FP64 form's sum of squares holds the squares' full 106 bits
(requires a GB300)."""
from fractions import Fraction

import numpy as np
import pytest

from paper_1503_06182_gb300 import vegas as v
from paper_1503_06182_gb300.workloads import DY_PARAMS

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("stage", ["plain", "hist", "pipe"])
def test_the_sum_of_squares_is_rounded_once(stage):
    """Stages of two events against exact rational sums of their weights, correctly
    rounded: the tile drops less than 2^-90 of the sum, so the roundings agree but
    once in 2^37.  (With 64 bits of each square, one in some 4000 did not.)"""
    ncall = 2
    p = list(DY_PARAMS)
    if stage == "pipe":
        p[9] = 2.0 ** -100  # beyond gv_x64_applies: the FP64 pipe
    g = v.Vegas(4, 16, 9)
    differ = 0
    try:
        g.set(v.VEGAS_OPT_ADAPT, 0)
        g.set(v.VEGAS_OPT_EPT, 4)
        if stage == "hist":
            g.hist_set(8, 60.0, 120.0)
        for it in range(12_000):
            w, _ = g.eval_events(v.VEGAS_DY, p, it, np.arange(ncall))
            g.iterate(ncall, 1, v.VEGAS_DY, p)
            s = g.last_sums()
            exact = [Fraction(x) for x in w]
            differ += s[0] != float(sum(exact)) or s[1] != float(sum(x * x for x in exact))
    finally:
        g.close()
    assert differ == 0
