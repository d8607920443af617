"""GPU path: the FP64 form on 64-bit significands against the FP64 pipe, which
keeps parameters outside gv_x64_applies (requires a GB300).  Two parameter sets
on either side of the rule whose weights are equal up to an exact power of
two; single FP64 operations differ by 2^-53, some 200 of them per weight and
the logarithms' magnification by 2^4 stay below 1e-12."""
import numpy as np
import pytest

from paper_1503_06182_gb300 import vegas as v
from paper_1503_06182_gb300.workloads import DY_PARAMS, DYNLO_PARAMS, EE3J_PARAMS

pytestmark = pytest.mark.gpu


def with_n(params, n):
    return params[:9] + (n,) + params[10:]


CASES = {
    # densities' normalisation N: the weight is proportional to N^2
    "dy": (v.VEGAS_DY, with_n(DY_PARAMS, 2.0 ** -99), with_n(DY_PARAMS, 2.0 ** -100), 4.0),
    "dy_nlo": (v.VEGAS_DY_NLO, with_n(DYNLO_PARAMS, 2.0 ** -99), with_n(DYNLO_PARAMS, 2.0 ** -100),
               4.0),
    # the total energy cancels
    "ee3j": (v.VEGAS_EE3J, EE3J_PARAMS, (EE3J_PARAMS[0], 1e101), 1.0),
}


@pytest.mark.parametrize("ndim", [5, 13])
@pytest.mark.parametrize("name", list(CASES))
def test_both_arithmetics_agree(name, ndim):
    iid, inside, outside, ratio = CASES[name]
    outs = []
    for p in (inside, outside):
        g = v.Vegas(ndim, 30, 5)
        try:
            w, bins = g.eval_events(iid, p, 3, np.arange(0, 50_000, 23))
            g.hist_set(20, 0.6 if iid == v.VEGAS_EE3J else 60.0,
                       1.0 if iid == v.VEGAS_EE3J else 120.0)
            per = g.iterate(20_000, 1, iid, p)[3]
            outs.append((w, bins, per, g.last_sums(), g.hist()[2], g.grid))
        finally:
            g.close()
    a, b = outs
    assert np.array_equal(a[1], b[1]) and np.array_equal(a[0] == 0, b[0] == 0)
    assert np.allclose(a[0], ratio * b[0], rtol=1e-12, atol=0)
    assert np.allclose(a[2], ratio * b[2], rtol=1e-12, atol=0)
    sums = a[3] / np.where(np.arange(len(a[3])) == 0, ratio, ratio ** 2)
    assert np.allclose(sums, b[3], rtol=2e-12, atol=0)
    assert np.allclose(a[4] / np.array([[ratio], [ratio ** 2]]), b[4], rtol=2e-12, atol=0)
    assert np.allclose(a[5], b[5], rtol=0, atol=1e-12)


def test_both_arithmetics_agree_on_the_gradient():
    _, inside, outside, ratio = CASES["dy"]
    outs = []
    for p in (inside, outside):
        g = v.Vegas(4, 30, 5)
        try:
            g.set(v.VEGAS_OPT_ADAPT, 0)
            outs.append(g.adjoint(20_011, 2, p))
        finally:
            g.close()
    (ga, ea, Ia, _, _), (gb, eb, Ib, _, _) = outs
    assert np.all(np.abs(ga - ratio * gb) <= 1e-11 * (np.abs(ga) + ea))
    assert np.allclose(ea, ratio * eb, rtol=1e-10, atol=0) and abs(Ia / (ratio * Ib) - 1) < 1e-12


def test_batch_mixes_both_arithmetics():
    """A batch's members on either side of the rule equal their single
    contexts."""
    members = [(5, 3000, c[0], p) for c in (CASES["dy"], CASES["ee3j"]) for p in c[1:3]]
    B = v.VegasBatch(members, 30, 5)
    try:
        per = B.iterate(2)[3]
        for b, (d, n, iid, p) in enumerate(members):
            g = v.Vegas(d, 30, 5)
            g.set(v.VEGAS_OPT_BATCH_ID, b)
            try:
                assert np.array_equal(g.iterate(n, 2, iid, p)[3], per[b])
            finally:
                g.close()
    finally:
        B.close()
