"""The 64-bit-significand form where a value reaches 1, the end of its
fractions: the header on the host, and on the GPU grids with a bin whose width
rounds to 1."""
import ctypes as C
import math
import os
import subprocess

import numpy as np
import pytest

from paper_1503_06182_gb300.workloads import DY_PARAMS

mpmath = pytest.importorskip("mpmath")
from mpmath import mp, mpf  # noqa: E402

CSRC = os.path.join(os.path.dirname(os.path.dirname(os.path.abspath(__file__))),
                    "paper_1503_06182_gb300", "csrc")
WRAP = r"""
#include "gv_xint.cuh"
extern "C" {
unsigned long long toq64(double x) { return x_to_q64(x_from(x)); }
// 1 - 2^-l for l = m 2^e, as the Drell-Yan weight forms it, in units of 2^-64
double oneminus(unsigned long long m, int e) {
  return x_to_double(x_one_minus(x_to_q64(x_exp2(m, e, true)))) * 0x1p64;
}
}
"""


@pytest.fixture(scope="module")
def lib(tmp_path_factory):
    d = tmp_path_factory.mktemp("x64e")
    src, so = d / "x.cpp", d / "x.so"
    src.write_text(WRAP)
    subprocess.run(["g++", "-O1", "-std=c++17", "-shared", "-fPIC", "-I", CSRC, str(src), "-o",
                    str(so)], check=True)
    L = C.CDLL(str(so))
    L.toq64.restype, L.oneminus.restype = C.c_ulonglong, C.c_double
    return L


def test_fractions_up_to_one(lib):
    """Exact below 1; 1 is the largest fraction."""
    for x in (0.5, 0.75, 1.0 - 2.0 ** -53, 2.0 ** -53, 2.0 ** -64, 0.3):
        assert lib.toq64(C.c_double(x)) == math.floor(x * 2.0 ** 64)
    assert lib.toq64(C.c_double(1.0)) == 2 ** 64 - 1
    assert lib.toq64(C.c_double(2.0 ** -65)) == 0


@pytest.mark.parametrize("e", [-60, -63, -68, -72, -80])
@pytest.mark.parametrize("m", [1, 2, 100, 1000, 1 << 20])
def test_one_minus_a_momentum_fraction(lib, m, e):
    """1 - 2^-l for the smallest l (a mass window close to the total energy has
    e = -72): the exponential's documented 2^-59, which is 32 units of the
    fraction, and its truncation to one; never 0, and never near 2^64."""
    with mp.workprec(200):
        want = float((1 - mpf(2) ** (-mpf(m) * mpf(2) ** e)) * mpf(2) ** 64)
    got = lib.oneminus(C.c_ulonglong(m), e)
    assert 1.0 <= got and abs(got - want) <= 33.0 + 2.0 ** -50 * want


@pytest.mark.gpu
@pytest.mark.parametrize("first", [[1e-20], [1e-30, 2e-30], [2.0 ** -54], [2.0 ** -53], [0.5]])
@pytest.mark.parametrize("name,ndim,params", [("gauss", 2, (0.3,)), ("dy", 4, DY_PARAMS)])
def test_widths_that_round_to_one(name, ndim, params, first):
    """A valid grid whose last bin is as wide as the axis: the events' weights
    against the oracle (some 200 FP64 roundings of 2^-53 apart, below 1e-12
    where 1 - x is not smaller than 1/16), and the sums against them."""
    import oracle
    from paper_1503_06182_gb300 import vegas as v
    iid = {"gauss": v.VEGAS_GAUSS, "dy": v.VEGAS_DY}[name]
    oid = {"gauss": oracle.GAUSS, "dy": oracle.DY}[name]
    edges = np.tile(np.array([0.0] + first + [1.0]), (ndim, 1))
    nbins, n = edges.shape[1] - 1, 600
    g = v.Vegas(ndim, nbins, 7)
    try:
        g.grid = edges
        w, bins = g.eval_events(iid, params, 0, np.arange(n))
        g.set(v.VEGAS_OPT_ADAPT, 0)
        g.iterate(n, 1, iid, params)
        sums = g.last_sums()
    finally:
        g.close()
    checked = 0
    for e in range(n):
        want, b, x = oracle.event(oid, ndim, nbins, edges, params, 7, 0, 0, e)
        assert list(b) == list(bins[e])
        if name == "gauss" or 1 / 16 <= x[1] <= 15 / 16:
            assert abs(w[e] - want) <= 1e-12 * abs(want)
            checked += 1
    assert checked > 50
    assert abs(sums[0] - math.fsum(w)) <= 2.0 ** -50 * abs(sums[0])
