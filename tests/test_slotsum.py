"""The reduce's slot sums (gv_slotsum.cuh) compiled for the host: the same bits
for every order and grouping of the tiles, and the value of the kept digits."""
import ctypes as C
import os
import random
import subprocess
from fractions import Fraction

import pytest

CSRC = os.path.join(os.path.dirname(os.path.dirname(os.path.abspath(__file__))),
                    "paper_1503_06182_gb300", "csrc")
WRAP = r"""
#include "gv_slotsum.cuh"
extern "C" {
// parts: 4 words each; thread t of nthr takes every nthr-th of them, `load` at a
// time, and the threads' sums are joined as the kernels do
int sum(const unsigned* v, const int* pos, int n, int nthr, int load, unsigned long long* window,
        int* sticky, int* e, int* neg) {
  GvAcc all = acc_zero();
  for (int t = 0; t < nthr; ++t) {
    GvAcc a = acc_zero();
    for (int i0 = t; i0 < n; i0 += nthr * load) {
      int top = 0;
      for (int i = i0; i < n && i < i0 + nthr * load; i += nthr)
        if (pos[i] > top) top = pos[i];
      if ((top >> 5) > a.g) acc_raise(a, top >> 5);
      for (int i = i0; i < n && i < i0 + nthr * load; i += nthr)
        if (pos[i]) {
          const int o = a.g - (pos[i] >> 5);
          (o <= 1 ? acc_add_near : acc_add_far)(a, v[4 * i], v[4 * i + 1], v[4 * i + 2],
                                                v[4 * i + 3], pos[i], o);
        }
    }
    const int g = a.g > all.g ? a.g : all.g;
    if (t & 1) {
      acc_raise(a, g);
      acc_raise(all, g);
      for (int j = 0; j < GV_SLOT_WORDS; ++j) all.w[j] += a.w[j];
    } else {
      GvAcc r;
      for (int j = 0; j < GV_SLOT_WORDS; ++j)
        r.w[j] = acc_word(a.w, 1, a.g, g, j) + acc_word(all.w, 1, all.g, g, j);
      r.g = g;
      all = r;
    }
  }
  bool s = false, m = false;
  const bool any = acc_window(all, window, &s, e, &m);
  *sticky = s;
  *neg = m;
  return any;
}
// the window known first
int sum_fixed(const unsigned* v, const int* pos, int n, unsigned long long* window, int* sticky,
              int* e, int* neg) {
  int g = 0;
  for (int i = 0; i < n; ++i)
    if ((pos[i] >> 5) > g) g = pos[i] >> 5;
  GvAccFixed a = {{0u, 0u, 0u, 0u, 0u, 0u}};
  for (int i = 0; i < n; ++i)
    if (pos[i]) acc_add_fixed(a, v[4 * i], v[4 * i + 1], v[4 * i + 2], v[4 * i + 3], pos[i], g);
  unsigned long long q[4];
  for (int j = 0; j < 3; ++j)
    q[j] = a.w[2 * j] | ((unsigned long long)a.w[2 * j + 1] << 32);
  q[3] = (unsigned long long)((long long)q[2] >> 63);
  bool s = false, m = false;
  const bool any = acc_leading(q, g, window, &s, e, &m);
  *sticky = s;
  *neg = m;
  return any;
}
}
"""


@pytest.fixture(scope="module")
def total(tmp_path_factory):
    d = tmp_path_factory.mktemp("slots")
    src, so = d / "s.cpp", d / "s.so"
    src.write_text(WRAP)
    subprocess.run(["g++", "-O1", "-std=c++17", "-shared", "-fPIC", "-I", CSRC, str(src), "-o",
                    str(so)], check=True)
    L = C.CDLL(str(so))

    def run(parts, nthr, load):
        """(window, sticky, exponent, sign) of the sum, or None for zero."""
        n = len(parts)
        v = (C.c_uint * (4 * n))(*[(x >> (32 * j)) & 0xFFFFFFFF for x, _ in parts for j in range(4)])
        pos = (C.c_int * n)(*[p for _, p in parts])
        w, s, e, m = C.c_ulonglong(), C.c_int(), C.c_int(), C.c_int()
        out = (C.byref(w), C.byref(s), C.byref(e), C.byref(m))
        any_ = L.sum(v, pos, n, nthr, load, *out) if nthr else L.sum_fixed(v, pos, n, *out)
        return (w.value, s.value, e.value, m.value) if any_ else None

    return run


def kept(parts):
    """The rule, in Python: digits at multiples of 32 bits, the top one signed;
    those more than one position below the highest partial's lowest digit drop."""
    g = max(p >> 5 for _, p in parts)
    out = 0
    for x, p in parts:
        if p == 0:
            continue
        y, q = x << (p & 31), p >> 5
        cut = max(0, min(g - 1 - q, 5))
        if cut < 5:
            out += (y >> (32 * cut)) << (32 * (q + cut))
    return out


CASES = {
    # a bin's sums of w^2 (up to 99 bits), 22-bit steps; a histogram's sums of w
    # of both signs; a channel's (up to 127 bits), any step
    "bins": lambda r: (r.getrandbits(r.randint(66, 99)), 156 + 22 * r.randint(90, 93)),
    "bins_wide": lambda r: (r.getrandbits(r.randint(66, 99)), 156 + 22 * r.randint(0, 190)),
    "hist": lambda r: (r.choice([-1, 1]) * r.getrandbits(r.randint(1, 95)), r.randint(900, 1100)),
    "channel": lambda r: (r.choice([-1, 1]) * r.getrandbits(r.randint(1, 127)),
                          r.randint(1200, 1240)),
    "one": lambda r: (r.getrandbits(96), 2000),
}


@pytest.mark.parametrize("kind", list(CASES))
@pytest.mark.parametrize("n", [1, 2, 9, 79, 300])
def test_every_order_gives_the_same_bits(total, kind, n):
    r = random.Random(n)
    for _ in range(20):
        parts = [CASES[kind](r) if r.random() < 0.9 else (0, 0) for _ in range(n)]
        if all(p == 0 for _, p in parts):
            continue
        want = kept(parts)
        outs = set()
        for nthr, load in ((0, 0), (1, 1), (8, 4), (32, 8), (256, 8), (3, 2)):
            for _ in range(2):
                outs.add(total(parts, nthr, load))
                r.shuffle(parts)
        assert len(outs) == 1
        got = outs.pop()
        if want == 0:
            assert got is None
            continue
        w, sticky, e, neg = got
        mag = abs(want)
        bits = mag.bit_length()
        assert neg == (want < 0) and w >> 63 == 1
        assert w == (mag >> (bits - 64) if bits >= 64 else mag << (64 - bits))
        assert bool(sticky) == (bits > 64 and mag & ((1 << (bits - 64)) - 1) != 0)
        assert e == bits - 1 - 2400


def test_what_is_dropped_is_small(total):
    """At least 32 bits below the largest partial's lowest one are kept: of 300
    partials at most 300 units there."""
    r = random.Random(5)
    for _ in range(200):
        parts = [CASES["bins_wide"](r) for _ in range(300)]
        exact = sum(Fraction(x) * Fraction(2) ** p for x, p in parts)
        lost = exact - kept(parts)
        assert 0 <= lost < 300 * Fraction(2) ** (max(p for _, p in parts) - 32)


@pytest.mark.gpu
@pytest.mark.parametrize("precision", ["fp64", "fp32"])
def test_batch_and_single_contexts_agree_bit_for_bit(precision):
    """Members of 2 to 2000 tiles whose weights span hundreds of binades, so that
    a bin's partials differ by many digits: a batch (two-level reduce over tile
    ranges) and single contexts (clusters, or a CTA per slot)."""
    np = pytest.importorskip("numpy")
    from paper_1503_06182_gb300 import vegas as v
    members = [(2, 257, v.VEGAS_GAUSS, (0.03,)), (2, 9_999, v.VEGAS_GAUSS, (0.03,)),
               (3, 77_824, v.VEGAS_GAUSS, (0.05,)), (2, 300_001, v.VEGAS_GAUSS, (0.03,)),
               (1, 1_000_000, v.VEGAS_GAUSS, (0.02,)), (2, 2_050_000, v.VEGAS_GAUSS, (0.04,))]
    B = v.VegasBatch(members, 12, 5, precision=precision)
    try:
        per = B.iterate(3)[3]
        grids = [B.grid(i) for i in range(len(members))]
    finally:
        B.close()
    for i, (d, n, iid, p) in enumerate(members):
        g = v.Vegas(d, 12, 5, precision=precision)
        try:
            g.set(v.VEGAS_OPT_BATCH_ID, i)
            assert np.array_equal(g.iterate(n, 3, iid, p)[3], per[i])
            assert np.array_equal(g.grid, grids[i])
        finally:
            g.close()
