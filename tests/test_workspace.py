"""The workspace a caller sizes for a stage serves every smaller stage: the
tile counts it is sized by (gv_tiles.cuh on the host), and on the GPU stages of
fewer calls in a caller's buffer."""
import ctypes as C
import os
import random
import subprocess

import pytest

from paper_1503_06182_gb300.workloads import DY_PARAMS

CSRC = os.path.join(os.path.dirname(os.path.dirname(os.path.abspath(__file__))),
                    "paper_1503_06182_gb300", "csrc")
WRAP = r"""
#include "gv_tiles.cuh"
extern "C" {
long long count(long long n, int form) { return gv_tile_count(n, form); }
long long most(long long n, int form) { return gv_most_tiles(n, form); }
// the first n in [1, last] whose gv_most_tiles is not the largest count so far, or 0
long long check(long long last, int form) {
  long long m = 0;
  for (long long n = 1; n <= last; ++n) {
    m = std::max(m, gv_tile_count(n, form));
    if (m != gv_most_tiles(n, form)) return n;
  }
  return 0;
}
}
"""


@pytest.fixture(scope="module")
def lib(tmp_path_factory):
    d = tmp_path_factory.mktemp("tiles")
    src, so = d / "t.cpp", d / "t.so"
    src.write_text(WRAP)
    subprocess.run(["g++", "-O2", "-std=c++17", "-shared", "-fPIC", "-I", CSRC, str(src), "-o",
                    str(so)], check=True)
    L = C.CDLL(str(so))
    for f in (L.count, L.most, L.check):
        f.restype, f.argtypes = C.c_longlong, [C.c_longlong, C.c_int]
    return L


@pytest.mark.parametrize("form", [0, 1, 2])  # FP64 pipe, FP32, 64-bit significands
def test_most_tiles_is_the_largest_count(lib, form):
    assert lib.check(700_000, form) == 0
    r = random.Random(2)
    for _ in range(300):  # beyond the listed multiples, and around their end
        n = r.choice([r.randint(700_000, 8_000_000), r.randint(3_700_000, 3_800_000),
                      r.randint(1, 1 << 40)])
        m = r.randint(1, n)
        assert lib.count(m, form) <= lib.most(m, form) <= lib.most(n, form)
        if n > 25 * 152 * 1024:
            assert lib.most(n, form) == -(-n // 1024)


@pytest.mark.gpu
@pytest.mark.parametrize("precision", ["fp64", "fp32"])
@pytest.mark.parametrize("ncall,smaller", [
    (100_000, [100_000, 77_824, 77_825, 19_456, 19_457, 2]), (20_000, [19_332, 19_456, 20_000]),
    (1_500_000, [1_500_000, 1_410_000, 1_400_000, 311_296, 155_649])])
def test_a_workspace_serves_every_smaller_stage(ncall, smaller, precision):
    torch = pytest.importorskip("torch")
    from paper_1503_06182_gb300 import vegas as v
    g = v.Vegas(4, 100, 3, precision=precision)
    try:
        nbytes = v.vegas_workspace_size(g.h, ncall, 3)
        buf = torch.empty(nbytes, dtype=torch.uint8, device="cuda")
        v.vegas_set_workspace(g.h, buf.data_ptr(), nbytes)
        for n in smaller:
            assert g.iterate(n, 3, v.VEGAS_DY, DY_PARAMS)[1] >= 0
            assert g.adjoint(n, 2, DY_PARAMS)[3] >= 0
    finally:
        g.close()
