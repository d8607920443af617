"""The 64-bit-significand arithmetic of the FP64 form (gv_x64.cuh, gv_xint.cuh)
compiled for the host and compared with 200-bit arithmetic."""
import ctypes as C
import math
import os
import random
import re
import subprocess
from fractions import Fraction

import pytest

mpmath = pytest.importorskip("mpmath")
from mpmath import mp, mpf  # noqa: E402

from paper_1503_06182_gb300.workloads import DY_PARAMS, DYNLO_PARAMS  # noqa: E402

CSRC = os.path.join(os.path.dirname(os.path.dirname(os.path.abspath(__file__))),
                    "paper_1503_06182_gb300", "csrc")
WRAP = r"""
#include "gv_xint.cuh"
extern "C" {
void mul(const GvX* a, const GvX* b, GvX* o) { *o = x_mul(*a, *b); }
void add(const GvX* a, const GvX* b, GvX* o) { *o = x_add(*a, *b); }
void rcp(const GvX* a, GvX* o) { *o = x_rcp(*a); }
void exp2x(const GvX* a, GvX* o) { *o = x_exp2(*a); }
void log2x(const GvX* a, GvX* o) { *o = x_log2(*a); }
void fromdouble(double a, GvX* o) { *o = x_from(a); }
double todouble(const GvX* a) { return x_to_double(*a); }
long long sqrtq(unsigned long long v) { return xi_sqrt_q62(v); }
void sincos(unsigned long long p, long long* s, long long* c) { x_sincos_turn(p, s, c); }
long long cosx(unsigned long long p) { return x_cos_turn(p); }
double gauss(const unsigned long long* x, int d, const GvX* K) {
  unsigned long long X[16] = {0};
  for (int i = 0; i < d; ++i) X[i] = x[i];
  return x_to_double(gv_gauss_x<16>(X, d, K));
}
double dy(const unsigned long long* x, const GvX* K, double* gr) {
  GvX g[5];
  const GvX r = gv_drell_yan_x<true>(x, K, g);
  for (int i = 0; i < 5; ++i) gr[i] = x_to_double(g[i]);
  return x_to_double(r);
}
double nlo(const unsigned long long* x, int d, const GvX* K) {
  unsigned long long X[16] = {0};
  for (int i = 0; i < d; ++i) X[i] = x[i];
  return x_to_double(gv_dy_nlo_x<16>(X, d, K));
}
double ee3j(const unsigned long long* x, const GvX* K) { return x_to_double(gv_ee3j_x(x, K)); }
}
"""


class X(C.Structure):
    _fields_ = [("m", C.c_uint64), ("e", C.c_int), ("s", C.c_uint)]

    @property
    def value(self):
        return (-1) ** self.s * mpf(self.m) * mpf(2) ** self.e


@pytest.fixture(scope="module")
def lib(tmp_path_factory):
    d = tmp_path_factory.mktemp("x64")
    src, so = d / "x.cpp", d / "x.so"
    src.write_text(WRAP)
    subprocess.run(["g++", "-O1", "-std=c++17", "-shared", "-fPIC", "-I", CSRC, str(src), "-o",
                    str(so)], check=True)
    L = C.CDLL(str(so))
    for f in ("todouble", "gauss", "dy", "nlo", "ee3j"):
        getattr(L, f).restype = C.c_double
    for f in ("sqrtq", "cosx"):
        getattr(L, f).restype = C.c_longlong
    with mp.workprec(200):
        yield L


def test_tables():
    text = open(os.path.join(CSRC, "gv_x64.cuh")).read()
    exp2 = re.search(r"gv_x_exp2_tab\[256\] = \{(.*?)\};", text, re.S).group(1)
    log2 = re.search(r"gv_x_log2_tab\[256\] = \{(.*?)\};", text, re.S).group(1)
    exp2 = [int(h, 16) for h in re.findall(r"0x([0-9a-f]+)ull", exp2)]
    log2 = [int(h, 16) for h in re.findall(r"0x([0-9a-f]+)ull", log2)]
    with mp.workprec(300):
        assert exp2 == [int(mp.floor(mpf(2) ** (mpf(j) / 256 + 63))) for j in range(256)]
        R = [int(mp.ceil(mpf(2) ** 31 / (1 + mpf(j) / 256))) for j in range(256)]
        assert log2[0::2] == R
        assert log2[1::2] == [int(mp.floor(-mp.log(mpf(r) / 2 ** 31, 2) * 2 ** 64)) for r in R]


def significand(r):
    return r.choice([r.getrandbits(63) | 1 << 63, (1 << 63) + r.getrandbits(r.randint(1, 40)),
                     (1 << 64) - 1 - r.getrandbits(r.randint(1, 60))])


def test_operations(lib):
    """Every operation and function within 2^-59 of its result (a sum: of the
    larger operand; sine, cosine and square root: absolute)."""
    r, o = random.Random(1), X()
    tol = mpf(2) ** -59
    for i in range(3000):
        a = X(significand(r), r.randint(-80, 20), r.getrandbits(1))
        b = X(significand(r), a.e + r.randint(-70, 70), r.getrandbits(1))
        if i % 3 == 0:  # cancellation
            b = X(a.m ^ r.getrandbits(r.randint(1, 60)), a.e, 1 - a.s)
        lib.mul(C.byref(a), C.byref(b), C.byref(o))
        assert abs(o.value / (a.value * b.value) - 1) < tol
        lib.add(C.byref(a), C.byref(b), C.byref(o))
        assert abs(o.value - (a.value + b.value)) <= tol * max(abs(a.value), abs(b.value))
        lib.rcp(C.byref(a), C.byref(o))
        assert o.m >> 63 and abs(o.value * a.value - 1) < tol
        t = X(significand(r), r.randint(-140, -54), r.getrandbits(1))
        lib.exp2x(C.byref(t), C.byref(o))
        assert o.m >> 63
        # the argument keeps 2^-64 of a unit: an absolute error of its fraction
        assert abs(o.value / mpf(2) ** t.value - 1) < tol
        p = X(significand(r), r.choice([-64, -63, -65, r.randint(-200, 100)]), 0)
        lib.log2x(C.byref(p), C.byref(o))
        want = mp.log(p.value, 2)
        assert abs(o.value - want) <= tol * max(1, abs(want))
        q = r.choice([r.getrandbits(64), r.getrandbits(20),
                      ((r.randint(0, 7) << 61) + r.randint(-5, 5)) % 2 ** 64])
        s, c = C.c_longlong(), C.c_longlong()
        lib.sincos(C.c_uint64(q), C.byref(s), C.byref(c))
        th = 2 * mp.pi * mpf(q) / mpf(2) ** 64
        assert abs(mpf(s.value) / 2 ** 62 - mp.sin(th)) < tol
        assert abs(mpf(c.value) / 2 ** 62 - mp.cos(th)) < tol
        assert lib.cosx(C.c_uint64(q)) == c.value
        v = r.choice([r.getrandbits(62), r.getrandbits(r.randint(1, 62)), 1 << 62])
        want = mp.sqrt(mpf(v) / 2 ** 62)
        assert abs(mpf(lib.sqrtq(C.c_uint64(v))) / 2 ** 62 - want) < tol
        # conversions: exact in, rounded to nearest even out (subnormals too)
        d = r.uniform(-1, 1) * 2.0 ** r.randint(-1070, 1020)
        lib.fromdouble(C.c_double(d), C.byref(o))
        assert lib.todouble(C.byref(o)) == d
        w = X(significand(r), r.choice([r.randint(-1100, 950), r.randint(-1140, -1070)]), 0)
        assert lib.todouble(C.byref(w)) == float(Fraction(w.m) * Fraction(2) ** w.e)
    big = X(1 << 63, 961, 1)
    assert lib.todouble(C.byref(big)) == -math.inf
    one = X(1 << 63, -63, 0)
    for e in (-200, -64, -63, 0):
        a = X(1 << 63, e, 0)
        lib.rcp(C.byref(a), C.byref(o))
        assert abs(o.value * a.value - 1) < tol
    huge = X(1 << 63, -40, 1)  # 2^-(2^23): zero
    lib.exp2x(C.byref(huge), C.byref(o))
    assert o.m == 0 and one.value == 1


def xc(v):
    """A real number as GvX (rounded down)."""
    v = mpf(v)
    if v == 0:
        return X(0, -(1 << 20), 0)
    s, v = (1, -v) if v < 0 else (0, v)
    e = int(mp.floor(mp.log(v, 2))) - 63
    return X(int(mp.floor(v * mpf(2) ** -e)), e, s)


def dy_constants(p):
    """The double constants of the Drell-Yan weight, and the GvX array in
    gv_xint.cuh's order."""
    sq, MZ, GZ, sw2, al, lo, hi, a, b, N = p[:10]
    beta = p[10] if len(p) > 10 else 0.0
    Vl, Al, dVl = -0.5 + 2 * sw2, -0.5, 2.0
    A0 = A1 = A2 = B1 = B2 = dA1 = dA2 = dB2 = 0.0
    for n, Q, T in ((2, 2 / 3, 0.5), (3, -1 / 3, -0.5)):
        Vq, Aq, dVq = T - 2 * Q * sw2, T, -2 * Q
        A0 += n * Q * Q
        A1 += n * (-2 * Q * Vl * Vq)
        A2 += n * (Al * Al + Vl * Vl) * (Aq * Aq + Vq * Vq)
        B1 += n * (-4 * Q * Al * Aq)
        B2 += n * 8 * Al * Vl * Aq * Vq
        dA1 += n * (-2 * Q * (dVl * Vq + Vl * dVq))
        dA2 += n * (2 * Vl * dVl * (Aq * Aq + Vq * Vq) + (Al * Al + Vl * Vl) * 2 * Vq * dVq)
        dB2 += n * 8 * Al * Aq * (dVl * Vq + Vl * dVq)
    k = 1 / (4 * sw2 * (1 - sw2))
    l0, L = math.log(lo * lo / sq ** 2), math.log((hi * hi) / (lo * lo))
    pref = al * al / 12 * 0.3893794e9 * 4 * math.pi
    dk = -k * (1 - 2 * sw2) / (sw2 * (1 - sw2))
    inv = 1 / float(mp.besseli(0, beta))
    e2, ln2 = 1 / mp.log(2), mp.log(2)
    B = xc(-mpf(l0) * e2)
    A = X(int(mp.floor(mpf(L) * e2 * mpf(2) ** -B.e)), 0, 0)
    K = [B, A, xc(mpf(L) * ln2 * pref)] + [xc(v) for v in (
        sq, -MZ * MZ, (GZ * MZ) ** 2, k, A0, A1, A2, B1, B2, a, b, 0.2 * N * N, MZ, GZ, dk, dA1,
        dA2, dB2)] + [xc(mpf(beta) * e2), xc(inv)]
    return (l0, L, pref, sq, MZ * MZ, (GZ * MZ) ** 2, k, A0, A1, A2, B1, B2, a, b, 0.2 * N * N, MZ,
            GZ, dk, dA1, dA2, dB2, beta, inv), (X * len(K))(*K)


def dy_exact(u, k):
    (l0, L, pref, sq, M2, G2, kap, A0, A1, A2, B1, B2, a, b, N, MZ, GZ, dk, dA1, dA2, dB2) = [
        mpf(v) for v in k[:21]]
    lt = l0 + u[0] * L
    x1, x2 = mp.exp(lt * (1 - u[1])), mp.exp(lt * u[1])
    o1, o2, sh, c = 1 - x1, 1 - x2, sq ** 2 * mp.exp(lt), 2 * u[2] - 1
    lo = mp.log(o1 * o2)
    cm = N * mp.exp(a * lt + b * lo)
    D = sh - M2
    den = D * D + G2
    r1, r2 = kap * sh * D / den, kap ** 2 * sh * sh / den
    ev, od = cm * (o1 ** 4 + o2 ** 4) * (1 + c * c), cm * (o2 ** 4 - o1 ** 4) * c
    P = mp.exp(lt) * L * -lt * pref / sh
    g = P * (ev * (A0 + A1 * r1 + A2 * r2) + od * (B1 * r1 + B2 * r2))
    s1, s2 = ev * A1 + od * B1, ev * A2 + od * B2
    dden = -(s1 * r1 + s2 * r2) / den
    dD = s1 * kap * sh / den + dden * 2 * D
    return g, [P * (dden * 2 * GZ ** 2 * MZ - dD * 2 * MZ), P * dden * 2 * GZ * MZ ** 2,
               P * ((s1 * sh * D / den + s2 * 2 * kap * sh * sh / den) * dk
                    + ev * (r1 * dA1 + r2 * dA2) + od * r2 * dB2), g * lt, g * lo]


@pytest.mark.parametrize("params", [
    DYNLO_PARAMS, DY_PARAMS[:7] + (0.75, 4.0, 2.0, -1.5),
    (1.0, 0.0912, 0.0025, 0.4, 1.0, 1e-6, 0.9, -1.25, 0.0, 1e-3, 20.0)])
def test_integrands(lib, params):
    """Weights and gradients at random points, against the same formulas in 200
    bits.  The logarithms carry 2^-59 of their size (at most 2^6 here) into the
    exponentials, 1 - x magnifies x's error by at most 2^4 for the points
    drawn, in up to 11 powers, and some forty operations add 2^-60 each: below
    2^-49 with the final rounding; the gradient's differences of terms lose
    up to ten more bits of the largest term."""
    r = random.Random(3)
    k, K = dy_constants(params)
    gr = (C.c_double * 5)()
    for _ in range(300):
        d = r.randint(4, 13)
        x = [r.getrandbits(64) for _ in range(d)]
        x[1] = int((0.05 + 0.9 * r.random()) * 2 ** 64)
        u = [mpf(v) / mpf(2) ** 64 for v in x]
        q = (C.c_uint64 * 16)(*x)
        g, dg = dy_exact(u, k)
        assert abs(lib.dy(q, K, gr) / g - 1) < mpf(2) ** -49
        for p in range(5):
            assert abs(gr[p] - dg[p]) <= mpf(2) ** -39 * max(abs(dg[p]), mpf(2) ** -10 * abs(g))
        for v in u[4:]:
            g *= mp.exp(mpf(k[21]) * mp.cos(2 * mp.pi * v)) * mpf(k[22])
        assert abs(lib.nlo(q, d, K) / g - 1) < mpf(2) ** -48


@pytest.mark.parametrize("sigma,shift", [(0.1, 0.0), (0.3, 0.1), (5.0, 0.0)])
def test_gauss(lib, sigma, shift):
    """The exponent (at most 16/4/(2 sigma^2) log2 e = 290) within 2^-60 of
    itself, and the final rounding."""
    r = random.Random(4)
    inv = 1 / (2 * sigma * sigma)
    K = (X * 2)(xc(mpf(inv) / mp.log(2)), xc(-mpf(shift)))
    for _ in range(300):
        d = r.randint(1, 16)
        x = [r.getrandbits(64) for _ in range(d)]
        q = sum((mpf(v) / mpf(2) ** 64 - mpf(1) / 2) ** 2 for v in x)
        g = mp.exp(-q * mpf(inv))
        got = lib.gauss((C.c_uint64 * 16)(*x), d, K)
        assert abs(got - (g - mpf(shift))) <= mpf(2) ** -51 * max(g, abs(g - mpf(shift)))


@pytest.mark.parametrize("ycut", [0.01, 0.2, 1e-6])
def test_ee3j(lib, ycut):
    """Fixed point to 2^-58 of the total energy squared against y13, y23 >=
    y_cut, and the final rounding; zero exactly outside the cuts."""
    r = random.Random(5)
    K = (X * 1)(X(int(mpf(ycut) * mpf(2) ** 64), 0, 0))
    inside = 0
    for _ in range(600):
        x = [r.getrandbits(64) for _ in range(5)]
        x1, x2 = mpf(x[0]) / mpf(2) ** 64, mpf(x[1]) / mpf(2) ** 64
        got = lib.ee3j((C.c_uint64 * 5)(*x), K)
        y = mpf(ycut)
        if 1 - x1 > y and 1 - x2 > y and x1 + x2 - 1 > y:
            inside += 1
            want = (x1 ** 2 + x2 ** 2) / ((1 - x1) * (1 - x2))
            lost = mpf(2) ** -57 * (1 / (1 - x1) + 1 / (1 - x2))
            assert abs(got / want - 1) <= mpf(2) ** -52 + lost
        else:
            assert got == 0.0
    assert inside > 30
