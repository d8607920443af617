// gv_xint.cuh -- the integrands of gv_integrands.cuh in the 64-bit-significand
// arithmetic of gv_x64.cuh (the FP64 form).  The same formulas, from the same
// derived constants; logarithms and exponentials are taken to base 2, the
// sampled variables come as 64-bit fractions of 1, and the 3-jet kinematics
// run in fixed point in units of the beam energy (the total energy cancels).
#pragma once
#include "gv_x64.cuh"

// Constants (GvX), derived from the double constants by gv_consts_kernel.
#define XK_B2 0       // -log2 tau_lo
#define XK_A2 1       // log2(tau_hi / tau_lo): significand in units of XK_B2's exponent
#define XK_CP 2       // ln(tau_hi / tau_lo) ln 2 times the prefactor
#define XK_SQRTS 3
#define XK_MMZ2 4     // -M_Z^2
#define XK_GM2 5
#define XK_KAPPA 6
#define XK_CA0 7
#define XK_CA1 8
#define XK_CA2 9
#define XK_CB1 10
#define XK_CB2 11
#define XK_A 12
#define XK_B 13
#define XK_NORM 14
#define XK_MZ 15
#define XK_GZ 16
#define XK_DKAPPA 17
#define XK_DCA1 18
#define XK_DCA2 19
#define XK_DCB2 20
#define XK_BETA2 21   // beta log2 e
#define XK_INVI0 22
#define XK_N 23
#define XK_INV2S2 0   // Gaussian: log2 e / (2 sigma^2)
#define XK_MSHIFT 1   //   -shift
#define XK_YCUT 0     // 3-jet: y_cut as a 64-bit fraction (in m)

#define GV_X_LN2 (GvX{0xb17217f7d1cf79abull, -64, 0u})
#define GV_X_LOG2E (GvX{0xb8aa3b295c17f0bbull, -63, 0u})

// ---------------------------------------------------------------------------
// Gaussian product minus a constant.  The squares are summed exactly (128
// bits and a carry word).
// ---------------------------------------------------------------------------
struct GvSumX {
  unsigned long long lo = 0ull, mid = 0ull;
  unsigned top = 0u;
  GV_X_FN void add(unsigned long long x) {
    const unsigned long long h = 1ull << 63, dx = x >= h ? x - h : h - x;
    const unsigned long long pl = dx * dx, ph = xi_mulhi(dx, dx);
    lo += pl;
    const unsigned long long c = ph + (lo < pl ? 1ull : 0ull);  // ph < 2^63: no carry within
    mid += c;
    top += mid < c ? 1u : 0u;
  }
};
GV_X_FN GvX gv_gauss_x(const GvSumX& s, const GvX* K) {
  GvX q;
  if (s.top) {
    const int k = 64 - xi_clz((unsigned long long)s.top);
    q = GvX{((unsigned long long)s.top << (64 - k)) | (s.mid >> k), -64 + k, 0u};
  } else if (s.mid) {
    const int lz = xi_clz(s.mid);
    q = GvX{lz ? (s.mid << lz) | (s.lo >> (64 - lz)) : s.mid, -64 - lz, 0u};
  } else {
    q = x_norm(s.lo, -128);
  }
  const GvX t = x_mul(q, K[XK_INV2S2]);
  const GvX g = x_exp2(t.m, t.e, true);
  return K[XK_MSHIFT].m ? x_add(g, K[XK_MSHIFT]) : g;
}
template <int MAXD>
GV_X_FN GvX gv_gauss_x(const unsigned long long (&x)[MAXD], int d, const GvX* K) {
  GvSumX s;
  for (int a = 0; a < d; ++a) s.add(x[a]);
  return gv_gauss_x(s, K);
}

// 1 - q for a fraction q
GV_X_FN GvX x_one_minus(unsigned long long q) {
  return q ? x_from_q64(0ull - q) : GvX{1ull << 63, -63, 0u};
}

// ---------------------------------------------------------------------------
// LO pp -> gamma*/Z -> mu- mu+ (see gv_drell_yan).
// ---------------------------------------------------------------------------
template <bool GRAD>
GV_X_FN GvX gv_drell_yan_x(const unsigned long long* x, const GvX* K, GvX* grad) {
  // -log2 tau and its split between the partons, all at one exponent:
  // x1 = sqrt(tau) e^y = tau^(1 - x[1]), x2 = tau^x[1]
  const int eB = K[XK_B2].e;
  const unsigned long long lt = K[XK_B2].m - xi_mulhi(K[XK_A2].m, x[0]);
  const unsigned long long l2 = xi_mulhi(lt, x[1]), l1 = lt - l2;
  if (l1 == 0ull || l2 == 0ull) {  // a parton with x = 1: the densities vanish
    if (GRAD)
      for (int p = 0; p < 5; ++p) grad[p] = x_zero();
    return x_zero();
  }
  const GvX X1 = x_exp2(l1, eB, true), X2 = x_exp2(l2, eB, true);
  const GvX o1 = x_one_minus(x_to_q64(X1)), o2 = x_one_minus(x_to_q64(X2));
  // momenta as light-cone components, and the invariants shat, -that, -uhat
  const GvX p1p = x_mul(K[XK_SQRTS], X1), p2m = x_mul(K[XK_SQRTS], X2);
  const GvX p3p = x_mul(p1p, x_from_q64(x[2]));   // (p1p / 2) (1 + cos theta)
  const GvX p3m = x_mul(p2m, x_one_minus(x[2]));  // (p2m / 2) (1 - cos theta)
  const GvX shat = x_mul(p1p, p2m), mt = x_mul(p1p, p3m), mu = x_mul(p2m, p3p);
  const GvX inv_shat = x_rcp(shat);
  const GvX c = x_mul(x_sub(mu, mt), inv_shat);
  const GvX one = GvX{1ull << 63, -63, 0u};
  const GvX opc2 = x_addp(one, x_sqr(c));
  // parton luminosities
  const GvX l12 = x_log2(x_mul(o1, o2));
  const GvX lx = x_norm(lt, eB, 1u);
  const GvX common =
      x_mul(K[XK_NORM], x_exp2(x_add(x_mul(K[XK_A], lx), x_mul(K[XK_B], l12))));
  const GvX q1 = x_sqr(x_sqr(o1)), q2 = x_sqr(x_sqr(o2));
  const GvX lf = x_mul(common, q2), lb = x_mul(common, q1);
  // gamma/Z propagator factors
  const GvX D = x_add(shat, K[XK_MMZ2]);
  GvX D2 = x_sqr(D);
  const GvX inv_den = x_rcp(x_addp(D2, K[XK_GM2]));
  const GvX ks = x_mul(K[XK_KAPPA], shat), ki = x_mul(ks, inv_den);
  const GvX chi1 = x_mul(ki, D), chi2 = x_mul(ki, ks);
  const GvX A = x_add(x_addp(x_mul(K[XK_CA2], chi2), K[XK_CA0]), x_mul(K[XK_CA1], chi1));
  const GvX B = x_add(x_mul(K[XK_CB2], chi2), x_mul(K[XK_CB1], chi1));
  const GvX even = x_mul(x_addp(lf, lb), opc2), odd = x_mul(x_sub(lf, lb), c);
  const GvX S = x_add(x_mul(even, A), x_mul(odd, B));
  GvX ly = x_neg(lx);
  const GvX P = x_mul(x_mul(x_mul(X1, X2), x_mul(ly, K[XK_CP])), inv_shat);
  const GvX g = x_mul(P, S);
  if (GRAD) {
    // reverse sweep from g = P S (as gv_drell_yan's)
    const GvX Ab = x_mul(P, even), Bb = x_mul(P, odd);
    const GvX gl = x_mul(g, GV_X_LN2);
    grad[3] = x_mul(gl, lx);   // g ln(x1 x2): g is proportional to (x1 x2)^a ..
    grad[4] = x_mul(gl, l12);  // .. and to ((1 - x1)(1 - x2))^b
    const GvX chi1b = x_add(x_mul(Ab, K[XK_CA1]), x_mul(Bb, K[XK_CB1]));
    const GvX chi2b = x_add(x_mul(Ab, K[XK_CA2]), x_mul(Bb, K[XK_CB2]));
    const GvX si = x_mul(shat, inv_den);
    // d chi1/d kappa = shat D / den, d chi2/d kappa = 2 kappa shat^2 / den
    const GvX kb = x_add(x_mul(chi1b, x_mul(si, D)), x_scale(x_mul(chi2b, x_mul(ks, si)), 1));
    // chi1 = (kappa shat) D / den, chi2 = (kappa shat)^2 / den
    const GvX invb = x_mul(ks, x_add(x_mul(chi1b, D), x_mul(chi2b, ks)));
    const GvX denb = x_neg(x_mul(invb, x_sqr(inv_den)));
    const GvX Db = x_add(x_mul(chi1b, ki), x_scale(x_mul(denb, D), 1));
    const GvX dg = x_scale(x_mul(denb, x_mul(K[XK_GZ], K[XK_MZ])), 1);
    // den = D^2 + GZ^2 MZ^2, D = shat - MZ^2
    grad[0] = x_sub(x_mul(dg, K[XK_GZ]), x_scale(x_mul(Db, K[XK_MZ]), 1));
    grad[1] = x_mul(dg, K[XK_MZ]);
    const GvX r = x_add(x_mul(x_mul(Ab, chi1), K[XK_DCA1]), x_mul(x_mul(Ab, chi2), K[XK_DCA2]));
    grad[2] = x_add(x_add(x_mul(kb, K[XK_DKAPPA]), r), x_mul(x_mul(Bb, chi2), K[XK_DCB2]));
  }
  return g;
}

// ---------------------------------------------------------------------------
// NLO-shaped stand-in: Drell-Yan times exp(beta cos 2 pi x_k) / I0(beta) for
// each further axis.  The cosines are summed exactly (Q62, as 16 hi + lo), so
// that an event takes one exponential instead of one per axis.
// ---------------------------------------------------------------------------
struct GvSumCos {
  long long hi = 0;
  unsigned lo = 0u;
  GV_X_FN void add(unsigned long long x) {
    const long long v = x_cos_turn(x);
    hi += v >> 4;
    lo += (unsigned)v & 15u;
  }
  GV_X_FN GvX value() const {  // |sum| <= 12: below 2^62 in hi
    long long h = hi + (long long)(lo >> 4);
    unsigned l = lo & 15u;
    const unsigned s = h < 0 ? 1u : 0u;
    if (s) {
      h = -h - (l ? 1 : 0);
      l = (16u - l) & 15u;
    }
    const unsigned long long m = (unsigned long long)h;
    return m >> 60 ? x_norm((m << 2) | (l >> 2), -60, s) : x_norm((m << 4) | l, -62, s);
  }
};
// 1 / I0(beta)^n
GV_X_FN GvX gv_nlo_norm_x(const GvX& inv, int n) {
  GvX r = {1ull << 63, -63, 0u};
  for (int k = 0; k < n; ++k) r = x_mul(r, inv);
  return r;
}
GV_X_FN GvX gv_nlo_x(const GvX& dy, const GvSumCos& c, const GvX& norm, const GvX* K) {
  return x_mul(x_mul(dy, norm), x_exp2(x_mul(K[XK_BETA2], c.value())));
}
template <int MAXD>
GV_X_FN GvX gv_dy_nlo_x(const unsigned long long (&x)[MAXD], int d, const GvX* K) {
  const GvX g = gv_drell_yan_x<false>(x, K, nullptr);
  GvSumCos c;
  for (int a = 4; a < d; ++a) c.add(x[a]);
  return gv_nlo_x(g, c, gv_nlo_norm_x(K[XK_INVI0], d - 4), K);
}

// ---------------------------------------------------------------------------
// e+e- -> q qbar g (see gv_ee3j), energies and momenta in units of the total
// energy, signed Q62.
// ---------------------------------------------------------------------------
GV_X_FN GvX gv_ee3j_x(const unsigned long long* x, const GvX* K) {
  const unsigned long long yc = K[XK_YCUT].m;
  const unsigned long long x1 = x[0], x2 = x[1], s = x1 + x2;  // s: x1 + x2 - 1 after the carry
  if (!(s < x1 && s > yc && x1 != 0ull && 0ull - x1 > yc && 0ull - x2 > yc)) return x_zero();
  const long long one = 1ll << 62;
  const long long e1 = (long long)(x1 >> 3), e2 = (long long)(x2 >> 3);  // x_i / 2
  const long long e3 = (long long)((0ull - s) >> 3);                    // x3 = 1 - s
  // cos of the angle between 1 and 2: 1 - 2 (1 - x3) / (x1 x2)
  const GvX q = x_mul(x_from_q64(s), x_rcp(x_norm(xi_mulhi(x1, x2), -64)));
  const int sh = -63 - q.e;  // 2 q in Q62
  const unsigned long long q2 = sh <= 0 ? ~0ull : (sh < 64 ? q.m >> sh : 0ull);
  const unsigned long long two = ~0ull >> 1;  // 2 less a unit
  const long long c12 = one - (long long)(q2 > two ? two : q2);
  const long long v12 = one - xi_mulq62(c12, c12);
  const long long s12 = xi_sqrt_q62(v12 > 0 ? (unsigned long long)v12 : 0ull);
  // event plane: p1 along z, p2 in the x-z plane, p3 balances
  const long long p1z = e1, p2x = xi_mulq62(e2, s12), p2z = xi_mulq62(e2, c12);
  const long long p3x = -p2x, p3z = -p1z - p2z;
  // R = Rz(phi) Ry(theta) Rz(psi), the columns that multiply x and z
  const long long ct = (long long)(x[2] >> 1) - one;
  const long long st = xi_sqrt_q62(xi_mulhi(x[2], 0ull - x[2]));  // 1 - ct^2 = 4 x (1 - x)
  long long sf, cf, sp, cp;
  x_sincos_turn(x[3], &sf, &cf);
  x_sincos_turn(x[4], &sp, &cp);
  const long long r00 = xi_mulq62(xi_mulq62(cf, ct), cp) - xi_mulq62(sf, sp), r02 = xi_mulq62(cf, st);
  const long long r10 = xi_mulq62(xi_mulq62(sf, ct), cp) + xi_mulq62(cf, sp), r12 = xi_mulq62(sf, st);
  const long long r20 = -xi_mulq62(st, cp), r22 = ct;
  const long long a[3] = {xi_mulq62(r02, p1z), xi_mulq62(r12, p1z), xi_mulq62(r22, p1z)};
  const long long b[3] = {xi_mulq62(r00, p2x) + xi_mulq62(r02, p2z),
                          xi_mulq62(r10, p2x) + xi_mulq62(r12, p2z),
                          xi_mulq62(r20, p2x) + xi_mulq62(r22, p2z)};
  const long long c[3] = {xi_mulq62(r00, p3x) + xi_mulq62(r02, p3z),
                          xi_mulq62(r10, p3x) + xi_mulq62(r12, p3z),
                          xi_mulq62(r20, p3x) + xi_mulq62(r22, p3z)};
  const long long d13 = xi_mulq62(a[0], c[0]) + xi_mulq62(a[1], c[1]) + xi_mulq62(a[2], c[2]);
  const long long d23 = xi_mulq62(b[0], c[0]) + xi_mulq62(b[1], c[1]) + xi_mulq62(b[2], c[2]);
  const GvX y13 = x_scale(x_from_q62(xi_mulq62(e1, e3) - d13), 1);
  const GvX y23 = x_scale(x_from_q62(xi_mulq62(e2, e3) - d23), 1);
  const unsigned long long sq = xi_mulhi(x1, x1), sr = xi_mulhi(x2, x2);
  const GvX num = x_addp(x_from_q64(sq), x_from_q64(sr));
  return x_mul(num, x_rcp(x_mul(y23, y13)));
}
