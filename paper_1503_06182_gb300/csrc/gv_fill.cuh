// gv_fill.cuh -- the fused per-event kernel of one VEGAS iteration.
//
// One CTA evaluates one tile of up to GV_TILE consecutive events (Section 2.1: each
// event generated and evaluated independently), with EPT events per thread:
//   pass 1: Philox words -> bins and in-bin positions -> x on the adaptive grid
//           ((edge, width) pairs and Jacobian factors staged in shared memory)
//           -> g(x) -> w = J g (J in FP64 in the FP64 form; FP32 mantissas
//           with an integer exponent in the FP32 form); the bins stay in registers
//           (d <= 4) or go to shared memory;
//   tile scale: block max of the weights' exponents (order-free): it places
//           the window of limbs of gv_limbs.cuh;
//   pass 2: w^2 cut once per event into 22-bit digits at absolute positions;
//           per axis three (FP32) or four 32-bit shared atomics add them to
//           the event's bin, and the same digits with those of w go to
//           per-lane columns for the tile's sums of w and w^2 (32-bit shared
//           atomics run several times faster than 64-bit ones here).  Weights
//           below the window take a further pass.
// With VEGAS+ (PLUS), each thread takes GV_PLUS_SEG consecutive events (one
// range): a binary search finds its first event's hypercube, the next events
// step across hypercube boundaries (every hypercube holds at least 2 events),
// and each event takes stratified words from its hypercube's digits.  The
// estimate's weight is F C/(nh n_h) and the bins' quantity F sqrt(1/(nh n_h)),
// F = J g.  The thread also sums F and F^2 over the run of each hypercube in
// its range, in event order (the range's segments), which the hypercube
// statistics add up after the iteration.
// With a histogram of the observable (HIST), every event with w != 0 also
// adds w^2 (the same digits) and w (21-bit signed digits, so negative weights
// add like positive ones) to its observable's bin.
// Integer sums are order-free, so the tile's result is the same for every
// block size / events-per-thread choice.  Apart from the Jacobian product and
// w = J g, the bookkeeping runs on the integer pipes: the FP64 pipe of this
// chip is a small fraction of its FP32 throughput.
#pragma once
#include "gv_integrands.cuh"
#include "gv_limbs.cuh"
#include "gv_plus_stat.cuh"
#include "gv_xint.cuh"

// The arithmetic of an event: Real = float, double or GvX (FP64 results on the
// integer pipes).  W: the weight's type; Coord: a sampled variable's.
template <typename Real>
struct GvForm {
  using W = Real;
  using Coord = Real;
  static constexpr int ID = sizeof(Real) == 4 ? GV_FORM_F32 : GV_FORM_F64;
};
template <>
struct GvForm<GvX> {
  using W = double;
  using Coord = unsigned long long;
  static constexpr int ID = GV_FORM_X64;
};

template <int IG>
struct GvTraits;
template <>
struct GvTraits<GV_GAUSS> {
  static constexpr int NK = 2, NX = 2;  // constants; as GvX
};
template <>
struct GvTraits<GV_DY> {
  static constexpr int NK = DK_NK, NX = XK_N;
};
template <>
struct GvTraits<GV_EE3J> {
  static constexpr int NK = 3, NX = 1;
};
template <>
struct GvTraits<GV_DYNLO> {
  static constexpr int NK = NK_NK, NX = XK_N;
};
static_assert(XK_N <= GV_NCONST_X, "room for the GvX constants");

// The GvX constants stay in (shared) memory: too many for registers.  1 / I0
// of the NLO-shaped integrand is there to the power of its further axes.
template <int NC>
struct GvConst<GvX, NC> {
  const GvX* k;
  __device__ __forceinline__ const GvX& operator[](int i) const { return k[i]; }
};
__device__ __forceinline__ const GvX* gv_x_consts(const double* kconst) {
  return reinterpret_cast<const GvX*>(kconst + GV_NCONST);
}
template <int IG>
__device__ __forceinline__ GvX gv_x_const(const double* kconst, int i, int d) {
  const GvX c = gv_x_consts(kconst)[i];
  return IG == GV_DYNLO && i == XK_INVI0 ? gv_nlo_norm_x(c, d - 4) : c;
}

// An integrand taken axis by axis: the variables that its formula needs at the
// end stay (x), the others are consumed as they come, so that an event of many
// axes holds few registers.  first(k, ..): axis k < 4, more(a, ..): axis
// a >= 4, in order; then value and observable.  The observable (the
// differential distributions of Section 3.2): Gauss x_0; Drell-Yan (both
// forms) the dilepton mass m_ll = sqrt(tau s) in GeV, with tau as the
// integrand forms it; 3-jet the thrust max(x1, x2, x3), x3 = 2 - x1 - x2.
template <int IG, typename Real>
struct GvStream {
  using Coord = typename GvForm<Real>::Coord;
  using W = typename GvForm<Real>::W;
  using Const = GvConst<Real, GvTraits<IG>::NK>;
  static constexpr bool X64 = GvForm<Real>::ID == GV_FORM_X64;
  Coord x[IG == GV_EE3J ? 5 : 4];
  Real f = Real();        // Gauss: the sum of squares; NLO-shaped: the factors' product
  // 64-bit significands: Gauss: the sum of squares; NLO-shaped: of the cosines
  [[maybe_unused]] std::conditional_t<IG == GV_DYNLO, GvSumCos, GvSumX> q;

  __device__ __forceinline__ void first(int k, const Coord& v, const Const& K) {
    x[k] = v;
    if constexpr (IG == GV_GAUSS) square(v);
  }
  __device__ __forceinline__ void more(int a, const Coord& v, const Const& K) {
    if constexpr (IG == GV_GAUSS) {
      square(v);
    } else if constexpr (IG == GV_EE3J) {
      if (a == 4) x[4] = v;
    } else if constexpr (IG == GV_DYNLO) {
      if constexpr (X64) {
        q.add(v);
      } else {
        const Real t = gv_nlo_factor<Real>(v, K);
        f = a == 4 ? t : f * t;
      }
    }
  }
  __device__ __forceinline__ void square(const Coord& v) {
    if constexpr (X64) {
      q.add(v);
    } else {
      const Real dx = v - (Real)0.5;
      f = GvMath<Real>::fma(dx, dx, f);
    }
  }
  __device__ __forceinline__ Real value(int d, const Const& K) const {
    if constexpr (X64) {
      if constexpr (IG == GV_GAUSS) return gv_gauss_x(q, K.k);
      if constexpr (IG == GV_DY) return gv_drell_yan_x<false>(x, K.k, nullptr);
      if constexpr (IG == GV_EE3J) return gv_ee3j_x(x, K.k);
      if constexpr (IG == GV_DYNLO) {
        const GvX g = gv_drell_yan_x<false>(x, K.k, nullptr);
        return d > 4 ? gv_nlo_x(g, q, K[XK_INVI0], K.k) : g;
      }
    } else {
      if constexpr (IG == GV_GAUSS)
        return GvMath<Real>::exp(-f * K[GK_INV2S2]) - K[GK_SHIFT];
      if constexpr (IG == GV_DY) return gv_drell_yan<Real, false>(x, K, nullptr);
      if constexpr (IG == GV_EE3J) return gv_ee3j<Real>(x, K);
      if constexpr (IG == GV_DYNLO) {
        const Real g = gv_drell_yan<Real, false>(x, K, nullptr);
        return d > 4 ? g * f : g;
      }
    }
  }
  __device__ __forceinline__ W observable(const Const& K) const {
    if constexpr (X64) {
      if constexpr (IG == GV_GAUSS) {
        return x_to_double(x_from_q64(x[0]));
      } else if constexpr (IG == GV_DY || IG == GV_DYNLO) {  // sqrt(s) 2^(log2(tau) / 2)
        const unsigned long long lt = K[XK_B2].m - xi_mulhi(K[XK_A2].m, x[0]);
        return x_to_double(x_mul(K[XK_SQRTS], x_exp2(lt, K[XK_B2].e - 1, true)));
      } else {  // (x3 = 2 - x1 - x2 where it is below 1; elsewhere the weight is 0)
        const unsigned long long x3 = 0ull - (x[0] + x[1]);
        const unsigned long long t = x[0] > x[1] ? x[0] : x[1];
        return x_to_double(x_from_q64(t > x3 ? t : x3));
      }
    } else {
      using Mt = GvMath<Real>;
      if constexpr (IG == GV_GAUSS) {
        return x[0];
      } else if constexpr (IG == GV_DY || IG == GV_DYNLO) {
        const Real tau = Mt::exp(Mt::fma(x[0], K[DK_L], K[DK_LOGTAULO]));
        return Mt::sqrt(tau * K[DK_S]);
      } else {
        const Real x1 = x[0], x2 = x[1], x3 = (Real)2 - x1 - x2;
        const Real t = x1 > x2 ? x1 : x2;
        return t > x3 ? t : x3;
      }
    }
  }
};

// Histogram bin of v among nh bins over [lo, lo + nh / invw): 0 below (and
// for a value that is not a number), nh + 1 above.
template <typename Real>
__device__ __forceinline__ int gv_hist_bin(Real v, Real lo, Real invw, int nh) {
  if (!(v >= lo)) return 0;
  const Real t = (v - lo) * invw;
  if (!(t < (Real)nh)) return nh + 1;
  return 1 + (int)t;
}

// One bin of one axis as staged in shared memory (FP32 form: GvBin32 of the
// grid pack).
struct __align__(16) GvBin64 {
  double e, w;
};
// A float widened to double by integer operations (exact; the FP64 pipe of
// this chip is scarce).  Zero, subnormal and non-finite inputs are handled.
__device__ __forceinline__ double gv_widen(float g) {
  const unsigned u = __float_as_uint(g);
  const unsigned long long sign = (unsigned long long)(u >> 31) << 63;
  const unsigned ef = (u >> 23) & 0xFFu;
  unsigned long long m = u & 0x7FFFFFu;
  unsigned long long bits;
  if (ef == 0xFFu) {
    bits = sign | 0x7FF0000000000000ull | (m << 29);
  } else if (ef != 0u) {
    bits = sign | ((unsigned long long)(ef + 896u) << 52) | (m << 29);
  } else if (m == 0ull) {
    bits = sign;
  } else {  // subnormal float m 2^-149, leading one at bit p = 23 - lz
    const int lz = __clzll((long long)m) - 40;
    m = (m << lz) & 0x7FFFFFull;
    bits = sign | ((unsigned long long)(897 - lz) << 52) | (m << 29);
  }
  return __longlong_as_double((long long)bits);
}
__device__ __forceinline__ double gv_widen(double g) { return g; }

// The Jacobian of one event: FP64 in the FP64 form; in the FP32 form the
// product of the FP32 mantissas and the sum of the exponents (no range limit,
// and nothing on the FP64 pipe, of which this chip has little).
template <typename Real>
struct GvJac;
template <>
struct GvJac<double> {
  double v;
};
template <>
struct GvJac<float> {
  float m;
  int e;
};
template <>
struct GvJac<GvX> {
  GvX v;
};

// x 2^E for a double x, on the integer pipes: zero, infinity and NaN pass
// through, a result beyond FP64 becomes infinity (counted as non-finite by
// the caller), one below the normal range becomes zero.
__device__ __forceinline__ double gv_ldexp_bits(double x, int E) {
  const long long b = __double_as_longlong(x);
  const int ef = (int)((b >> 52) & 0x7FF);
  if (ef == 0 || ef == 0x7FF || E == 0) return x;
  const int nf = ef + E;
  const long long sign = b & (long long)0x8000000000000000ull;
  if (nf >= 0x7FF) return __longlong_as_double(sign | 0x7FF0000000000000ll);
  if (nf <= 0) return __longlong_as_double(sign);
  return __longlong_as_double((b & ~0x7FF0000000000000ll) | ((long long)nf << 52));
}

// w = J g as a double.
__device__ __forceinline__ double gv_weight(const GvJac<double>& J, double g) {
  return __dmul_rn(J.v, g);
}
__device__ __forceinline__ double gv_weight(const GvJac<GvX>& J, const GvX& g) {
  return x_to_double(x_mul(J.v, g));
}
__device__ __forceinline__ double gv_weight(const GvJac<float>& J, float g) {
  const float p = __fmul_rn(J.m, g);
  const unsigned u = __float_as_uint(p);
  const int ef = (int)((u >> 23) & 0xFFu);
  const int nf = ef + 896 + J.e;  // the double's exponent field
  if (ef != 0 && ef != 0xFF && nf > 0 && nf < 0x7FF)  // normal in and out: one assembly
    return __longlong_as_double((long long)(((unsigned long long)(u >> 31) << 63) |
                                            ((unsigned long long)nf << 52) |
                                            ((unsigned long long)(u & 0x7FFFFFu) << 29)));
  return gv_ldexp_bits(gv_widen(p), J.e);
}

// The double gv_weight assembles, from the product's bits.
__device__ __forceinline__ double gv_weight_bits(unsigned u, int e) {
  return gv_ldexp_bits(gv_widen(__uint_as_float(u)), e);
}

template <typename Real>
struct GvPair;
template <>
struct GvPair<float> {
  using T = GvBin32;
};
template <>
struct GvPair<double> {
  using T = GvBin64;
};
// One bin as the 64-bit-significand form reads it: edge and width as
// fractions, and the Jacobian factor N w = jm 2^je, jm in [2^63, 2^64).
struct __align__(16) GvBinX {
  unsigned long long e, w, jm;
  long long je;
};
template <>
struct GvPair<GvX> {
  using T = GvBinX;
};

// Shared-memory layout of the fill kernel (bytes), 16-byte aligned pieces:
//   evs  [R][T]   u32     the events between the two passes (GvEvent), slot
//                         k B + tid the thread's k-th event
//   wd   [W][T]   u32     the tile's Philox words, generated before the kernel
//                         waits for its predecessor (see below), W = 4
//                         ceil(d/4); over evs: a thread replaces its event's
//                         words by the event
//   ew   [d*N]    GvBin32 (e, w, jm, je) in FP32, GvBin64 (e, w) on the FP64
//                         pipe, GvBinX with 64-bit significands
//   jac  [d*N]    f64     Jacobian factor N*(e_{i+1}-e_i) (FP64 pipe only)
// After the first pass the forward fill's limbs lie over what follows evs:
//   hist [d*N][L] u32     the bins' limbs
//   hh   [nhist][L] u32, hw [nhist][LW] i32  the histogram's limbs of w^2 and w,
//        hc copies (events of a warp share few bins of an observable with a
//        peak: 8 passes per atomic for Drell-Yan masses, 4 with lane l adding
//        to copy l % 4; ten iterations of 1e6 events with 60 bins 553 -> 537 us)
//   lq   [L (FP64: + 2)][32] u32, lw [rows][32] i32   the lanes' columns of w^2 and w
// and beside both:
//   bins [d][T]   u8      the events' bins (more than 4 axes), their high bytes
//                         in as many again where N > 256
//   po   [GV_PLUS_WIN] i32 hypercube offsets relative to the tile (VEGAS+)
//   ps   [GV_PLUS_WIN + GV_TILE/GV_PLUS_SEG] double2  the tile's segments
//                         (VEGAS+): each window hypercube's first, then each
//                         range's continuation of an earlier hypercube
__host__ __device__ inline unsigned gv_align16(unsigned b) { return (b + 15u) & ~15u; }

// The forward fill generates its tile's Philox words before it waits for the
// previous kernel (the words depend only on the seed, the counter and the
// event), where the launch overlaps the previous iteration's reduce and
// refinement (VEGAS+: its layout; the stratified fill stratifies the words
// after the wait); not beyond 8 axes, nor where the words' shared memory
// would take the layout past GV_WORDS_SMEM_MAX (the host sets
// GvFillArgs::hoist accordingly).
#define GV_WORDS_SMEM_MAX (200 * 1024)
__host__ __device__ inline bool gv_fill_hoistable(bool forward, int d) {
  return forward && d <= 8;
}

// A tile of GV_TILE events meets at most GV_TILE/2 + 1 hypercubes (each has
// at least 2 events): the window holds their offsets and the next one.
#define GV_PLUS_WIN (GV_TILE / 2 + 4)

#define GV_PLUS_SEGS (GV_PLUS_WIN + GV_TILE / GV_PLUS_SEG)

// Words of one event between the passes (GvEvent's layout).
__host__ __device__ constexpr int gv_event_words32(bool f64, bool reg_bins, bool plus) {
  return f64 ? (plus ? 4 : 2) + (reg_bins ? 2 : 1) : (plus ? 4 : (reg_bins ? 3 : 2));
}

struct GvFillSmem {
  unsigned wd, ew, jac, limbs, hist, hh, hw, lq, lw, bins, po, ps, total;
  unsigned hs;  // bytes from one copy of the histogram's limbs to the next
  int L, hc;    // limbs of a bin's row, copies of the histogram
  __host__ __device__ GvFillSmem(int d, int N, int form, bool forward, bool bins_smem,
                                 int nhist = 0, bool plus = false, bool words = false,
                                 int T = GV_TILE) {
    hc = 1;
    place(d, N, form, forward, bins_smem, nhist, plus, words, T);
    if (forward && nhist > 0) {  // copies where four CTAs still fit an SM
      const unsigned more = 3u * copy_bytes(nhist, form != GV_FORM_F32);
      if (total + more <= 56u * 1024u) {
        hc = 4;
        place(d, N, form, forward, bins_smem, nhist, plus, words, T);
      }
    }
  }
  // a copy's rows, and words to 8 past a multiple of 32: the same row stands in
  // other banks in each copy
  __host__ __device__ unsigned copy_bytes(int nhist, bool f64) const {
    const unsigned w = (unsigned)(nhist * (L + gv_hist_w_limbs(f64, L)));
    return 4u * (w + (40u - w % 32u) % 32u);
  }
  __host__ __device__ void place(int d, int N, int form, bool forward, bool bins_smem, int nhist,
                                 bool plus, bool words, int T) {
    const unsigned dN = (unsigned)(d * N);
    const bool f64 = form != GV_FORM_F32;
    L = gv_limbs(d * N, nhist == 0 && !plus);
    const unsigned evs = forward ? gv_event_words32(f64, !bins_smem, plus) * T * 4 : 0;
    const unsigned wds = words ? (d + 3) / 4 * 4 * T * 4 : 0;
    wd = 0;
    ew = wds > evs ? wds : evs;
    jac = ew + dN * (form == GV_FORM_X64 ? 32 : 16);
    const unsigned first = gv_align16(jac + (form == GV_FORM_F64 ? dN * 8 : 0));
    limbs = evs;
    hist = limbs;
    hh = hist + (forward ? dN * L * 4 : 0);
    hw = hh + (forward ? nhist * L * 4 : 0);
    hs = forward && nhist > 0 ? copy_bytes(nhist, f64) : 0;
    lq = hh + hc * hs;
    lw = lq + (forward ? (L + (f64 ? GvSig<double>::LOW : 0)) * 32 * 4 : 0);
    const unsigned second = gv_align16(lw + (forward ? gv_lane_rows(f64, L) * 32 * 4 : 0));
    bins = first > second ? first : second;
    po = gv_align16(bins + ((forward && bins_smem) ? d * T * (N > 256 ? 2 : 1) : 0));
    ps = gv_align16(po + (plus ? GV_PLUS_WIN * 4 : 0));
    total = gv_align16(ps + (plus ? GV_PLUS_SEGS * 16 : 0));
  }
  // bytes of the limbs, from `limbs`
  __host__ __device__ unsigned limb_bytes(bool f64) const {
    return lw + gv_lane_rows(f64, L) * 32 * 4 - limbs;
  }
};

// VEGAS+: the hypercube of the tile's local event `local` (the last window
// entry at or below it), and the stratified words of hypercube h:
// r' = floor((c_a 2^32 + r_a) / s) with c_a the base-s digits of h (the
// next two functions).
__device__ __forceinline__ int gv_plus_cube(const int* s_off, int local) {
  int lo = 0, hi = GV_PLUS_WIN;
  while (hi - lo > 1) {
    const int mid = (lo + hi) >> 1;
    if (s_off[mid] <= local)
      lo = mid;
    else
      hi = mid;
  }
  return lo;
}

// A range's segment of window hypercube j (sums s1, s2): the hypercube's
// first segment if it begins in the range (at or after local event r0),
// else the range's continuation of it.  Staged in shared memory (s_seg:
// first segments by window index, then continuations by the tile's range);
// the segments of a hypercube that crosses a tile boundary (offsets outside
// [0, GV_TILE]: the finishing kernel forms its statistics) go to memory too.
__device__ __forceinline__ void gv_plus_put_segment(const GvPlusFill* pf, const int* s_off,
                                                    double2* s_seg, long long h0, int j,
                                                    long long tile0, int r0, double s1,
                                                    double s2) {
  const double2 v = make_double2(s1, s2);
  const bool crossing = s_off[j] < 0 || s_off[j + 1] > GV_TILE;
  if (s_off[j] >= r0) {
    s_seg[j] = v;
    if (crossing) pf->seg_h[h0 + j] = v;
  } else {
    s_seg[GV_PLUS_WIN + r0 / GV_PLUS_SEG] = v;
    if (crossing) pf->seg_r[(tile0 + r0) / GV_PLUS_SEG] = v;
  }
}

// The statistics of every hypercube whose events all lie in the tile, from
// its staged segments in range order (as the finishing kernel adds a crossing
// hypercube's), and the tile's sums of their v/n and weights: thread t takes
// window hypercubes t, t + B, .. in order; then warp 0's lane l adds threads
// (B/32) l .. (B/32)(l + 1) - 1 in order, and a butterfly adds the lanes.
// Few FP64 instructions, one chain.  Written by thread 0 to tpart[tile].
template <int B>
__device__ __forceinline__ void gv_plus_tile_stats(const GvPlusFill* pf, const int* s_off,
                                                   const double2* s_seg, long long h0,
                                                   long long tile, double2* s_red) {
  const int tid = threadIdx.x;
  double vn = 0.0, dd = 0.0;
  for (int j = tid; j < GV_PLUS_WIN - 1; j += B) {
    const int o = s_off[j], e = s_off[j + 1];
    if (o < 0 || e > GV_TILE || h0 + j >= pf->nh) continue;  // crossing, or past the last
    double s1 = s_seg[j].x, s2 = s_seg[j].y;
    for (int r = o / GV_PLUS_SEG + 1; r <= (e - 1) / GV_PLUS_SEG; ++r) {
      s1 += s_seg[GV_PLUS_WIN + r].x;
      s2 += s_seg[GV_PLUS_WIN + r].y;
    }
    const GvPlusStat st = gv_plus_stat(s1, s2, e - o, pf->inv, pf->beta_j);
    pf->var[h0 + j] = st.v;
    pf->dw[h0 + j] = st.w;
    vn += st.vn;
    dd += st.w;
  }
  constexpr int L = B / 32;
  s_red[tid] = make_double2(vn, dd);
  __syncthreads();
  if (tid < 32) {
    double2 r = s_red[L * tid];
#pragma unroll
    for (int i = 1; i < L; ++i) {
      r.x += s_red[L * tid + i].x;
      r.y += s_red[L * tid + i].y;
    }
#pragma unroll
    for (int m = 16; m > 0; m >>= 1) {
      r.x += __shfl_xor_sync(0xffffffffu, r.x, m);
      r.y += __shfl_xor_sync(0xffffffffu, r.y, m);
    }
    if (tid == 0) pf->tpart[tile] = r;
  }
}

// The base-s digits c_a of hypercube h (h < 2^22 is exact in FP32: h / s
// from a float estimate, corrected to the floor).
template <int MAXD>
__device__ __forceinline__ void gv_plus_digits(unsigned h, int d, unsigned s, float inv_s,
                                               unsigned (&c)[MAXD]) {
#pragma unroll
  for (int ax = 0; ax < MAXD; ++ax) {
    if (ax < d) {
      unsigned q = (unsigned)((float)h * inv_s);
      if (q * s > h)
        --q;
      else if ((q + 1u) * s <= h)
        ++q;
      c[ax] = h - q * s;
      h = q;
    }
  }
}

// The stratified words floor(X / s), X = c_a 2^32 + r_a < 2^54: the product
// with floor((2^64-1)/s) is the quotient or one less.
template <int MAXD>
__device__ __forceinline__ void gv_plus_strat(const unsigned (&c)[MAXD], int d, unsigned s,
                                              unsigned long long magic, uint32_t (&r)[MAXD]) {
#pragma unroll
  for (int ax = 0; ax < MAXD; ++ax) {
    if (ax < d) {
      const unsigned long long X = ((unsigned long long)c[ax] << 32) | r[ax];
      unsigned long long t = __umul64hi(X, magic);
      if ((t + 1ull) * s <= X) ++t;
      r[ax] = (uint32_t)t;
    }
  }
}

// A bin's record from its edge and width (e in [0, 1), 0 < w <= 1, exact to
// 2^-64; a width is 1 where the other bins of the axis are below 2^-53); N w is
// exact: 53 + 10 bits.
__device__ __forceinline__ GvBinX gv_bin_x(double e, double w, int N) {
  const GvX E = x_from(e), W = x_from(w);
  const GvX j = x_norm((W.m >> 11) * (unsigned long long)N, W.e + 11);
  return GvBinX{E.m ? x_to_q64(E) : 0ull, x_to_q64(W), j.m, (long long)j.e};
}

// Stage the grid of one integration into shared memory.
template <typename Real>
__device__ __forceinline__ void gv_stage_grid(const double* grid, int d, int N, double* s_jac,
                                              typename GvPair<Real>::T* s_ew, int tid,
                                              int nthr) {
  const GvGridLayout L{d, N};
  const int dN = d * N;
  if constexpr (sizeof(Real) == 4) {
    const uint4* g = reinterpret_cast<const uint4*>(grid + L.off_bin32());
    for (int k = tid; k < dN; k += nthr) reinterpret_cast<uint4*>(s_ew)[k] = __ldcg(g + k);
  } else if constexpr (GvForm<Real>::ID == GV_FORM_X64) {
    for (int k = tid; k < dN; k += nthr) {
      const int a = k / N, i = k - a * N;
      s_ew[k] = gv_bin_x(grid[L.off_e64() + a * (N + 1) + i], grid[L.off_wd64() + k], N);
    }
  } else {
    for (int k = tid; k < dN; k += nthr) {
      const int a = k / N, i = k - a * N;
      s_jac[k] = grid[L.off_jac() + k];
      GvBin64 b;
      b.e = grid[L.off_e64() + a * (N + 1) + i];
      b.w = grid[L.off_wd64() + k];
      s_ew[k] = b;
    }
  }
}

// One axis of an event: its word through the axis' row of the grid (s_ew, and
// s_jac on the FP64 pipe): the variable, its bin, and the axis' factor into
// the Jacobian J (which starts from the first factor).
// FP64 pipe: x = e_i + f*(e_{i+1}-e_i) with f = (lo + 1/2) 2^-32, rounded as
// written, J the FP64 product of the factors N (e_{i+1}-e_i); FP32: x with
// FP32 edges and one fma, J as FP32 mantissa product and exponent sum; 64-bit
// significands: x = e + w (2 lo + 1) 2^-33 in fractions, J the product of the
// normalised factors.
template <typename Real>
__device__ __forceinline__ typename GvForm<Real>::Coord gv_map_axis(
    uint32_t r, int N, const double* s_jac, const typename GvPair<Real>::T* s_ew, bool first,
    GvJac<Real>& J, int& bin) {
  const unsigned long long v = (unsigned long long)r * (unsigned)N;
  const int i = (int)(v >> 32);
  const uint32_t lo = (uint32_t)v;
  const auto ew = s_ew[i];
  bin = i;
  if constexpr (GvForm<Real>::ID == GV_FORM_X64) {
    const GvX j = {ew.jm, (int)ew.je, 0u};
    J.v = first ? j : x_mul(J.v, j);
    return ew.e + xi_mul64x32(ew.w, lo) + (ew.w >> 33);
  } else if constexpr (sizeof(Real) == 4) {
    const float f = fmaf(__uint2float_rn(lo), 0x1p-32f, 0x1p-33f);
    J.m = first ? ew.jm : __fmul_rn(J.m, ew.jm);
    J.e = first ? ew.je : J.e + ew.je;
    return fmaf(f, ew.w, ew.e);
  } else {
    const double f = ((double)lo + 0.5) * 0x1p-32;
    const double jf = s_jac[i];
    J.v = first ? jf : __dmul_rn(J.v, jf);
    return __dadd_rn(ew.e, __dmul_rn(f, ew.w));
  }
}

// |x| bits of a double, and its finiteness, on the integer pipes.
__device__ __forceinline__ unsigned long long gv_abs_bits(double x) {
  return (unsigned long long)__double_as_longlong(x) & 0x7FFFFFFFFFFFFFFFull;
}
__device__ __forceinline__ bool gv_finite_bits(unsigned long long absbits) {
  return absbits < 0x7FF0000000000000ull;
}

// The significand of the FP32 form's weight u 2^e (u the bits of the FP32
// product J.m g): 1 with w set (m in [2^23, 2^24)), 0 if the weight is zero or
// below the FP64 normal range, -1 if it is not finite or beyond FP64 -- as the
// double that gv_weight assembles.
__device__ __forceinline__ int gv_sig(unsigned u, int e, GvSig<float>& w) {
  int ef = (int)((u >> 23) & 0xFFu);
  unsigned m = (u & 0x7FFFFFu) | 0x800000u;
  if (ef == 0) {  // subnormal product
    m &= 0x7FFFFFu;
    if (m == 0u) return 0;
    const int lz = __clz((int)m) - 8;
    m <<= lz;
    ef = 1 - lz;
  }
  const int nf = ef + 896 + e;  // the double's exponent field
  if (ef == 0xFF || nf >= 0x7FF) return -1;
  if (nf <= 0) return 0;
  w.m = m;
  w.e2 = nf - 1046;
  w.neg = (u >> 31) != 0u;
  return 1;
}
// The FP64 form's: m in [2^52, 2^53), or 0 for a zero weight.
__device__ __forceinline__ GvSig<double> gv_sig(double x) {
  const GvDecoded d = gv_decode(x);
  GvSig<double> w;
  w.m = d.m;
  w.e2 = d.e2;
  w.neg = d.neg;
  if (d.e2 == -1074 && d.m != 0ull && (d.m >> 52) == 0ull) {  // subnormal
    const int lz = __clzll((long long)d.m) - 11;
    w.m <<= lz;
    w.e2 -= lz;
  }
  return w;
}

// One event between the two passes, in shared memory (evs, array j of slot s
// at evs[j T + s]): FP32 form, 0: sign and significand of w (0: no weight),
// 1: e2 + GV_SQ_OFF (12 bits) | bin 0 | bin 1 (10 bits each), 2: bin 2 | bin 3
// | the histogram's bin; with VEGAS+, 2: bin 2 | bin 3 | e2 of q, 3: q's sign
// and significand.  FP64 form: the double w (two words), then bins 0, 1 and
// bins 2, 3 | the histogram's bin; with VEGAS+ the double q at the end.  More
// than 4 axes: the bins elsewhere, the histogram's bin in word 1 (FP64: 2).
template <typename Real, bool REG, bool PLUS, int T>
struct GvEvent {
  static constexpr bool F64 = sizeof(Real) == 8;
  static constexpr int Q = F64 ? (REG ? 4 : 3) : 3;  // VEGAS+: first word of q's value
  unsigned* e;                                       // evs + slot
  // bins: 0, 1 and 2, 3 as pairs of 10 bits (at most 4 axes; else zero)
  __device__ __forceinline__ void put(const GvSig<float>& w, const GvSig<float>& q, uint2 bins,
                                      int hbin) const {
    e[0] = w.m | (w.neg ? 0x80000000u : 0u);
    e[T] = ((unsigned)(w.e2 + GV_SQ_OFF) << 20) | (REG ? bins.x : (unsigned)hbin);
    if constexpr (PLUS) {
      e[2 * T] = ((unsigned)(q.e2 + GV_SQ_OFF) << 20) | bins.y;
      e[Q * T] = q.m | (q.neg ? 0x80000000u : 0u);
    } else if constexpr (REG) {
      e[2 * T] = ((unsigned)hbin << 20) | bins.y;
    }
  }
  __device__ __forceinline__ void put(double w, double q, uint2 bins, int hbin) const {
    const unsigned long long b = (unsigned long long)__double_as_longlong(w);
    e[0] = (unsigned)b;
    e[T] = (unsigned)(b >> 32);
    if constexpr (REG) {
      e[2 * T] = bins.x;
      e[3 * T] = ((unsigned)hbin << 20) | bins.y;
    } else {
      e[2 * T] = (unsigned)hbin << 20;
    }
    if constexpr (PLUS) {
      const unsigned long long c = (unsigned long long)__double_as_longlong(q);
      e[Q * T] = (unsigned)c;
      e[(Q + 1) * T] = (unsigned)(c >> 32);
    }
  }
  __device__ __forceinline__ void none() const {
    e[0] = 0u;
    if constexpr (F64) e[T] = 0u;
    if constexpr (PLUS) e[Q * T] = 0u;
    if constexpr (PLUS && F64) e[(Q + 1) * T] = 0u;
  }
  // the weight (VEGAS+: which = 1, the bins' quantity); m = 0: none
  template <int WHICH>
  __device__ __forceinline__ GvSig<Real> get() const {
    if constexpr (!F64) {
      const unsigned sm = e[WHICH ? Q * T : 0];
      const unsigned x = e[WHICH ? 2 * T : T];
      return GvSig<float>{sm & 0xFFFFFFu, (int)(x >> 20) - GV_SQ_OFF, (sm >> 31) != 0u};
    } else {
      const unsigned long long b =
          ((unsigned long long)e[WHICH ? (Q + 1) * T : T] << 32) | e[WHICH ? Q * T : 0];
      return gv_sig(__longlong_as_double((long long)b));
    }
  }
  // bins 0, 1 (lo) and 2, 3 (hi), 10 bits each, for at most 4 axes
  __device__ __forceinline__ uint2 bins() const {
    return F64 ? make_uint2(e[2 * T], e[3 * T]) : make_uint2(e[T], e[2 * T]);
  }
  __device__ __forceinline__ int hbin() const {
    if constexpr (F64) return (int)(e[(REG ? 3 : 2) * T] >> 20);
    return REG ? (int)(e[2 * T] >> 20) : (int)(e[T] & 0xFFFFFu);
  }
};

// In memory: 48 bits of the upper word (two's complement), the position above.
__device__ __forceinline__ void gv_store_partial(ulonglong2* p, const GvPartial& v) {
  *p = make_ulonglong2(v.lo, (v.hi & 0xFFFFFFFFFFFFull) | ((unsigned long long)(unsigned)v.pos << 48));
}
__device__ __forceinline__ GvPartial gv_load_partial(const ulonglong2* p) {
  const ulonglong2 v = *p;
  return GvPartial{v.x, (unsigned long long)((long long)(v.y << 16) >> 16), (int)(v.y >> 48)};
}

// ---------------------------------------------------------------------------
// Forward fill of one tile: channel 0 = w, with per-bin sums of w^2.  The grid
// of the integration must be staged (followed by a barrier) before the call;
// `words`: the tile's Philox words lie in shared memory.  Used by the
// per-integration kernel and by the persistent batched kernel, so that a
// tile's partial is the same whichever kernel computes it.
//
// Both passes are rolled loops over the thread's events, which wait between
// them in shared memory (in the place of their words): unrolled over events in
// registers, the loop's constants no longer fit and were loaded again for
// every event.
// ---------------------------------------------------------------------------
template <int IG, typename Real, int EPT, int MAXD, bool HIST = false, bool PLUS = false>
__device__ __forceinline__ void gv_fill_tile(const GvFillArgs& a, long long tile,
                                             unsigned char* smem, const GvFillSmem& lay,
                                             uint32_t it, bool words = false) {
  constexpr int B = GV_TILE / EPT, T = GV_TILE;  // T: stride of the arrays
  constexpr int NW = B / 32;
  using W = typename GvForm<Real>::W;
  constexpr bool F64 = sizeof(W) == 8;
  using Pair = typename GvPair<Real>::T;
  constexpr bool REG = MAXD <= 4;  // bins held in the event's words
  using Event = GvEvent<W, REG, PLUS, T>;
  __shared__ int s_max[2][NW];
  const int d = a.ndim, N = a.nbins, dN = d * N, L = lay.L;
  const int hb = HIST ? a.nhist : 0;
  const int* s_off = reinterpret_cast<const int*>(smem + lay.po);
  double2* s_seg = reinterpret_cast<double2*>(smem + lay.ps);
  const GvPlusFill* pf = a.plus;
  const long long ncall = PLUS ? *pf->ncall : a.ncall;
  const long long h0 = PLUS ? pf->tile_h0[tile] : 0;
  const double* s_jac = reinterpret_cast<const double*>(smem + lay.jac);
  const Pair* s_ew = reinterpret_cast<const Pair*>(smem + lay.ew);
  unsigned char* s_bin = smem + lay.bins;                      // [d][T]
  unsigned char* s_binh = N > 256 ? s_bin + d * T : nullptr;  // their high bytes
  unsigned* evs = reinterpret_cast<unsigned*>(smem + lay.wd);
  const int tid = threadIdx.x;
  const long long tile0 = tile * a.tile_events;
  const int n_ev = (int)min((long long)a.tile_events, ncall - tile0);  // events of this tile
  const int nk = PLUS ? EPT : (a.tile_events + B - 1) / B;             // events per thread

  int mw = GV_EMPTY;                   // the largest exponent of the thread's weights
  [[maybe_unused]] int mq = GV_EMPTY;  // and (VEGAS+) of the bins' quantities F b_h
  {
    GvConst<Real, GvTraits<IG>::NK> K;
    if constexpr (GvForm<Real>::ID == GV_FORM_X64) {
      constexpr int NX = GvTraits<IG>::NX;
      __shared__ GvX s_k[NX];
      if (tid < NX) s_k[tid] = gv_x_const<IG>(a.kconst, tid, d);
      __syncthreads();
      K.k = s_k;
    } else {
      K.load(a.kconst);
    }
    unsigned nbad = 0u;
    // VEGAS+: this thread's range (events tile0 + tid EPT ..), the window index
    // of its current hypercube, that hypercube's digits and factors, and the
    // running segment sums
    static_assert(!PLUS || EPT == GV_PLUS_SEG, "a stratified fill thread holds one range");
    [[maybe_unused]] int jc = PLUS ? gv_plus_cube(s_off, tid * EPT) : 0;
    [[maybe_unused]] int jcur = -1;  // the open segment's window index
    [[maybe_unused]] double sg1 = 0.0, sg2 = 0.0;
    constexpr bool KEEP_DIGITS = MAXD <= 4;  // registers to spare only for few axes
    [[maybe_unused]] unsigned cdig[PLUS ? MAXD : 1];
#pragma unroll 1
    for (int k = 0; k < nk; ++k) {
      const int local = PLUS ? tid * EPT + k : k * B + tid;
      const int slot = k * B + tid;
      const Event event{evs + slot};
      if (local >= n_ev) {
        event.none();
        continue;
      }
      GvStream<IG, Real> S;
      GvJac<Real> J;
      uint2 bins = make_uint2(0u, 0u);
      const auto put_bin = [&](int ax, int bin) {
        if constexpr (!REG) {
          s_bin[ax * T + slot] = (unsigned char)bin;
          if (s_binh) s_binh[ax * T + slot] = (unsigned char)(bin >> 8);
        }
      };
      // four coordinates before the first is used or its bin stored: their loads
      // and products overlap (ten iterations of 1e6 Drell-Yan events 429 -> 417
      // us in FP32, 1249 -> 1207 in FP64; the Gaussian and three jets, whose
      // axes do less, gain nothing)
      const auto map4 = [&](int ax, const uint32_t* r, auto use) {
        typename GvForm<Real>::Coord v[4];
        int bin[4];
#pragma unroll
        for (int k = 0; k < 4; ++k)
          v[k] = gv_map_axis<Real>(r[k], N, s_jac + (ax + k) * N, s_ew + (ax + k) * N,
                                   ax + k == 0, J, bin[k]);
#pragma unroll
        for (int k = 0; k < 4; ++k) use(k, v[k], bin[k]);
      };
      const auto first = [&](int k, const auto& v, int bin) {
        S.first(k, v, K);
        if constexpr (REG)
          (k < 2 ? bins.x : bins.y) |= (unsigned)bin << (10 * (k & 1));
        else
          put_bin(k, bin);
      };
      const auto axes4 = [&](const uint32_t* r) {  // axes 0..3
        if constexpr (IG == GV_DY || IG == GV_DYNLO) {
          map4(0, r, first);
        } else {
#pragma unroll
          for (int k = 0; k < 4; ++k) {
            if (IG != GV_GAUSS || k < d) {  // (the others have four or more)
              int bin;
              const auto v =
                  gv_map_axis<Real>(r[k], N, s_jac + k * N, s_ew + k * N, k == 0, J, bin);
              first(k, v, bin);
            }
          }
        }
      };
      const auto axis = [&](int ax, uint32_t r) {  // an axis past those
        int bin;
        S.more(ax, gv_map_axis<Real>(r, N, s_jac + ax * N, s_ew + ax * N, false, J, bin), K);
        put_bin(ax, bin);
      };
      if constexpr (PLUS) {
        uint32_t r[MAXD];
        if (words) {  // generated before the wait, by this thread
#pragma unroll
          for (int j = 0; j < MAXD; ++j)
            if (j < d) r[j] = evs[j * T + slot];
        } else {
          gv_event_words<MAXD>(a.seed, it, a.batch, (unsigned long long)(tile0 + local), d, r);
        }
        while (jc + 1 < GV_PLUS_WIN && s_off[jc + 1] <= local) ++jc;
        if (jc != jcur) {  // a new hypercube: close the previous segment
          if (jcur >= 0)
            gv_plus_put_segment(pf, s_off, s_seg, h0, jcur, tile0, tid * EPT, sg1, sg2);
          jcur = jc;
          sg1 = 0.0;
          sg2 = 0.0;
          if (KEEP_DIGITS)
            gv_plus_digits<MAXD>((unsigned)(h0 + jc), d, (unsigned)pf->s, pf->inv_s, cdig);
        }
        if (!KEEP_DIGITS)
          gv_plus_digits<MAXD>((unsigned)(h0 + jc), d, (unsigned)pf->s, pf->inv_s, cdig);
        gv_plus_strat<MAXD>(cdig, d, (unsigned)pf->s, pf->magic, r);
        axes4(r);
#pragma unroll
        for (int ax = 4; ax < MAXD; ++ax)
          if (ax < d) axis(ax, r[ax]);
      } else {
        // one Philox block (4 axes) at a time
        const unsigned long long ev = (unsigned long long)(tile0 + local);
        const auto block = [&](int j, uint32_t (&r)[4]) {
          if (words) {  // generated before the wait, by this thread
#pragma unroll
            for (int k = 0; k < 4; ++k)
              if (4 * j + k < d) r[k] = evs[(4 * j + k) * T + slot];
          } else {
            const uint4 o = gv_philox(make_uint4((uint32_t)ev, (uint32_t)(ev >> 32), it,
                                                 (a.batch << 8) | (uint32_t)j),
                                      (uint32_t)a.seed, (uint32_t)(a.seed >> 32));
            r[0] = o.x;
            r[1] = o.y;
            r[2] = o.z;
            r[3] = o.w;
          }
        };
        uint32_t r[4];
        block(0, r);
        axes4(r);
        if constexpr (!REG) {
#pragma unroll 1
          for (int j = 1; 4 * j < d; ++j) {
            block(j, r);
            if ((IG == GV_DY || IG == GV_DYNLO) && 4 * j + 4 <= d) {
              map4(4 * j, r, [&](int k, const auto& v, int bin) {
                S.more(4 * j + k, v, K);
                put_bin(4 * j + k, bin);
              });
            } else {
#pragma unroll
              for (int k = 0; k < 4; ++k)
                if (4 * j + k < d) axis(4 * j + k, r[k]);
            }
          }
        }
      }
      const Real g = S.value(d, K);
      int hbin = 0;
      if constexpr (HIST) {
        if constexpr (F64)
          hbin = gv_hist_bin<W>(S.observable(K), a.h_lo, a.h_invw, hb - 2);
        else
          hbin = gv_hist_bin<W>(S.observable(K), a.h_lo_f, a.h_invw_f, hb - 2);
      }
      if constexpr (!F64) {
        const unsigned u = __float_as_uint(__fmul_rn(J.m, g));
        // VEGAS+: the estimate's weight u a_h and the bins' quantity u b_h,
        // FP32 products with the hypercube's factors rounded to FP32
        unsigned uw = u;
        [[maybe_unused]] unsigned uq = u;
        if constexpr (PLUS) {
          const float2 f = pf->ab32[h0 + jc];
          uw = __float_as_uint(__fmul_rn(__uint_as_float(u), f.x));
          uq = __float_as_uint(__fmul_rn(__uint_as_float(u), f.y));
        }
        GvSig<float> sw = {0u, 0, false}, sq = {0u, 0, false};
        const int kw = gv_sig(uw, J.e, sw);
        const int kq = PLUS ? gv_sig(uq, J.e, sq) : kw;
        const bool fin = kw >= 0 && kq >= 0;
        if constexpr (PLUS) {
          if (fin && (u & 0x7FFFFFFFu) != 0u) {
            // F = u 2^e, widened exactly, into the segment (a rounded
            // product, then the sum, as the statistics define them: the
            // variance cancels where a hypercube's values are nearly equal)
            double Fv = gv_weight_bits(u, J.e);
            Fv = gv_finite_bits(gv_abs_bits(Fv)) ? Fv : 0.0;
            sg1 += Fv;
            sg2 += Fv * Fv;
          }
          if (fin && kq > 0) mq = max(mq, sq.e2);
        }
        if (fin && kw > 0) mw = max(mw, sw.e2);
        if (fin && (kw > 0 || kq > 0)) {
          if (kw <= 0) sw = GvSig<float>{0u, 0, false};
          if (PLUS && kq <= 0) sq = GvSig<float>{0u, 0, false};
          event.put(sw, sq, bins, hbin);
        } else {
          event.none();
        }
        if (!fin) ++nbad;  // counted, contributes nothing
      } else {
        double wv = gv_weight(J, g);
        [[maybe_unused]] double qk = 0.0;
        bool fin = gv_finite_bits(gv_abs_bits(wv));
        if constexpr (PLUS) {
          // F = J g into the segment (0 if not finite); the estimate's weight
          // F C/(nh n_h), the bins' F sqrt(1/(nh n_h))
          // (a rounded product, then the sum, as the statistics define them: the
          // variance cancels where a hypercube's values are nearly equal)
          const double Fv = fin ? wv : 0.0;
          sg1 += Fv;
          sg2 += Fv * Fv;
          const double2 f = pf->ab[h0 + jc];
          qk = wv * f.y;
          wv = wv * f.x;
          fin = gv_finite_bits(gv_abs_bits(wv)) && gv_finite_bits(gv_abs_bits(qk));
        }
        if (fin) {
          event.put(wv, qk, bins, hbin);
          if (gv_abs_bits(wv) != 0ull) mw = max(mw, gv_scale_exp(gv_abs_bits(wv)) - 53);
          if constexpr (PLUS)
            if (gv_abs_bits(qk) != 0ull) mq = max(mq, gv_scale_exp(gv_abs_bits(qk)) - 53);
        } else {
          event.none();
          ++nbad;  // counted, contributes nothing
        }
      }
    }
    if constexpr (PLUS) {
      // the range's last segment and its first hypercube
      if (jcur >= 0) gv_plus_put_segment(pf, s_off, s_seg, h0, jcur, tile0, tid * EPT, sg1, sg2);
    }
    if (nbad) atomicAdd(&a.st->nonfinite_iter, (unsigned long long)nbad);
  }

  // pass 2, once for each window of limbs (one, unless weights lie below it)
  unsigned* hist = reinterpret_cast<unsigned*>(smem + lay.hist);  // [dN][L]
  [[maybe_unused]] unsigned* hh = reinterpret_cast<unsigned*>(smem + lay.hh);  // [hb][L]
  [[maybe_unused]] int* hw = reinterpret_cast<int*>(smem + lay.hw);            // [hb][HW]
  unsigned* lq = reinterpret_cast<unsigned*>(smem + lay.lq);
  int* lw = reinterpret_cast<int*>(smem + lay.lw);
  [[maybe_unused]] const int HW = gv_hist_w_limbs(F64, L);
  const int lane = tid & 31, wid = tid >> 5;
  const unsigned a_hist = gv_shared_address(hist), a_lq = gv_shared_address(lq + lane),
                 a_lw = gv_shared_address(lw + lane);
  [[maybe_unused]] const unsigned hcopy = (unsigned)(lane & (lay.hc - 1)) * lay.hs;
  [[maybe_unused]] const unsigned a_hh = gv_shared_address(hh) + hcopy,
                                  a_hw = gv_shared_address(hw) + hcopy;
  const unsigned L4 = 4u * (unsigned)L, axis4 = L4 * (unsigned)N;  // bytes of a bin, of an axis
  // the tile's slots: slot k at out[k ks] (tile-major or slot-major partials)
  const size_t ks = a.slot_major ? (size_t)a.n_tiles : (size_t)1;
  ulonglong2* out = a.part + (a.slot_major ? (size_t)tile : (size_t)tile * a.nacc);
  int E = GV_EMPTY;         // the tile's scale: |w| < 2^E
  // the tile's sums (gv_lane_sum) of w^2 and of w, by the last two warps: the first
  // ones have more bins below (wsum 0 and 1; the others 2 and more)
  const int wsum = NW - 1 - wid;
  u192 sum = {0ull, 0ull, 0ull};
  // weights at limb indices of at least up_w have been added (VEGAS+: q, up_q)
  int up_w = 0x40000000;
  [[maybe_unused]] int up_q = 0x40000000;
  bool first = true;
  for (;;) {
    mw = __reduce_max_sync(0xffffffffu, mw);
    if constexpr (PLUS) mq = __reduce_max_sync(0xffffffffu, mq);
    if (lane == 0) {
      s_max[0][wid] = mw;
      if constexpr (PLUS) s_max[1][wid] = mq;
    }
    __syncthreads();
    mw = __reduce_max_sync(0xffffffffu, s_max[0][lane % NW]);
    if constexpr (PLUS) mq = __reduce_max_sync(0xffffffffu, s_max[1][lane % NW]);
    const bool have_w = mw != GV_EMPTY, have_q = PLUS ? mq != GV_EMPTY : have_w;
    GvWindow vw = gv_window<W>(have_w ? mw : 0, L);
    GvWindow vq = PLUS ? gv_window<W>(have_q ? mq : 0, L) : vw;
    if (!have_w) vw.base = up_w;  // nothing (left)
    if (PLUS && !have_q) vq.base = up_q;
    if (first && have_w) E = mw + GvSig<W>::BITS;
    {
      uint4* z = reinterpret_cast<uint4*>(smem + lay.limbs);
      const int nz = (int)((lay.limb_bytes(F64) + 15) / 16);
      for (int k = tid; k < nz; k += B) z[k] = make_uint4(0u, 0u, 0u, 0u);
    }
    __syncthreads();
    mw = GV_EMPTY;
    mq = GV_EMPTY;
#pragma unroll 1
    for (int k = 0; k < nk; ++k) {
      const int slot = k * B + tid;
      const Event event{evs + slot};
      const auto add_bins = [&](const unsigned (&l)[4], int pos) {
        unsigned row = a_hist + 4u * (unsigned)pos;
        if constexpr (REG) {
          const uint2 b = event.bins();
#pragma unroll
          for (int ax = 0; ax < 4; ++ax) {
            if (ax < d) {
              gv_bin_add_square<W>(l, row + (((ax < 2 ? b.x : b.y) >> (10 * (ax & 1))) & 0x3FFu) * L4);
              row += axis4;
            }
          }
        } else {
#pragma unroll 4
          for (int ax = 0; ax < d; ++ax) {
            unsigned bin = s_bin[ax * T + slot];
            if (s_binh) bin |= (unsigned)s_binh[ax * T + slot] << 8;
            gv_bin_add_square<W>(l, row + bin * L4);
            row += axis4;
          }
        }
      };
      {
        const GvSig<W> s = event.template get<0>();
        const int h = s.e2 + GvSig<W>::H;
        const int limb = gv_limb_index(h), pos = limb - vw.base;
        if (s.m != 0 && limb < up_w) {
          if (pos >= 0) {
            unsigned l[4];
            const int rem = h + GV_SQ_OFF - 11 * limb;
            gv_square_digits(s, rem, l);
            gv_lane_add_square(s, rem, l, a_lq + pos * 128);
            gv_lane_add_w(s, a_lw, vw.wbase);
            if constexpr (!PLUS) add_bins(l, pos);
            if constexpr (HIST) {
              const int hbin = event.hbin();
              gv_bin_add_square<W>(l, a_hh + 4 * (pos + hbin * L));
              gv_hist_add_w<W>(s, a_hw + 4 * (hbin * HW), vw.hbase);
            }
          } else {
            mw = max(mw, s.e2);
          }
        }
      }
      if constexpr (PLUS) {
        const GvSig<W> s = event.template get<1>();
        const int h = s.e2 + GvSig<W>::H;
        const int limb = gv_limb_index(h), pos = limb - vq.base;
        if (s.m != 0 && limb < up_q) {
          if (pos >= 0) {
            unsigned l[4];
            gv_square_digits(s, h + GV_SQ_OFF - 11 * limb, l);
            add_bins(l, pos);
          } else {
            mq = max(mq, s.e2);
          }
        }
      }
    }
    const bool more = __syncthreads_or((int)(mw != GV_EMPTY || (PLUS && mq != GV_EMPTY))) != 0;
    if (first) gv_allow_next_grid();
    if constexpr (HIST) {
      const int hsw = (int)(lay.hs / 4);
      if (lay.hc > 1)  // the copies into the first one
        for (int k = tid; k < hb * (L + HW); k += B)
          hh[k] += hh[k + hsw] + hh[k + 2 * hsw] + hh[k + 3 * hsw];
    }
    if (have_w && wsum == 0)
      add192(sum, gv_lane_sum<false>(lq, L + GvSig<W>::LOW,
                                     vw.base - GvSig<W>::LOW - gv_square_cut(E)));
    else if (have_w && wsum == 1)
      add192(sum, gv_lane_sum<true>(reinterpret_cast<const unsigned*>(lw), gv_lane_rows(F64, L),
                                    vw.wbase - gv_w_cut(E)));
    ulonglong2* o = out + (size_t)(2 + tid) * ks;
    for (int k = tid; k < dN; k += B, o += (size_t)B * ks) {
      GvPartial v = gv_bin_partial(hist + k * L, L, vq.base);
      if (!first) {  // few bins have weights below the first window
        if (v.pos == 0) continue;
        const GvPartial x = gv_load_partial(o);
        if (x.pos) v = gv_bin_partial_more(x, hist + k * L, L, vq.base);
      }
      gv_store_partial(o, v);
    }
    if constexpr (HIST) {
      if (lay.hc > 1) __syncthreads();
      for (int k = tid; k < hb; k += B) {
        ulonglong2* o = out + (2 + dN + k) * ks;
        GvPartial v = gv_bin_partial(hh + k * L, L, vw.base);
        if (!first) {
          if (v.pos == 0) continue;  // (nor has the bin a sum of w)
          const GvPartial x = gv_load_partial(o);
          if (x.pos) v = gv_bin_partial_more(x, hh + k * L, L, vw.base);
        }
        gv_store_partial(o, v);
        o = out + (2 + dN + hb + k) * ks;
        v = gv_hist_partial(hw + k * HW, HW, vw.hbase);
        if (!first) v = gv_hist_partial_add(v, gv_load_partial(o));
        gv_store_partial(o, v);
      }
    }
    if (!more) break;
    first = false;
    up_w = vw.base;
    if constexpr (PLUS) up_q = vq.base;
  }
  if (lane == 0 && wsum < 2) {  // at the tile's scale, bits below a unit dropped once
    if (E != GV_EMPTY)
      sum = sar192(sum, wsum == 0 ? 2 * E - GV_FB + 2 * GV_SQ_OFF - 22 * gv_square_cut(E)
                                 : E - GV_FB + GV_SQ_OFF - 22 * gv_w_cut(E));
    out[wsum == 0 ? ks : (size_t)0] = make_ulonglong2(sum.l0, sum.l1);
  }
  if (tid == 0) a.tileE[tile] = E;
  if constexpr (PLUS) {
    // the hypercubes this tile holds whole (the barriers above ordered the
    // staged segments)
    __shared__ double2 s_pr[PLUS ? B : 1];
    gv_plus_tile_stats<B>(pf, s_off, s_seg, h0, tile, s_pr);
  }
}

// The Philox words of a tile's events at counter `it` into shared memory
// (word a of slot s at s_words[a T + s]); each thread makes the words of the
// events it will evaluate, so no barrier is needed before use.
template <int T, int B, bool PLUS>
__device__ __forceinline__ void gv_tile_words(const GvFillArgs& a, uint32_t it, long long tile,
                                              unsigned* s_words) {
  const int d = a.ndim;
  const long long t0 = tile * a.tile_events;
  const int nk = PLUS ? T / B : (a.tile_events + B - 1) / B;
#pragma unroll 1
  for (int k = 0; k < nk; ++k) {
    const int local = PLUS ? (int)threadIdx.x * (T / B) + k : k * B + (int)threadIdx.x;
    const int slot = k * B + (int)threadIdx.x;
    const unsigned long long ev = (unsigned long long)(t0 + local);
#pragma unroll 1
    for (int j = 0; 4 * j < d; ++j) {
      const uint4 o = gv_philox(
          make_uint4((uint32_t)ev, (uint32_t)(ev >> 32), it, (a.batch << 8) | (uint32_t)j),
          (uint32_t)a.seed, (uint32_t)(a.seed >> 32));
      unsigned* w = s_words + 4 * j * T + slot;
      w[0] = o.x;
      w[T] = o.y;
      w[2 * T] = o.z;
      w[3 * T] = o.w;
    }
  }
}

// Minimum resident CTAs per SM in the fill's launch bound (0: none), i.e. its
// register budget: 64 registers for FP32 fills at any width, 80 for the
// stratified ones of 5 to 8 axes and none above (they would spill); FP64
// fills: none.
template <typename Real, int EPT, int MAXD, bool PLUS>
struct GvFillBlocks {
  static constexpr int B = GV_TILE / EPT;
  static constexpr int value = GvForm<Real>::ID != GV_FORM_F32 ? 0
                               : (PLUS && MAXD == 16)  ? 0
                               : (PLUS && MAXD == 8)   ? 3
                                                       : 65536 / (64 * B);
};

template <int IG, typename Real, int EPT, int MAXD, bool HIST = false, bool PLUS = false>
__global__ void __launch_bounds__(GV_TILE / EPT, (GvFillBlocks<Real, EPT, MAXD, PLUS>::value))
    gv_fill_kernel(const GvFillArgs a) {
  constexpr int B = GV_TILE / EPT, T = GV_TILE;
  extern __shared__ __align__(16) unsigned char smem[];
  const int d = a.ndim, N = a.nbins;
  const bool hoist = a.hoist;  // set by the host (gv_fill_hoistable)
  const GvFillSmem lay(d, N, GvForm<Real>::ID, true, MAXD > 4, HIST ? a.nhist : 0, PLUS, hoist);
  // the tile's words at the counter this iteration should have (the stage's
  // first counter, which no running kernel writes, plus the iteration index),
  // made while the previous iteration's reduce and refinement finish
  unsigned* s_words = reinterpret_cast<unsigned*>(smem + lay.wd);
  uint32_t itg = 0u;
  if (hoist) {
    itg = (uint32_t)(a.st->it0 + (unsigned long long)a.kst);
    gv_tile_words<T, B, PLUS>(a, itg, blockIdx.x, s_words);
  }
  gv_wait_prior_grid();  // grid, constants and iteration counter come from earlier kernels
  if constexpr (PLUS) {
    // VEGAS+ sizes the grid for the most events an allocation can have; the
    // iteration's events fill the first tiles_used tiles, which alone the
    // reduce reads, and a tile past them does nothing
    const long long ncall = *a.plus->ncall;
    if (blockIdx.x == 0 && threadIdx.x == 0)
      *a.plus->tiles_used = (int)((ncall + GV_TILE - 1) / GV_TILE);
    if ((long long)blockIdx.x * GV_TILE >= ncall) return;
  }
  gv_stage_grid<Real>(a.grid, d, N, reinterpret_cast<double*>(smem + lay.jac),
                      reinterpret_cast<typename GvPair<Real>::T*>(smem + lay.ew), threadIdx.x, B);
  if constexpr (PLUS) {
    // the offsets of the hypercubes this tile can meet, relative to its first
    // event and clamped to [-1, GV_TILE + 1]
    int* s_off = reinterpret_cast<int*>(smem + lay.po);
    const GvPlusFill* pf = a.plus;
    const long long h0 = pf->tile_h0[blockIdx.x];
    const long long t0 = (long long)blockIdx.x * GV_TILE;
    for (int j = threadIdx.x; j < GV_PLUS_WIN; j += B) {
      int v = GV_TILE + 1;
      if (h0 + j <= pf->nh) {
        const long long o = pf->off[h0 + j] - t0;
        v = o < -1 ? -1 : (o > GV_TILE ? GV_TILE + 1 : (int)o);
      }
      s_off[j] = v;
    }
  }
  const uint32_t it = (uint32_t)a.st->it;
  if (hoist && it != itg) gv_tile_words<T, B, PLUS>(a, it, blockIdx.x, s_words);  // (not expected)
  __syncthreads();
  gv_fill_tile<IG, Real, EPT, MAXD, HIST, PLUS>(a, blockIdx.x, smem, lay, it,
                                                hoist);
}

// Single-event diagnostics (no shared memory): weight and bins of the given
// events at iteration `it`, with the same map and integrand code as the fill.
template <int IG, typename Real>
__global__ void gv_eval_events_kernel(const GvFillArgs a, uint32_t it, const long long* events,
                                      long long n, double* w, int* bins) {
  constexpr int MAXD = GV_MAXD;
  const long long j = (long long)blockIdx.x * blockDim.x + threadIdx.x;
  const int d = a.ndim, N = a.nbins;
  GvConst<Real, GvTraits<IG>::NK> K;
  if constexpr (GvForm<Real>::ID == GV_FORM_X64) {
    __shared__ GvX s_k[GvTraits<IG>::NX];
    if (threadIdx.x < GvTraits<IG>::NX)
      s_k[threadIdx.x] = gv_x_const<IG>(a.kconst, (int)threadIdx.x, d);
    __syncthreads();
    K.k = s_k;
  } else {
    K.load(a.kconst);
  }
  if (j >= n) return;
  const GvGridLayout L{d, N};
  const double* e64 = a.grid + L.off_e64();
  const double* wd64 = a.grid + L.off_wd64();
  const double* jac = a.grid + L.off_jac();
  const GvBin32* b32 = reinterpret_cast<const GvBin32*>(a.grid + L.off_bin32());
  uint32_t r[MAXD];
  gv_event_words<MAXD>(a.seed, it, a.batch, (unsigned long long)events[j], d, r);
  GvStream<IG, Real> S;
  GvJac<Real> J;
#pragma unroll
  for (int ax = 0; ax < MAXD; ++ax) {
    if (ax < d) {
      // the bin's record, as gv_stage_grid stages it, on its own
      const int i = (int)(((unsigned long long)r[ax] * (unsigned)N) >> 32), k = ax * N + i;
      typename GvPair<Real>::T rec;
      if constexpr (GvForm<Real>::ID == GV_FORM_X64)
        rec = gv_bin_x(e64[ax * (N + 1) + i], wd64[k], N);
      else if constexpr (sizeof(Real) == 4)
        rec = b32[k];
      else
        rec = GvBin64{e64[ax * (N + 1) + i], wd64[k]};
      int bin;
      const auto x = gv_map_axis<Real>(r[ax], N, jac + ax * N, &rec - i, ax == 0, J, bin);
      if (ax < 4)
        S.first(ax < 4 ? ax : 0, x, K);
      else
        S.more(ax, x, K);
      bins[j * d + ax] = bin;
    }
  }
  w[j] = gv_weight(J, S.value(d, K));
}
