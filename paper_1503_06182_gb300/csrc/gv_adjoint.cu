// Adjoint fill kernels (Drell-Yan gradient).
//
// Six channels per event: the weight w and dw/d(M_Z, Gamma_Z, sw2, a, b) from
// the reverse sweep of the integrand.  No bin sums: the grid is frozen during
// a gradient stage.  Each channel gets its own tile scale E_c (the exponent of
// the tile's largest |value| in that channel) and contributes two exact 128-bit
// fixed-point sums (values and squares) to the tile's partial, as the forward
// fill does for its one channel.
//
// Bound by instruction issue.  As in the forward fill, both passes are rolled
// loops and the events' six values wait between them in shared memory (FP32
// form: the FP32 products J.m g and the exponent J.e, 28 KB a tile; FP64 form:
// the weights, 48 KB); the second pass adds each value's and its square's
// digits to per-lane columns of limbs (gv_limbs.cuh): about 45 instructions a
// channel, where 128-bit shifts and adds in registers and a reduce-scatter of
// twelve 128-bit sums per warp took twice that.  1e8 FP32 events on 4 axes: 3.60
// ms before, 2.74 now (1136 and 925 instructions per event, 84% of issue slots);
// 1e5 FP64 events 75 and 38 us.
#include "gv_fill_inst.cuh"

namespace {

constexpr int kNch = GV_MAXCH;   // channels
constexpr int kNsum = 2 * kNch;  // per channel: sum v, sum v^2
constexpr int kL = 9;            // limbs of a square's column

// Shared memory of the adjoint fill (bytes, 16-byte aligned): the events'
// values, the lanes' columns, the grid.
template <typename Real>
struct AdjSmem {
  static constexpr bool F64 = GvForm<Real>::ID != GV_FORM_F32;
  static constexpr int WORDS = F64 ? 2 * kNch : kNch + 1;  // per event
  static constexpr int SQ = kL + (F64 ? GvSig<double>::LOW : 0);
  static constexpr int ROWS = SQ + gv_lane_rows(F64);      // per channel: of v^2, then of v
  static constexpr size_t lanes = (size_t)WORDS * GV_TILE * 4;
  static constexpr size_t grid = lanes + (size_t)kNch * ROWS * 32 * 4;
};

// Register budget of the FP32 kernels: 64 registers at 1024 or 512 threads
// (one or two CTAs per SM), and four CTAs at 256.  The FP64 kernels would
// spill under it and keep their own.
template <typename Real, int EPT>
struct AdjBlocks {
  static constexpr int value = GvForm<Real>::ID == GV_FORM_F32 ? (EPT == 4 ? 4 : (EPT == 2 ? 2 : 1)) : 1;
};

}  // namespace

template <typename Real, int EPT, int MAXD>
__global__ void __launch_bounds__(GV_TILE / EPT, AdjBlocks<Real, EPT>::value)
    gv_fill_adjoint_kernel(const GvFillArgs a) {
  constexpr int B = GV_TILE / EPT, T = GV_TILE;  // T: stride of the events' arrays
  constexpr int NW = B / 32;
  using Lay = AdjSmem<Real>;
  using W = typename GvForm<Real>::W;
  using Pair = typename GvPair<Real>::T;
  constexpr bool F64 = Lay::F64;
  constexpr int kOdd = 1 << 30;  // on J.e: a product or exponent out of the ordinary
  extern __shared__ __align__(16) unsigned char smem[];
  __shared__ int s_max[kNch][NW], s_E[kNch];
  __shared__ int4 s_win[kNch];  // the window's base and wbase, the limb index below which
                                // values are still to be added, whether there are any
  __shared__ u128 s_sum[kNsum];
  const int d = a.ndim, N = a.nbins;
  const GvFillSmem lay(d, N, GvForm<Real>::ID, false, false);
  double* s_jac = reinterpret_cast<double*>(smem + Lay::grid + lay.jac);
  Pair* s_ew = reinterpret_cast<Pair*>(smem + Lay::grid + lay.ew);
  unsigned* evs = reinterpret_cast<unsigned*>(smem);            // [WORDS][T]
  unsigned* cols = reinterpret_cast<unsigned*>(smem + Lay::lanes);  // [channel][ROWS][32]
  const int tid = threadIdx.x, lane = tid & 31, wid = tid >> 5;
  gv_wait_prior_grid();
  gv_stage_grid<Real>(a.grid, d, N, s_jac, s_ew, tid, B);
  GvConst<Real, DK_NK> K;
  if constexpr (GvForm<Real>::ID == GV_FORM_X64) {
    __shared__ GvX s_k[XK_N];  // (the barrier below)
    if (tid < XK_N) s_k[tid] = gv_x_consts(a.kconst)[tid];
    K.k = s_k;
  } else {
    K.load(a.kconst);
  }
  if (tid < kNsum) s_sum[tid] = u128{0ull, 0ull};
  if (tid < kNch) s_E[tid] = GV_EMPTY;
  const uint32_t it = (uint32_t)a.st->it;
  __syncthreads();

  const long long tile = blockIdx.x;
  const long long tile0 = tile * a.tile_events;
  const int n_ev = (int)min((long long)a.tile_events, a.ncall - tile0);
  const int nk = (a.tile_events + B - 1) / B;
  int mE[kNch];  // per channel the largest exponent of the thread's values
#pragma unroll
  for (int c = 0; c < kNch; ++c) mE[c] = GV_EMPTY;
  unsigned nbad = 0u;
#pragma unroll 1
  for (int k = 0; k < nk; ++k) {
    const int slot = k * B + tid;
    bool keep = false;
    if (slot < n_ev) {
      uint32_t r[MAXD];
      gv_event_words<MAXD>(a.seed, it, a.batch, (unsigned long long)(tile0 + slot), d, r);
      typename GvForm<Real>::Coord x[MAXD];
      GvJac<Real> J;
#pragma unroll
      for (int ax = 0; ax < MAXD; ++ax) {
        int bin;
        if (ax < d)
          x[ax] = gv_map_axis<Real>(r[ax], N, s_jac + ax * N, s_ew + ax * N, ax == 0, J, bin);
      }
      Real gr[1 + GV_NGRAD];
      if constexpr (GvForm<Real>::ID == GV_FORM_X64)
        gr[0] = gv_drell_yan_x<true>(x, K.k, gr + 1);
      else
        gr[0] = gv_drell_yan<Real, true>(x, K, gr + 1);
      int ex[kNch];
      keep = true;  // every channel finite
      if constexpr (!F64) {
        // ordinary: every product zero or a normal FP32 number, and every
        // weight in FP64's normal range whatever the product's exponent;
        // otherwise gv_sig sorts it out, here and below
        bool odd = J.e < -890 || J.e > 890;
        unsigned pu[kNch];
#pragma unroll
        for (int c = 0; c < kNch; ++c) {
          pu[c] = __float_as_uint(__fmul_rn(J.m, gr[c]));
          const unsigned ef = (pu[c] >> 23) & 0xFFu;
          odd = odd || ef == 0xFFu || (ef == 0u && (pu[c] << 1) != 0u);
          ex[c] = ef ? (int)ef + J.e - 150 : GV_EMPTY;
          evs[c * T + slot] = pu[c];
        }
        if (odd) {
#pragma unroll
          for (int c = 0; c < kNch; ++c) {
            GvSig<float> s;
            const int ks = gv_sig(pu[c], J.e, s);
            keep = keep && ks >= 0;
            ex[c] = ks > 0 ? s.e2 : GV_EMPTY;
          }
        }
        evs[kNch * T + slot] = (unsigned)(odd ? J.e + kOdd : J.e);
      } else {
#pragma unroll
        for (int c = 0; c < kNch; ++c) {
          const double v = gv_weight(J, gr[c]);
          const unsigned long long b = gv_abs_bits(v);
          keep = keep && gv_finite_bits(b);
          ex[c] = b ? gv_scale_exp(b) - 53 : GV_EMPTY;
          const unsigned long long u = (unsigned long long)__double_as_longlong(v);
          evs[2 * c * T + slot] = (unsigned)u;
          evs[(2 * c + 1) * T + slot] = (unsigned)(u >> 32);
        }
      }
      if (keep) {
#pragma unroll
        for (int c = 0; c < kNch; ++c) mE[c] = max(mE[c], ex[c]);
      } else {
        ++nbad;  // counted, contributes nothing
      }
    }
    if (!keep) {
#pragma unroll
      for (int j = 0; j < Lay::WORDS; ++j) evs[j * T + slot] = 0u;
    }
  }
  gv_allow_next_grid();

  // pass 2, once for each set of windows (see gv_fill_tile)
  bool first = true;
  for (;;) {
#pragma unroll
    for (int c = 0; c < kNch; ++c) {
      const int m = __reduce_max_sync(0xffffffffu, mE[c]);
      if (lane == 0) s_max[c][wid] = m;
    }
    __syncthreads();
    if (tid < kNch) {
      int m = s_max[tid][0];
#pragma unroll
      for (int w = 1; w < NW; ++w) m = max(m, s_max[tid][w]);
      const bool have = m != GV_EMPTY;
      const int up = first ? 0x40000000 : s_win[tid].x;
      const GvWindow v = gv_window<W>(have ? m : 0, kL);
      if (first && have) s_E[tid] = m + GvSig<W>::BITS;
      s_win[tid] = make_int4(have ? v.base : up, v.wbase, up, have);
    }
    {
      uint4* z = reinterpret_cast<uint4*>(cols);
      for (int k = tid; k < kNch * Lay::ROWS * 8; k += B) z[k] = make_uint4(0u, 0u, 0u, 0u);
    }
    __syncthreads();
    const unsigned a_cols = gv_shared_address(cols + lane);
#pragma unroll
    for (int c = 0; c < kNch; ++c) mE[c] = GV_EMPTY;
#pragma unroll 1
    for (int k = 0; k < nk; ++k) {
      const int slot = k * B + tid;
      [[maybe_unused]] const int je = F64 ? 0 : (int)evs[(F64 ? 0 : kNch) * T + slot];
#pragma unroll
      for (int c = 0; c < kNch; ++c) {
        GvSig<W> s;
        bool any;
        if constexpr (!F64) {
          const unsigned u = evs[c * T + slot];
          if (je < kOdd / 2) {
            const int ef = (int)((u >> 23) & 0xFFu);
            any = ef != 0;
            s.m = (u & 0x7FFFFFu) | 0x800000u;
            s.e2 = ef + je - 150;
            s.neg = (u >> 31) != 0u;
          } else {
            any = gv_sig(u, je - kOdd, s) > 0;
          }
        } else {
          s = gv_sig(__longlong_as_double((long long)(
              ((unsigned long long)evs[(2 * c + 1) * T + slot] << 32) | evs[2 * c * T + slot])));
          any = s.m != 0ull;
        }
        const int4 win = s_win[c];
        const int h = s.e2 + GvSig<W>::H, limb = gv_limb_index(h);
        if (any && limb < win.z) {
          const int pos = limb - win.x;
          if (pos >= 0) {
            unsigned l[4];
            const int rem = h + GV_SQ_OFF - 11 * limb;
            gv_square_digits(s, rem, l);
            gv_lane_add_square(s, rem, l, a_cols + (c * Lay::ROWS + pos) * 128);
            gv_lane_add_w(s, a_cols + (c * Lay::ROWS + Lay::SQ) * 128, win.y);
          } else {
            mE[c] = max(mE[c], s.e2);
          }
        }
      }
    }
    bool left = false;
#pragma unroll
    for (int c = 0; c < kNch; ++c) left = left || mE[c] != GV_EMPTY;
    const bool more = __syncthreads_or((int)left) != 0;
    for (int j = wid; j < kNsum; j += NW) {
      const int c = j >> 1, E = s_E[c];
      const int4 win = s_win[c];
      if (!win.w) continue;
      const unsigned* col = cols + c * Lay::ROWS * 32;
      const u128 t =
          (j & 1) ? gv_lane_total<false>(col, Lay::SQ, 22 * (win.x - GvSig<W>::LOW) -
                                                           2 * GV_SQ_OFF - 2 * E + GV_FB)
                  : gv_lane_total<true>(col + Lay::SQ * 32, gv_lane_rows(F64),
                                        22 * win.y - GV_SQ_OFF - E + GV_FB);
      if (lane == 0) s_sum[j] = add128(s_sum[j], t);
    }
    if (!more) break;
    first = false;
    __syncthreads();  // the windows and the columns, read above
  }
  __syncthreads();
  if (tid < kNsum) {
    const u128 t = s_sum[tid];
    ulonglong2* out = a.part + (a.slot_major ? (size_t)tid * a.n_tiles + tile : (size_t)tile * a.nacc + tid);
    *out = make_ulonglong2(t.lo, t.hi);
    if ((tid & 1) == 0) a.tileE[tile * kNch + tid / 2] = s_E[tid / 2];
  }
  if (nbad) atomicAdd(&a.st->nonfinite_iter, (unsigned long long)nbad);
}

template <typename Real, int EPT, int MAXD>
static cudaError_t gv_launch_adj_t(const GvFillArgs& a, int n_tiles, size_t smem, cudaStream_t s,
                                   bool pdl) {
  auto k = gv_fill_adjoint_kernel<Real, EPT, MAXD>;
  const size_t total = AdjSmem<Real>::grid + smem;  // the events and columns, then the grid
  cudaError_t e = gv_prepare(k, total);
  if (e != cudaSuccess) return e;
  return gv_launch(k, dim3(n_tiles), dim3(GV_TILE / EPT), total, s, pdl, a);
}

template <typename Real, int MAXD>
static cudaError_t gv_launch_adj_ept(int ept, const GvFillArgs& a, int n_tiles, size_t smem,
                                     cudaStream_t s, bool pdl) {
  switch (ept) {
    case 1: return gv_launch_adj_t<Real, 1, MAXD>(a, n_tiles, smem, s, pdl);
    case 2: return gv_launch_adj_t<Real, 2, MAXD>(a, n_tiles, smem, s, pdl);
    case 4: return gv_launch_adj_t<Real, 4, MAXD>(a, n_tiles, smem, s, pdl);
  }
  return cudaErrorInvalidValue;
}

namespace gv {
cudaError_t launch_fill_adjoint(int form, int ept, const GvFillArgs& a, int n_tiles, size_t smem,
                                cudaStream_t s, bool pdl) {
  if (a.ndim <= 4)
    return form == GV_FORM_F32   ? gv_launch_adj_ept<float, 4>(ept, a, n_tiles, smem, s, pdl)
           : form == GV_FORM_X64 ? gv_launch_adj_ept<GvX, 4>(ept, a, n_tiles, smem, s, pdl)
                                 : gv_launch_adj_ept<double, 4>(ept, a, n_tiles, smem, s, pdl);
  if (a.ndim <= 16)
    return form == GV_FORM_F32   ? gv_launch_adj_ept<float, 16>(ept, a, n_tiles, smem, s, pdl)
           : form == GV_FORM_X64 ? gv_launch_adj_ept<GvX, 16>(ept, a, n_tiles, smem, s, pdl)
                                 : gv_launch_adj_ept<double, 16>(ept, a, n_tiles, smem, s, pdl);
  return cudaErrorInvalidValue;
}
}  // namespace gv
