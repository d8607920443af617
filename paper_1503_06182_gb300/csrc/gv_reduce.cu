// gv_reduce.cu -- combination of all events of an iteration and the grid
// optimisation (Section 2.1: the grid optimisation is serial so that it can
// use the results of all events).
//
// Forward stages and small adjoint ones: gv_reduce_cluster_kernel and
// gv_reduce_slots_kernel (below).  gv_reduce_kernel and the batched form: the
// grid is (slot blocks of 32) x (tile ranges): each CTA owns 32 slots and a
// range of tiles; its 8 warps stride over the tiles, the warps' sums are combined
// in shared memory and published.  All of them form a slot's sum by the rule of
// gv_slotsum.cuh (channel sums: at the tiles' scales; bin sums: at the bins' own
// positions, gv_limbs.cuh).  No sum is formed with atomics, and none depends on
// the order of its tiles: the totals are the same in every kernel, launch shape
// and batch.
//
// Tickets instead of waiting: each CTA publishes its sums and counts itself
// on its block of 32 slots; the CTA that completes a block combines the
// block's sums, rounds them once to FP64 and counts the block on each axis
// its bins belong to.  The CTA whose count completes an axis refines that
// axis at once (Lepage's VEGAS, cited in Section 2.1: smoothing,
// normalisation, compression ((1-rho)/(-ln rho))^alpha, redistribution into
// N equal shares), so the axes are refined in parallel by different CTAs
// while others still reduce; the CTA that completes block 0 (the channel
// sums) records I_k and sigma_k and combines the stage.  No CTA ever waits
// for another.
//
// On this chip a dependent FP64 operation waits ~56-64 cycles, a warp-wide
// FP64 instruction occupies the SM's FP64 pipe for ~19 cycles, and the FP64
// library log takes ~2000 cycles: the serial code here keeps its FP64 chains
// short (reciprocals passed in, a table-driven log, one thread per bin).
#include <algorithm>

#include "gv_combine.cuh"
#include "gv_ff.cuh"
#include "gv_integrands.cuh"
#include "gv_limbs.cuh"
#include "gv_slotsum.cuh"
#include "gv_xint.cuh"

// A value rounded to nearest-even, assembled with integer operations only, from
// its magnitude's leading 64 bits (bit 63 set, worth 2^(e - 63)) and whether
// anything lies below them.
__device__ __forceinline__ double assemble_double(unsigned long long window, bool sticky, int e,
                                                  bool neg) {
  // round the 64-bit window to 53 bits (nearest, ties to even)
  unsigned long long mant = window >> 11;
  const unsigned long long rest = window & 0x7FFull;
  const bool half = (rest & 0x400ull) != 0ull;
  const bool above = (rest & 0x3FFull) != 0ull || sticky;
  if (half && (above || (mant & 1ull))) ++mant;
  if (mant >> 53) {
    mant >>= 1;
    ++e;
  }
  double r;
  if (e > 1023) {
    r = __longlong_as_double(0x7FF0000000000000ll);  // beyond FP64, as a sum of doubles would be
  } else if (e >= -1022) {
    r = __longlong_as_double((long long)(((unsigned long long)(e + 1023) << 52) |
                                         (mant & 0xFFFFFFFFFFFFFull)));
  } else if (e >= -1022 - 600) {
    // below the normal range: scale into it, then one multiply by 2^-600
    // (the product rounds to the subnormal grid; rare, and on the FP64 pipe)
    r = __longlong_as_double((long long)(((unsigned long long)(e + 600 + 1023) << 52) |
                                         (mant & 0xFFFFFFFFFFFFFull))) *
        0x1p-600;
  } else {
    r = 0.0;
  }
  return neg ? -r : r;
}
__device__ __forceinline__ double acc_to_double(const GvAcc& a) {
  unsigned long long window;
  bool sticky, neg;
  int e;
  return acc_window(a, &window, &sticky, &e, &neg) ? assemble_double(window, sticky, e, neg) : 0.0;
}

// Barrier of a group of nthr threads (a multiple of 32); id 0 is the whole CTA.
__device__ __forceinline__ void gv_bar(int id, int nthr) {
  asm volatile("bar.sync %0, %1;" ::"r"(id), "r"(nthr) : "memory");
}

// The iteration's finalisation, by one warp of a group (tid: the thread's index in
// the group): the iteration record, the stage's combination and the per-iteration
// state.
__device__ void finalize_iteration(const GvReduceArgs& a, int tid) {
  const int lane = tid & 31, wid = tid >> 5;
  GvState* st = a.st;
  // the sums, each rounded once to FP64 by the CTA that completed its block
  if (wid == 0) {
    // warp 0: the iteration record (one lane per channel) and the stage
    const int stride = a.mode ? 2 + 2 * GV_NGRAD : 2;
    if (lane < a.nch) {
      double* rec = a.per_iter + (size_t)a.k * stride + 2 * lane;
      double I, s;
      mean_sigma(__ldcg(a.sums + 2 * lane), __ldcg(a.sums + 2 * lane + 1), a.inv_c, a.inv_cm1,
                 &I, &s);
      rec[0] = I;
      if (!a.plus) rec[1] = s;  // VEGAS+: sigma_k comes from the hypercube statistics
      if (a.host_rec) {
        a.host_rec[(size_t)a.k * stride + 2 * lane] = I;
        a.host_rec[(size_t)a.k * stride + 2 * lane + 1] = s;
      }
    }
    __syncwarp();
    if (a.last && !a.plus) combine_stage_warp(a.per_iter, stride, a.k + 1, a.inv_m1, st, a.mode != 0);
    if (a.last && a.plus) {
      // the hypercube statistics run beside this kernel: the second of the
      // two to finish the stage's last iteration combines it
      int t = 0;
      if (lane == 0) {
        __threadfence();  // this iteration's I_k before the arrival
        t = atomicAdd(&st->join, 1);
      }
      t = __shfl_sync(0xffffffffu, t, 0);
      if (t == 1) {
        __threadfence();  // the statistics' sigma_k, published before their arrival
        combine_stage_warp(a.per_iter, stride, a.k + 1, a.inv_m1, st, false);
        if (lane == 0) st->join = 0;
      }
    }
    if (lane == 0) {
      const unsigned long long nf = __ldcg(&st->nonfinite_iter);
      st->nonfinite = (a.k == 0 ? 0ull : st->nonfinite) + nf;
      if (a.k == 0) st->status = 0;
      st->nonfinite_iter = 0ull;
    }
  }
  if (tid == 0) {
    st->it = st->it + 1ull;
    if (a.last) st->it0 = st->it;  // the next stage's first counter
    if (a.last && a.host_it) *a.host_it = st->it;
    if (a.last && a.host_st) {
      // the state the host reads after the stage: this thread wrote all of it
      a.host_st->it = st->it;
      a.host_st->nonfinite = st->nonfinite;
      a.host_st->status = st->status;
      a.host_st->integral = st->integral;
      a.host_st->error = st->error;
      a.host_st->chi2 = st->chi2;
    }
  }
}

// ---------------------------------------------------------------------------
// Grid refinement (Lepage's VEGAS, cited in Section 2.1), one axis at a time:
// every step of it -- smoothing, normalisation, compression, redistribution
// -- involves one axis only, so the CTA whose reduction completes an axis
// refines it at once, while other CTAs are still reducing.
// ---------------------------------------------------------------------------
// Write the edges e_src (N+1 values) of axis ax into the grid pack with the
// axis' derived tables.
// (and the edges to mapped host memory, if given).
__device__ __forceinline__ void pack_axis_tables(double* grid, const double* e_src, int ax, int d, int N, int tid,
                                 int nthr, double* host = nullptr) {
  const GvGridLayout L{d, N};
  double* e64 = grid + L.off_e64() + (size_t)ax * (N + 1);
  double* wd64 = grid + L.off_wd64() + (size_t)ax * N;
  double* jac = grid + L.off_jac() + (size_t)ax * N;
  GvBin32* b32 = reinterpret_cast<GvBin32*>(grid + L.off_bin32()) + (size_t)ax * N;
  for (int i = tid; i <= N; i += nthr) {
    const double e = e_src[i];
    e64[i] = e;
    if (host) host[(size_t)ax * (N + 1) + i] = e;
    if (i < N) {
      const double w = e_src[i + 1] - e;
      const double j = (double)N * w;
      wd64[i] = w;
      jac[i] = j;
      // j = m 2^x with m in [1,2): exponent from the bits (j > 0; a subnormal
      // j is scaled into the normal range first)
      const bool sub = j < 0x1p-1000;
      const double js = sub ? j * 0x1p200 : j;
      const long long b = __double_as_longlong(js);
      const int x = (int)((b >> 52) & 0x7FF) - 1023;
      const double m = __longlong_as_double((b & 0xFFFFFFFFFFFFFll) | 0x3FF0000000000000ll);
      b32[i] = GvBin32{(float)e, (float)w, (float)m, sub ? x - 200 : x};
    }
  }
}

// 1/x and 1/sqrt(x) for positive normal x: the hardware approximations
// (PTX rcp.approx.ftz.f64 and rsqrt.approx.ftz.f64, about 20 correct bits)
// refined by two Newton-Raphson steps, y <- y + y (1 - x y) and
// z <- z + z (1 - x z^2) / 2, each of which squares the relative error.
// Measured against the correctly rounded results over six decades: the
// reciprocal agrees bit for bit, the square root within 2.7e-16.  They
// replace the library's correctly rounded routines, whose special-case
// handling costs this chip's scarce FP64 pipe more instructions.
__device__ __forceinline__ double gv_rcp_nr(double x) {
  double y;
  asm("rcp.approx.ftz.f64 %0, %1;" : "=d"(y) : "d"(x));
  double e = fma(-x, y, 1.0);
  y = fma(y, e, y);
  e = fma(-x, y, 1.0);
  return fma(y, e, y);
}
__device__ __forceinline__ double gv_rsqrt_nr(double x) {
  double z;
  asm("rsqrt.approx.ftz.f64 %0, %1;" : "=d"(z) : "d"(x));
#pragma unroll
  for (int s = 0; s < 2; ++s) {
    const double h = x * z;
    const double e = fma(-h, z, 1.0);
    z = fma(0.5 * z, e, z);
  }
  return z;
}
struct GvRefineMem {
  double *r, *slope;    // [N] 6 x smoothed sums, then compressed values; bin sums, then slopes
  double *C, *e, *ne;   // [N + 1] prefix sums, old and new edges
};
__device__ __forceinline__ GvRefineMem refine_mem(double* sm, int N) {
  GvRefineMem m;
  m.r = sm;
  m.slope = m.r + N;
  m.C = m.slope + N;
  m.e = m.C + (N + 1);
  m.ne = m.e + (N + 1);
  return m;
}

// ((1 - rho)/(-ln rho))^alpha for 0 < rho < 1, with the common exponents
// evaluated by reciprocals and roots rather than pow.  In the refinement
// rho <= 3/5 (a smoothed bin holds at most 3/5 of the smoothed total), so
// 1 - rho >= 2/5 and -ln rho >= 0.51: both are positive normal numbers.
// Out of line: the usual alpha takes compress15_ff, and the code it walks past is
// fetched cold in every reduce (ten axes, 4 x 1000 + 10 x 1e4 events: 241 us
// inlined, 238 so).
__device__ __noinline__ double compress(double rho, double alpha) {
  if (rho <= 0.0) return 0.0;
  if (rho >= 1.0) return 1.0;
  const double L = -gv_log_pos(rho);
  const double om = 1.0 - rho;
  if (alpha == 1.5) {  // om^(3/2) L^(-3/2) = (om^2 / sqrt(om)) (1/sqrt(L))^3
    const double y = gv_rsqrt_nr(L), z = gv_rsqrt_nr(om);
    return (om * om * z) * (y * y * y);
  }
  if (alpha == 1.0) return om * gv_rcp_nr(L);
  if (alpha == 0.5) return om * gv_rsqrt_nr(om) * gv_rsqrt_nr(L);
  if (alpha == 2.0) {
    const double q = om * gv_rcp_nr(L);
    return q * q;
  }
  if (alpha == 0.0) return 1.0;
  return pow(om * __drcp_rn(L), alpha);
}

// The compressed value r = ((1 - rho)/(-ln rho))^(3/2) (alpha = 3/2) and the
// slope de / r in FP32 pairs (gv_ff.cuh), for 2^-100 < rho <= 3/5 and
// 2^-100 < de <= 1.  -ln rho by the table reduction of gv_log_pos: rho =
// 2^k m, r' = m R_j - 1 (|r'| < 2^-7), ln rho = k ln2 + L_j + ln(1 + r'),
// with ln(1 + r') = r' + r'^2 P(r'), P = -1/2 + r'/3 - r'^2/4 + ... + r'^5/7
// (truncation below 2^-60); the leading -1/2 and r' P's product are paired,
// the rest of P (scaled by r'^3 < 2^-21) is FP32.
__device__ __forceinline__ void compress15_ff(double rho, double de, double& rv, double& sl) {
  const long long b = __double_as_longlong(rho);
  const int k = (int)(b >> 52) - 1023;
  const int j = (int)((b >> 45) & 127);
  const GvFF m = gv_ff_from_double(
      __longlong_as_double((b & 0xFFFFFFFFFFFFFll) | 0x3FF0000000000000ll));
  const double2 RL = __ldg(reinterpret_cast<const double2*>(gv_log_tab) + j);
  const GvFF p = gv_ff_mul(m, gv_ff_from_double(RL.x));
  const GvFF r = gv_two_sum(__fsub_rn(p.hi, 1.0f), p.lo);  // p.hi - 1 is exact
  const float x = r.hi;
  float Q = __fmaf_rn(x, 1.0f / 7.0f, -1.0f / 6.0f);
  Q = __fmaf_rn(Q, x, 0.2f);
  Q = __fmaf_rn(Q, x, -0.25f);
  Q = __fmaf_rn(Q, x, 1.0f / 3.0f);
  const GvFF P = gv_two_sum(-0.5f, __fmul_rn(x, Q));
  const GvFF l1p = gv_ff_add(r, gv_ff_mul(gv_ff_mul(r, r), P));
  // ln 2 = 0x1.62e43p-1 + (-0x1.05c61p-29), to 9e-17
  const GvFF kln2 = gv_ff_mul_f(GvFF{0x1.62e43p-1f, -0x1.05c61p-29f}, (float)k);
  const GvFF lnrho = gv_ff_add(gv_ff_add(kln2, gv_ff_from_double(RL.y)), l1p);
  const GvFF L = {-lnrho.hi, -lnrho.lo};
  const GvFF R = gv_ff_from_double(rho);
  const GvFF om = gv_ff_add(GvFF{1.0f, 0.0f}, GvFF{-R.hi, -R.lo});
  const GvFF q = gv_ff_div(om, L);
  const GvFF c = gv_ff_mul(q, gv_ff_sqrt(q));
  rv = gv_ff_to_double(c);
  sl = gv_ff_to_double(gv_ff_div(gv_ff_from_double(de), c));
}

// alpha values whose compressed values are at least (1/745)^2 > 1e-6 (the
// reciprocal approximation then sees normal numbers only)
__device__ __forceinline__ bool fast_alpha(double alpha) {
  return alpha == 1.5 || alpha == 1.0 || alpha == 0.5 || alpha == 2.0 || alpha == 0.0;
}

// Shared memory of refine_axis: r[N], slope[N], C[N+1], e[N+1], ne[N+1].
__host__ __device__ inline size_t refine_axis_smem(int N) {
  return sizeof(double) * (2 * (size_t)N + 3 * ((size_t)N + 1));
}

// Refinement of axis ax by a group of nthr threads (local index tid, barrier
// id bar, group number q), once every block holding the axis has rounded its
// bin sums d_i to FP64 (the oracle's arithmetic from here on):
//   1. 6 x the smoothed sums, s_i = 3 (d_0 + d_1) at the ends and
//      2 (d_{i-1} + d_i + d_{i+1}) inside, and their total (a fixed-order
//      tree), then per bin the share rho = s_i / total, the compressed value
//      r = ((1-rho)/(-ln rho))^alpha and the slope (e_{i+1}-e_i)/r;
//   2. one warp: the prefix sums C of r;
//   3. per new edge: the old bin where C reaches j R/N -- binary search on
//      the bit patterns of the nonnegative doubles -- then
//      e_i + (target - C_i) * slope_i; e'_0 = 0 and e'_N = 1 exactly;
//   4. the axis' tables.
// An axis whose bins are all zero keeps its edges.
// The same steps in 64-bit integer significands are 5 to 15 us faster over the
// 9 to 14 iterations of the small stages, but their edges differ in the last
// places, and an FP32 table entry that rounds the other way moves events across
// an integrand's cuts: a batch with three-jet members then leaves 1e-9 in one
// run of four.
// A cluster's sums are in shared memory already (LOADED: d in slope, the edges
// in e, and a barrier passed).
template <bool LOADED>
__device__ __forceinline__ void refine_axis(const GvReduceArgs& a, int ax, double* sm, int tid, int nthr, int bar,
                            int q) {
  const int N = a.nbins, lane = tid & 31, wid = tid >> 5;
  __shared__ double s_inv[8], s_step[8];
  const GvRefineMem m = refine_mem(sm, N);
  double *r = m.r, *slope = m.slope, *C = m.C, *e = m.e, *ne = m.ne;
  if (!LOADED) {
    const double* d = a.sums + 2 * a.nch + ax * N;
    const double* e64 = a.grid + GvGridLayout{a.ndim, N}.off_e64() + (size_t)ax * (N + 1);
    for (int k = tid; k <= N; k += nthr) e[k] = e64[k];
    for (int i = tid; i < N; i += nthr) slope[i] = __ldcg(d + i);
    gv_bar(bar, nthr);
  }
  for (int i = tid; i < N; i += nthr) {  // (the ends add a zero: no second path for their lanes)
    const bool end = i == 0 || i == N - 1;
    const int k = max(i, 1);
    r[i] = (end ? 3.0 : 2.0) * (slope[k - 1] + slope[k] + (end ? 0.0 : slope[min(i + 1, N - 1)]));
  }
  gv_bar(bar, nthr);
  if (wid == 0) {
    // the total in an order fixed by N alone (whatever the group's size):
    // 32 consecutive chunks in order, then a fixed pairwise tree
    const int chunk = (N + 31) / 32;
    const int i0 = min(N, lane * chunk), i1 = min(N, i0 + chunk);
    double part = 0.0;
    if (chunk <= 4) {
      // a fixed pairwise tree over the chunk (zeros past its end add exactly)
      double v[4];
#pragma unroll
      for (int k = 0; k < 4; ++k) v[k] = i0 + k < i1 ? r[i0 + k] : 0.0;
      part = (v[0] + v[1]) + (v[2] + v[3]);
    } else {
      for (int i = i0; i < i1; ++i) part += r[i];
    }
#pragma unroll
    for (int m = 16; m > 0; m >>= 1) part += __shfl_down_sync(0xffffffffu, part, m);
    if (lane == 0) {
      const double t = part;
      s_inv[q] = !(t > 0.0) ? 0.0 : (t > 0x1p-1000 && t < 0x1p1000) ? gv_rcp_nr(t) : __drcp_rn(t);
    }
  }
  gv_bar(bar, nthr);
  const double inv = s_inv[q];
  const bool fast = fast_alpha(a.alpha);
  if (inv > 0.0) {
    for (int i = tid; i < N; i += nthr) {
      double rv = 0.0, sl = 0.0;
      const double s6 = r[i];
      if (s6 > 0.0) {
        const double rho = s6 * inv, de = e[i + 1] - e[i];
        if (a.alpha == 1.5 && rho > 0x1p-100 && rho <= 0.6 && de > 0x1p-100 && de <= 1.0) {
          compress15_ff(rho, de, rv, sl);
        } else {
          rv = compress(rho, a.alpha);
          if (rv > 0.0) sl = de * (fast ? gv_rcp_nr(rv) : __drcp_rn(rv));
        }
      }
      r[i] = rv;
      slope[i] = sl;
    }
    gv_bar(bar, nthr);
    if (wid == 0) {
      const int chunk = (N + 31) / 32;
      const int i0 = min(N, lane * chunk), i1 = min(N, i0 + chunk);
      // the chunk's own running sums (in order), formed before the scan so
      // that each C below is one addition away from its chunk's base
      double lp[4];
      double local = 0.0;
      if (chunk <= 4) {
#pragma unroll
        for (int k = 0; k < 4; ++k) {
          local = i0 + k < i1 ? local + r[i0 + k] : local;
          lp[k] = local;
        }
      } else {
        for (int i = i0; i < i1; ++i) local += r[i];
      }
      // inclusive prefix sums of the 32 chunk sums (Hillis-Steele; the lanes
      // below the distance add a zero), then each chunk's exclusive prefix
#pragma unroll
      for (int m = 1; m < 32; m <<= 1) {
        const double v = __shfl_up_sync(0xffffffffu, local, m);
        local += lane >= m ? v : 0.0;
      }
      double run = __shfl_up_sync(0xffffffffu, local, 1);  // of this lane's chunk
      if (lane == 0) run = 0.0;
      if (lane == 0) C[0] = 0.0;
      if (chunk <= 4) {
#pragma unroll
        for (int k = 0; k < 4; ++k)
          if (i0 + k < i1) C[i0 + k + 1] = run + lp[k];
      } else {
        for (int i = i0; i < i1; ++i) {
          run += r[i];
          C[i + 1] = run;
        }
      }
      __syncwarp();
      if (lane == 0) s_step[q] = C[N] * a.inv_nbins;
    }
    gv_bar(bar, nthr);
    const double step = s_step[q];
    const long long* Cb = reinterpret_cast<const long long*>(C);
    for (int j = tid; j <= N; j += nthr) {
      double v;
      if (j == 0) {
        v = 0.0;
      } else if (j == N) {
        v = 1.0;
      } else {
        const double target = step * j;
        const long long tb = __double_as_longlong(target);
        int lo = 0, hi = N - 1;  // first bin i with C[i+1] > target (N-1 if none)
        while (lo < hi) {
          const int mid = (lo + hi) >> 1;
          if (Cb[mid + 1] > tb)
            hi = mid;
          else
            lo = mid + 1;
        }
        v = fma(target - C[lo], slope[lo], e[lo]);
      }
      ne[j] = v;
    }
  } else {
    for (int j = tid; j <= N; j += nthr) ne[j] = e[j];
  }
  gv_bar(bar, nthr);
  pack_axis_tables(a.grid, ne, ax, a.ndim, N, tid, nthr, a.last ? a.host_grid : nullptr);
}

// Axes that one block of 32 slots can touch, and the dynamic shared memory
// the reduce kernels need to refine that many axes side by side.
__host__ __device__ inline int gv_axes_per_block(int N) {
  const int k = (31 + N - 1) / N + 1;
  return k < 7 ? k : 7;
}

#define GV_RED_TILES_PER_LOAD 8

// One slot's tile partials.  Channel slots: 128-bit two's complement at
// 2^(pw e - GV_FB), e the tile's scale, pw = 1 (sums of v) or 2 (of v^2); bin slots
// (axis bins and histogram bins): 112 bits and their position (GvPartial).
struct SlotPartials {
  const ulonglong2* src;
  size_t stride;
  const int* tileE;
  int nch, pw;
  bool bin;
  __device__ __forceinline__ SlotPartials(const GvReduceArgs& a, int k, size_t first, size_t stride_)
      : src(a.part + first),
        stride(stride_),
        tileE(a.tileE + (k >> 1)),
        nch(a.nch),
        pw((k & 1) + 1),
        bin(a.has_bins && k >= 2 * a.nch) {}
  __device__ __forceinline__ ulonglong2 load(int t) const { return __ldcg(src + t * stride); }
  // bit position of a partial v of tile t (0: none), and its top word
  __device__ __forceinline__ int position(const ulonglong2& v, int t) const {
    if (bin) return (int)(v.y >> 48);
    const int e = __ldcg(tileE + (size_t)t * nch);
    return e == GV_EMPTY ? 0 : pw * e - GV_FB + GV_POS_OFF;
  }
  __device__ __forceinline__ unsigned word3(const ulonglong2& v) const {
    const unsigned h = (unsigned)(v.y >> 32);
    return bin ? (unsigned)(int)(short)h : h;
  }
};
// The partials t0 + g step below nt, g < G, and their positions (0: none): every
// load before the first use, and no branch among them (a load under a condition
// that also uses it waits for it: 8 round trips through L2 instead of one).
// Returns the highest position.  (nt = 0 reads the first tile and takes nothing.)
template <int G>
__device__ __forceinline__ int load_tiles(const SlotPartials& s, int t0, int step, int nt,
                                          ulonglong2 (&v)[G], int (&pos)[G]) {
  const int end = max(nt, 1) - 1;
  int top = 0;
#pragma unroll
  for (int g = 0; g < G; ++g) v[g] = s.load(min(t0 + g * step, end));
  if (s.bin) {
#pragma unroll
    for (int g = 0; g < G; ++g) pos[g] = s.position(v[g], 0);
  } else {
#pragma unroll
    for (int g = 0; g < G; ++g) pos[g] = s.position(v[g], min(t0 + g * step, end));
  }
#pragma unroll
  for (int g = 0; g < G; ++g) {
    if (t0 + g * step >= nt) pos[g] = 0;
    top = max(top, pos[g]);
  }
  return top;
}

// The sum of the partials t = u, u + step, .. below nt, each read once: the window
// moves up when a higher one comes.  (`lane`: of threads with consecutive u, 0
// otherwise.)
template <int G>
__device__ __forceinline__ GvAcc sum_tiles(const SlotPartials& p, int u, int lane, int step,
                                           int nt) {
  GvAcc s = acc_zero();
  for (int t0 = u; t0 < nt; t0 += G * step) {
    ulonglong2 v[G];
    int pos[G];
    const int top = load_tiles(p, t0, step, nt, v, pos);
    if ((top >> 5) > s.g) acc_raise(s, top >> 5);
    unsigned far = 0u;
#pragma unroll
    for (int g = 0; g < G; ++g) {
      if (g > 0 && t0 - lane + g * step >= nt) break;  // no lane has another
      const int o = s.g - (pos[g] >> 5);
      const bool near = pos[g] != 0 && o <= 1;
      if (pos[g] != 0 && o > 1) far |= 1u << g;
      acc_add_near(s, near ? (unsigned)v[g].x : 0u, near ? (unsigned)(v[g].x >> 32) : 0u,
                   near ? (unsigned)v[g].y : 0u, near ? p.word3(v[g]) : 0u, pos[g], o);
    }
    // read again: few, and their code stays out of the loop above
    while (far) {
      const int t = t0 + (__ffs((int)far) - 1) * step;
      far &= far - 1u;
      const ulonglong2 x = p.load(t);
      const int q = p.position(x, t);
      acc_add_far(s, (unsigned)x.x, (unsigned)(x.x >> 32), (unsigned)x.y, p.word3(x), q,
                  s.g - (q >> 5));
    }
  }
  return s;
}

// The sum over a warp of at most 32 G partials, one slot: the highest position
// first.  In every lane.
template <int G>
__device__ __forceinline__ double warp_sum_tiles(const SlotPartials& p, int nt) {
  constexpr unsigned all = 0xffffffffu, M = (1u << 26) - 1u;
  const int lane = threadIdx.x & 31;
  ulonglong2 v[G];
  int pos[G];
  const int g0 = __reduce_max_sync(all, load_tiles(p, lane, 32, nt, v, pos)) >> 5;
  if (g0 == 0) return 0.0;
  GvAccFixed a = {{0u, 0u, 0u, 0u, 0u, 0u}};
#pragma unroll
  for (int g = 0; g < G; ++g) {
    if (32 * g >= nt) break;
    const bool any = pos[g] != 0;
    acc_add_fixed(a, any ? (unsigned)v[g].x : 0u, any ? (unsigned)(v[g].x >> 32) : 0u,
                  any ? (unsigned)v[g].y : 0u, any ? p.word3(v[g]) : 0u, any ? pos[g] : 32 * g0, g0);
  }
  // in eight parts of 26 bits: of the even and the odd ones no two overlap
  unsigned s[8];
#pragma unroll
  for (int i = 0; i < 8; ++i) {
    const int j = 26 * i / 32, r = 26 * i % 32;
    s[i] = __reduce_add_sync(
        all, i == 7 ? a.w[5] >> r : __funnelshift_r(a.w[j], a.w[min(j + 1, 5)], r) & M);
  }
  unsigned long long q[4], h[3];
  q[0] = s[0] | ((unsigned long long)s[2] << 52);
  q[1] = ((unsigned long long)s[2] >> 12) | ((unsigned long long)s[4] << 40);
  q[2] = ((unsigned long long)s[4] >> 24) | ((unsigned long long)s[6] << 28);
  h[0] = ((unsigned long long)s[1] << 26);
  h[1] = ((unsigned long long)s[3] << 14);
  h[2] = ((unsigned long long)s[5] << 2) | ((unsigned long long)s[7] << 54);
  asm("add.cc.u64 %0, %0, %3;\n\t"
      "addc.cc.u64 %1, %1, %4;\n\t"
      "addc.u64 %2, %2, %5;"
      : "+l"(q[0]), "+l"(q[1]), "+l"(q[2])
      : "l"(h[0]), "l"(h[1]), "l"(h[2]));
  q[3] = (unsigned long long)((long long)q[2] >> 63);
  unsigned long long window;
  bool sticky, neg;
  int e;
  return acc_leading(q, g0, &window, &sticky, &e, &neg) ? assemble_double(window, sticky, e, neg)
                                                        : 0.0;
}

// The sum over a warp's lanes, in every lane: counters in a low part
// of 27 bits and the rest, which fits 32 bits for 2^21 partials a lane; more
// (`many`) take three parts.
__device__ __forceinline__ GvAcc warp_sum_acc(GvAcc a, bool many) {
  constexpr unsigned M = (1u << 27) - 1u, all = 0xffffffffu;
  const int g = __reduce_max_sync(all, a.g);
  if (a.g < g) acc_raise(a, g);
#pragma unroll
  for (int j = 0; j < GV_SLOT_WORDS; ++j) {
    const long long v = (long long)a.w[j];
    unsigned long long t = __reduce_add_sync(all, (unsigned)v & M);
    if (!many)
      t += (unsigned long long)(long long)__reduce_add_sync(all, (int)(v >> 27)) << 27;
    else
      t += ((unsigned long long)__reduce_add_sync(all, (unsigned)(v >> 27) & M) << 27) +
           ((unsigned long long)__reduce_add_sync(all, (unsigned)(v >> 54)) << 54);
    a.w[j] = t;
  }
  return a;
}

// One reduce CTA (256 threads) of one integration: slot block bx (32 slots,
// one per lane), tile range by, of nblk CTAs in total for that integration.
//   A. every CTA: each slot's sum over its tiles (no atomics), published;
//   B. the CTA that completes a slot block (ticket): the block's sums over all
//      tile ranges, each rounded once to FP64;
//   C. the CTA whose block completes an axis (second ticket) refines the
//      axis; the CTA that completes block 0 (the channel sums) finalises the
//      iteration.
// The sums depend on the data alone (gv_slotsum.cuh), not on the launch shape or
// on timing.
static_assert(GV_SLOT_BYTES == 8 * (GV_SLOT_WORDS + 1), "a published sum");
struct GvTaskMem {
  unsigned long long w[GV_SLOT_WORDS][8][32];  // the warps' sums: counters ..
  int g[8][32];                                // .. and windows
  int flags[4], won[GV_MAXD];
};
// The sum over the CTA's warps of their lanes' sums: warp j < GV_SLOT_WORDS
// returns counter j, and every warp the window.
__device__ __forceinline__ unsigned long long task_combine(GvTaskMem& m, const GvAcc& a, int* g) {
  const int lane = threadIdx.x & 31, wid = threadIdx.x >> 5;
#pragma unroll
  for (int j = 0; j < GV_SLOT_WORDS; ++j) m.w[j][wid][lane] = a.w[j];
  m.g[wid][lane] = a.g;
  __syncthreads();
  int top = 0;
#pragma unroll
  for (int w = 0; w < 8; ++w) top = max(top, m.g[w][lane]);
  *g = top;
  unsigned long long t = 0ull;
  if (wid < GV_SLOT_WORDS) {
#pragma unroll
    for (int w = 0; w < 8; ++w) t += acc_word(&m.w[0][w][lane], 8 * 32, m.g[w][lane], top, wid);
  }
  return t;
}
__device__ __forceinline__ void gv_reduce_task(const GvReduceArgs& a, int bx, int by, int nblk,
                                               GvTaskMem& mem, double* sm) {
  const int lane = threadIdx.x & 31, wid = threadIdx.x >> 5;
  const int k = bx * 32 + lane;
  const int gx = (a.nacc + 31) / 32, gy = nblk / gx;
  const int t0 = by * a.tiles_per_cta;
  const int t1 = min(a.n_tiles, t0 + a.tiles_per_cta);
  const size_t row = 32 * (size_t)gx;  // of the published sums: [range][counters, window][row]
  gv_wait_prior_grid();

  // ---- A: this CTA's tiles
  GvAcc sum = acc_zero();
  if (k < a.nacc)
    sum = sum_tiles<GV_RED_TILES_PER_LOAD / 2>(SlotPartials(a, k, k, a.nacc), t0 + wid, 0, 8, t1);
  int g;
  unsigned long long t = task_combine(mem, sum, &g);
  if (wid <= GV_SLOT_WORDS) {
    a.cpart[(size_t)(by * (GV_SLOT_WORDS + 1) + wid) * row + k] =
        wid < GV_SLOT_WORDS ? t : (unsigned long long)g;
    __threadfence();
  }
  __syncthreads();
  if (threadIdx.x == 0)
    mem.flags[0] = atomicAdd(a.tickets + gv_ticket_group(bx), 1) == gy - 1 ? 1 : 0;
  __syncthreads();
  if (!mem.flags[0]) return;

  // ---- B: this CTA completes slot block bx
  __threadfence();  // the other CTAs' sums, published before their tickets
  gv_allow_next_grid();  // what is left is short: the next fill's CTAs may come in
  if (threadIdx.x == 0) a.tickets[gv_ticket_group(bx)] = 0;
  sum = acc_zero();
#pragma unroll 1
  for (int y = wid; y < gy; y += 8) {
    const unsigned long long* c = a.cpart + (size_t)y * (GV_SLOT_WORDS + 1) * row + k;
    GvAcc r;
#pragma unroll
    for (int j = 0; j < GV_SLOT_WORDS; ++j) r.w[j] = __ldcg(c + j * row);
    r.g = (int)__ldcg(c + GV_SLOT_WORDS * row);
    const int top = max(r.g, sum.g);
    acc_raise(r, top);
    acc_raise(sum, top);
#pragma unroll
    for (int j = 0; j < GV_SLOT_WORDS; ++j) sum.w[j] += r.w[j];
  }
  t = task_combine(mem, sum, &g);
  __syncthreads();  // (a counter may be read at another's place)
  if (wid < GV_SLOT_WORDS) mem.w[wid][0][lane] = t;
  __syncthreads();
  const int N = a.nbins;
  // the axis bins of this block (the histogram slots after them have no axis)
  const int j_first = max(0, bx * 32 - 2 * a.nch);
  const int j_last = min(min(a.nacc - 1, bx * 32 + 31) - 2 * a.nch, a.ndim * N - 1);
  if (wid == 0) {
    // the slot's sum over all events, rounded once to FP64
#pragma unroll
    for (int j = 0; j < GV_SLOT_WORDS; ++j) sum.w[j] = mem.w[j][0][lane];
    sum.g = g;
    if (k < a.nacc) a.sums[k] = acc_to_double(sum);
    __threadfence();
    // second tickets, one lane per axis the block touches: the block whose
    // count completes an axis refines it
    const int ax0 = j_first / N;
    const int nax =
        (a.has_bins && a.refine_follows && j_last >= j_first) ? j_last / N - ax0 + 1 : 0;
    bool won = false;
    if (lane < nax) {
      const int ax = ax0 + lane;
      const int x_lo = (2 * a.nch + ax * N) / 32, x_hi = (2 * a.nch + (ax + 1) * N - 1) / 32;
      int* tk = a.tickets + gv_ticket_axis(a.nacc, ax);
      if (atomicAdd(tk, 1) == x_hi - x_lo) {
        *tk = 0;
        won = true;
      }
    }
    const unsigned mask = __ballot_sync(0xffffffffu, won);
    if (won) mem.won[__popc(mask & ((1u << lane) - 1u))] = ax0 + lane;
    if (lane == 0) mem.flags[1] = __popc(mask);
  }
  __syncthreads();
  // block 0 holds the channel sums: it finalises the iteration
  const int n_won = mem.flags[1], fin = bx == 0;
  if (n_won == 0 && !fin) return;

  // ---- C
  if (n_won) __threadfence();  // the other blocks' sums, published before their tickets
  // the won axes and the finalisation side by side on groups of warps: the
  // finalisation takes warp 7, the axes the other warps, min(n_won, 7) groups,
  // each with its own barrier and shared memory
  if (fin && wid == 7) {
    finalize_iteration(a, threadIdx.x - 32 * 7);
  } else if (n_won > 0) {
    const int ng = min(n_won, 7), wpg = (fin ? 7 : 8) / ng, q = wid / wpg;
    if (q < ng) {
      const int per = (int)(refine_axis_smem(a.nbins) / sizeof(double));
      for (int it = q; it < n_won; it += ng)
        refine_axis<false>(a, mem.won[it], sm + (size_t)q * per, threadIdx.x - 32 * wpg * q, 32 * wpg,
                    2 + q, q);
    }
  }
}

__global__ void __launch_bounds__(256) gv_reduce_kernel(const GvReduceArgs a) {
  extern __shared__ __align__(16) double sm[];
  __shared__ GvTaskMem mem;
  gv_reduce_task(a, blockIdx.x, blockIdx.y, gridDim.x * gridDim.y, mem, sm);
}

// ---------------------------------------------------------------------------
// Single-level reduce of an iteration with slot-major partials (slot k of tile
// t at part[k n_tiles + t]): a CTA owns one slot and reads it over every tile;
// the sum is rounded once to FP64.  Compared with the two-level reduce there is no published
// per-range sum and no ticket between the levels: one L2 round trip for the
// partials, then one fence and one ticket per slot.
// Tickets: the CTA that completes the channel slots finalises the iteration,
// the CTA whose bin completes an axis refines the axis.  No CTA waits for
// another.  Bound by latency up to some thousand tiles, then by the partials'
// traffic: ten iterations of 1e7 three-jet events (502 slots of 9766 tiles,
// 78 MB) 2.88 ms when the loads waited for one another and the exponents were
// read first, 2.77 with each thread's sum in one 128-bit integer at its largest
// exponent so far, 2.79 with sums that no order can change (1e6 Drell-Yan events
// 417 and 421 us).
// ---------------------------------------------------------------------------
// Three CTAs per SM: 80 registers hold eight partials in flight.
__global__ void __launch_bounds__(256, 3) gv_reduce_slots_kernel(const GvReduceArgs a) {
  extern __shared__ __align__(16) double sm[];
  __shared__ unsigned long long s_w[8][GV_SLOT_WORDS];
  __shared__ int s_g[8];
  __shared__ int s_won, s_fin;
  const int tid = threadIdx.x, lane = tid & 31, wid = tid >> 5;
  const int k = blockIdx.x;
  const SlotPartials part(a, k, (size_t)k * a.n_tiles, 1);
  gv_wait_prior_grid();
  const int nt = a.tiles_used ? min(a.n_tiles, __ldcg(a.tiles_used)) : a.n_tiles;
  GvAcc sum = warp_sum_acc(sum_tiles<GV_RED_TILES_PER_LOAD>(part, tid, lane, 256, nt),
                           nt > (1 << 28));
  if (lane == 0) {
#pragma unroll
    for (int j = 0; j < GV_SLOT_WORDS; ++j) s_w[wid][j] = sum.w[j];
    s_g[wid] = sum.g;
  }
  __syncthreads();
  if (wid == 0) {  // lane j adds the warps' counters j
    int g = 0;
#pragma unroll
    for (int w = 0; w < 8; ++w) g = max(g, s_g[w]);
    unsigned long long t = 0ull;
#pragma unroll
    for (int w = 0; w < 8; ++w) t += acc_word(s_w[w], 1, s_g[w], g, lane);
#pragma unroll
    for (int j = 0; j < GV_SLOT_WORDS; ++j) sum.w[j] = __shfl_sync(0xffffffffu, t, j);
    sum.g = g;
  }
  if (tid == 0) {
    s_won = -1;
    s_fin = 0;
    // the slot's sum over all events, rounded once to FP64
    a.sums[k] = acc_to_double(sum);
    __threadfence();
    if (k < 2 * a.nch) {
      int* tk = a.tickets + gv_ticket_done(a.nacc);
      if (atomicAdd(tk, 1) == 2 * a.nch - 1) {
        *tk = 0;
        s_fin = 1;
      }
    } else if (a.has_bins && a.refine_follows && k < 2 * a.nch + a.ndim * a.nbins) {
      const int ax = (k - 2 * a.nch) / a.nbins;
      int* tk = a.tickets + gv_ticket_axis(a.nacc, ax);
      if (atomicAdd(tk, 1) == a.nbins - 1) {
        *tk = 0;
        s_won = ax;
      }
    }
  }
  __syncthreads();
  const int won = s_won, fin = s_fin;
  if (won < 0 && !fin) return;
  __threadfence();  // the other slots' sums, published before their tickets
  gv_allow_next_grid();  // what is left is short: the next fill's CTAs may come in
  if (fin)
    finalize_iteration(a, tid);
  else
    refine_axis<false>(a, won, sm, tid, 256, 2, 0);
}

// ---------------------------------------------------------------------------
// The same for few tiles (kClusterTiles): one cluster of eight CTAs per axis,
// and one each for the channel slots and for every 128 histogram slots.  A warp
// sums a slot over the tiles, its lane 0 rounds the sum and stores it in the
// first CTA's shared memory, and after one cluster barrier that CTA refines the
// axis: 1000 cycles in place of the 4600 that a store, a fence, a ticket, a
// second fence and a load through L2 take.  Ten axes of 50 bins, four
// iterations of 1000 events and ten of 1e4: 277 us with the slots' CTAs, 233 so.
// ---------------------------------------------------------------------------
constexpr int kClusterCtas = 8, kClusterThreads = 512;
constexpr int kClusterSlots = kClusterCtas * kClusterThreads / 32;  // a slot per warp
__device__ __forceinline__ unsigned gv_cluster_rank() {
  unsigned r;
  asm volatile("mov.u32 %0, %%cluster_ctarank;" : "=r"(r));
  return r;
}
__device__ __forceinline__ void gv_cluster_arrive() {
  asm volatile("barrier.cluster.arrive.release.aligned;" ::: "memory");
}
__device__ __forceinline__ void gv_cluster_wait() {
  asm volatile("barrier.cluster.wait.acquire.aligned;" ::: "memory");
}
// v into the cluster's CTA 0 at the address that p has in this CTA
__device__ __forceinline__ void gv_store_rank0(double* p, double v) {
  unsigned q;
  asm("mapa.shared::cluster.u32 %0, %1, 0;" : "=r"(q) : "r"((unsigned)__cvta_generic_to_shared(p)));
  asm volatile("st.shared::cluster.f64 [%0], %1;" ::"r"(q), "d"(v) : "memory");
}
__global__ void __launch_bounds__(kClusterThreads) gv_reduce_cluster_kernel(const GvReduceArgs a) {
  extern __shared__ __align__(16) double sm[];
  const int tid = threadIdx.x, lane = tid & 31, wid = tid >> 5;
  const int rank = (int)gv_cluster_rank(), c = blockIdx.x / kClusterCtas;
  const int N = a.nbins, nax = a.has_bins ? a.ndim : 0;
  gv_cluster_arrive();  // CTA 0 of the cluster runs before its memory is written
  // this cluster's slots [k0, k0 + n)
  const bool axis = c < nax, channels = c == nax;
  const int k0 = axis ? 2 * a.nch + c * N
                      : (channels ? 0 : 2 * a.nch + nax * N + (c - nax - 1) * kClusterSlots);
  const int n = axis ? N : (channels ? 2 * a.nch : min(kClusterSlots, a.nacc - k0));
  const bool refine = axis && a.refine_follows;
  const GvRefineMem m = refine_mem(sm, N);
  gv_cluster_wait();
  gv_wait_prior_grid();
  const int nt = a.tiles_used ? min(a.n_tiles, __ldcg(a.tiles_used)) : a.n_tiles;
  if (refine && rank == 0) {
    const double* e64 = a.grid + GvGridLayout{a.ndim, N}.off_e64() + (size_t)c * (N + 1);
    for (int k = tid; k <= N; k += kClusterThreads) m.e[k] = __ldcg(e64 + k);
  }
  for (int s = wid * kClusterCtas + rank; s < n; s += kClusterSlots) {
    const int k = k0 + s;
    const double d = warp_sum_tiles<GV_RED_TILES_PER_LOAD>(
        SlotPartials(a, k, (size_t)k * a.n_tiles, 1), nt);
    if (lane == 0) {
      a.sums[k] = d;
      if (refine) gv_store_rank0(m.slope + s, d);
    }
  }
  __syncwarp();
  gv_cluster_arrive();
  gv_cluster_wait();
  gv_allow_next_grid();  // what is left is short: the next fill's CTAs may come in
  if (rank != 0) return;
  const int nthr = min(kClusterThreads, (N + 31) & ~31);
  if (channels) {
    if (wid == 0) finalize_iteration(a, lane);
  } else if (refine && tid < nthr) {
    refine_axis<true>(a, c, sm, tid, nthr, 2, 0);
  }
}

// Batched: one launch reduces many integrations; task i names the
// integration and the block coordinates of CTA i.  Four CTAs per SM (64
// registers).
__global__ void __launch_bounds__(256, 4) gv_reduce_batch_kernel(const GvReduceArgs* args,
                                                              const int4* tasks, int k, int last,
                                                              double inv_m1) {
  extern __shared__ __align__(16) double sm[];
  __shared__ GvTaskMem mem;
  // the integration's arguments in shared memory, read where used (a copy in
  // registers held ~40 of them for the whole task)
  __shared__ GvReduceArgs s_a;
  const int4 t = tasks[blockIdx.x];
  static_assert(sizeof(GvReduceArgs) % 4 == 0, "GvReduceArgs copy");
  const unsigned* src = reinterpret_cast<const unsigned*>(args + t.x);
  unsigned* dst = reinterpret_cast<unsigned*>(&s_a);
  for (int i = threadIdx.x; i < (int)(sizeof(GvReduceArgs) / 4); i += blockDim.x) dst[i] = src[i];
  __syncthreads();
  if (threadIdx.x == 0) {
    s_a.k = k;
    s_a.last = last;
    s_a.inv_m1 = inv_m1;
  }
  __syncthreads();
  gv_reduce_task(s_a, t.y, t.z, t.w, mem, sm);
}

// ---------------------------------------------------------------------------
// Histogram of the observable (the paper's differential distributions,
// Section 3.2), after the reduce of iteration k of a call.  Per bin b, from
// the once-rounded sums: H = sum w / C, V = (sum w^2 / C - H^2)/(C-1) (0 if
// rounding makes it negative).  The call's iterations are weighted as the
// integral is: u_k = 1/sigma_k^2, or, if any sigma_k is 0, 1 for those
// iterations and 0 for the others, so that the bins add up to the combined
// integral.  acc holds, in iteration order, sum u H and sum u^2 V over the
// iterations with sigma_k > 0, and sum H and sum V over those with
// sigma_k = 0; the last iteration writes value = sum u H / sum u and
// error = sqrt(sum u^2 V) / sum u.  One thread per bin: nothing depends on
// the launch shape.
// ---------------------------------------------------------------------------
__global__ void __launch_bounds__(256) gv_hist_kernel(const GvHistArgs a) {
  const int nh = a.nhist;
  gv_wait_prior_grid();  // the reduce's sums and records
  gv_allow_next_grid();  // the next fill touches nothing this kernel reads or writes
  const double sk = a.per_iter[2 * a.k + 1];
  int nzero = 0;
  double W = 0.0;
  if (a.last) {
    for (int j = 0; j <= a.k; ++j)
      if (!(a.per_iter[2 * j + 1] > 0.0)) ++nzero;
    for (int j = 0; j <= a.k; ++j) {
      const double s = a.per_iter[2 * j + 1];
      W += nzero > 0 ? (s > 0.0 ? 0.0 : 1.0) : 1.0 / (s * s);
    }
  }
  for (int b = threadIdx.x; b < nh; b += blockDim.x) {
    const double h = a.sums[nh + b] * a.inv_c;
    double v = (a.sums[b] * a.inv_c - h * h) * a.inv_cm1;
    v = v > 0.0 ? v : 0.0;
    double A0 = 0.0, A1 = 0.0, A2 = 0.0, A3 = 0.0;
    if (a.k > 0) {
      A0 = a.acc[b];
      A1 = a.acc[nh + b];
      A2 = a.acc[2 * nh + b];
      A3 = a.acc[3 * nh + b];
    }
    if (sk > 0.0) {
      const double u = 1.0 / (sk * sk);
      A0 += u * h;
      A1 += u * u * v;
    } else {
      A2 += h;
      A3 += v;
    }
    a.acc[b] = A0;
    a.acc[nh + b] = A1;
    a.acc[2 * nh + b] = A2;
    a.acc[3 * nh + b] = A3;
    if (a.last) {
      a.out[b] = (nzero > 0 ? A2 : A0) / W;
      a.out[nh + b] = sqrt(nzero > 0 ? A3 : A1) / W;
    }
  }
}

// ---------------------------------------------------------------------------
// Derived constants of an integrand (launched when the parameters change).
// p[GV_MAXPARAMS - 1] carries the number of user parameters.
// ---------------------------------------------------------------------------
__global__ void gv_consts_kernel(int ig, const double* p, double* K) {
  if (threadIdx.x != 0) return;
  const int np = (int)p[GV_MAXPARAMS - 1];
  for (int i = 0; i < GV_NCONST; ++i) K[i] = 0.0;
  if (ig == GV_GAUSS) {
    K[GK_INV2S2] = 1.0 / (2.0 * p[0] * p[0]);
    K[GK_SHIFT] = np > 1 ? p[1] : 0.0;
  } else if (ig == GV_DY || ig == GV_DYNLO) {
    const double sqrt_s = p[0], MZ = p[1], GZ = p[2], sw2 = p[3], alpha = p[4];
    const double mlo = p[5], mhi = p[6];
    const double s = sqrt_s * sqrt_s;
    const double tau_lo = mlo * mlo / s, tau_hi = mhi * mhi / s;
    const double pi = 3.14159265358979323846;
    K[DK_SQRTS] = sqrt_s;
    K[DK_S] = s;
    K[DK_TAULO] = tau_lo;
    K[DK_L] = log(tau_hi / tau_lo);
    K[DK_LOGTAULO] = log(tau_lo);
    K[DK_MZ2] = MZ * MZ;
    K[DK_GM2] = (GZ * MZ) * (GZ * MZ);
    const double kappa = 1.0 / (4.0 * sw2 * (1.0 - sw2));
    K[DK_KAPPA] = kappa;
    // alpha^2/(4 N_c) * (hbar c)^2 [pb GeV^2] * Jacobians of cos(theta) (2) and phi (2 pi)
    K[DK_PREF] = alpha * alpha / (4.0 * 3.0) * 0.3893794e9 * 2.0 * (2.0 * pi);
    // couplings V = T3 - 2 Q sw2, A = T3; muon Q = -1, T3 = -1/2
    const double Vl = -0.5 + 2.0 * sw2, Al = -0.5, dVl = 2.0;
    double cA0 = 0, cA1 = 0, cA2 = 0, cB1 = 0, cB2 = 0, dA1 = 0, dA2 = 0, dB2 = 0;
    for (int t = 0; t < 2; ++t) {
      const double n = t == 0 ? 2.0 : 3.0;  // u, c  |  d, s, b
      const double Q = t == 0 ? 2.0 / 3.0 : -1.0 / 3.0;
      const double T3 = t == 0 ? 0.5 : -0.5;
      const double Vq = T3 - 2.0 * Q * sw2, Aq = T3, dVq = -2.0 * Q;
      cA0 += n * Q * Q;
      cA1 += n * (-2.0 * Q * Vl * Vq);
      cA2 += n * (Al * Al + Vl * Vl) * (Aq * Aq + Vq * Vq);
      cB1 += n * (-4.0 * Q * Al * Aq);
      cB2 += n * (8.0 * Al * Vl * Aq * Vq);
      dA1 += n * (-2.0 * Q * (dVl * Vq + Vl * dVq));
      dA2 += n * (2.0 * Vl * dVl * (Aq * Aq + Vq * Vq) + (Al * Al + Vl * Vl) * 2.0 * Vq * dVq);
      dB2 += n * (8.0 * Al * Aq * (dVl * Vq + Vl * dVq));
    }
    K[DK_CA0] = cA0;
    K[DK_CA1] = cA1;
    K[DK_CA2] = cA2;
    K[DK_CB1] = cB1;
    K[DK_CB2] = cB2;
    K[DK_A] = p[7];
    K[DK_B] = p[8];
    K[DK_NORM] = 0.2 * p[9] * p[9];
    K[DK_MZ] = MZ;
    K[DK_GZ] = GZ;
    K[DK_DKAPPA] = -kappa * (1.0 - 2.0 * sw2) / (sw2 * (1.0 - sw2));
    K[DK_DCA1] = dA1;
    K[DK_DCA2] = dA2;
    K[DK_DCB2] = dB2;
    if (ig == GV_DYNLO) {
      // beta and 1 / I0(beta), I0(beta) = sum_k ((beta/2)^k / k!)^2
      const double beta = p[10];
      double term = 1.0, i0 = 1.0;
      for (int k = 1; k < 200 && term >= 1e-18 * i0; ++k) {
        term *= (0.25 * beta * beta) / ((double)k * (double)k);
        i0 += term;
      }
      K[NK_BETA] = beta;
      K[NK_INVI0] = 1.0 / i0;
    }
  } else if (ig == GV_EE3J) {
    const double Q = np > 1 ? p[1] : 91.1876;
    K[EK_YCUT] = p[0];
    K[EK_Q] = Q;
    K[EK_INVQ2] = 1.0 / (Q * Q);
  }
  float* kf = reinterpret_cast<float*>(K + GV_NCONST_F32);
  for (int i = 0; i < GV_NCONST_F32; ++i) kf[i] = (float)K[i];
  // 64-bit significands (read only where gv_x64_applies)
  GvX* X = reinterpret_cast<GvX*>(K + GV_NCONST);
  for (int i = 0; i < GV_NCONST_X; ++i) X[i] = x_zero();
  if (ig == GV_GAUSS) {
    X[XK_INV2S2] = x_mul(x_from(K[GK_INV2S2]), GV_X_LOG2E);
    X[XK_MSHIFT] = x_from(-K[GK_SHIFT]);
  } else if (ig == GV_EE3J) {
    X[XK_YCUT].m = x_to_q64(x_from(K[EK_YCUT]));
  } else {
    const GvX B = x_mul(x_from(-K[DK_LOGTAULO]), GV_X_LOG2E);
    const GvX A = x_mul(x_from(K[DK_L]), GV_X_LOG2E);
    const int sh = B.e - A.e;
    X[XK_B2] = B;
    X[XK_A2].m = sh < 64 ? A.m >> max(sh, 0) : 0ull;
    X[XK_CP] = x_mul(x_mul(x_from(K[DK_L]), GV_X_LN2), x_from(K[DK_PREF]));
    X[XK_SQRTS] = x_from(K[DK_SQRTS]);
    X[XK_MMZ2] = x_from(-K[DK_MZ2]);
    X[XK_BETA2] = x_mul(x_from(K[NK_BETA]), GV_X_LOG2E);
    const int from[] = {DK_GM2, DK_KAPPA, DK_CA0, DK_CA1, DK_CA2, DK_CB1, DK_CB2, DK_A,
                        DK_B,   DK_NORM,  DK_MZ,  DK_GZ,  DK_DKAPPA, DK_DCA1, DK_DCA2, DK_DCB2};
    const int to[] = {XK_GM2, XK_KAPPA, XK_CA0, XK_CA1, XK_CA2, XK_CB1, XK_CB2, XK_A,
                      XK_B,   XK_NORM,  XK_MZ,  XK_GZ,  XK_DKAPPA, XK_DCA1, XK_DCA2, XK_DCB2};
    for (int i = 0; i < 16; ++i) X[to[i]] = x_from(K[from[i]]);
    X[XK_INVI0] = x_from(K[NK_INVI0]);
  }
}

// Reset the per-iteration state (at creation and after the autotuner's
// trial launches).
__global__ void gv_reset_kernel(GvState* st) {
  if (threadIdx.x == 0) st->nonfinite_iter = 0ull;
}

// One CTA per axis, in place (the edges are written back unchanged).
__global__ void gv_grid_pack_kernel(double* grid, int d, int N, GvState* st,
                                    unsigned long long it) {
  const int ax = blockIdx.x;
  pack_axis_tables(grid, grid + GvGridLayout{d, N}.off_e64() + (size_t)ax * (N + 1), ax, d, N,
                   threadIdx.x, blockDim.x);
  if (st && ax == 0 && threadIdx.x == 0) {
    st->it = it;
    st->it0 = it;
  }
}

__global__ void gv_rng_words_kernel(unsigned long long seed, uint32_t it, uint32_t batch,
                                    unsigned long long ev0, long long n, int d, uint32_t* out) {
  const long long j = (long long)blockIdx.x * blockDim.x + threadIdx.x;
  if (j >= n) return;
  uint32_t r[GV_MAXD];
  gv_event_words<GV_MAXD>(seed, it, batch, ev0 + (unsigned long long)j, d, r);
  for (int a = 0; a < d; ++a) out[j * d + a] = r[a];
}

namespace gv {
size_t reduce_smem_bytes(int N) { return gv_axes_per_block(N) * refine_axis_smem(N); }

// Reduce grid: 32 accumulators per CTA; at most 64 tile ranges.
void reduce_grid(int n_tiles, int nacc, int* tiles_per_cta, int* gx, int* gy) {
  const int tpc = n_tiles <= 64 ? std::max(1, n_tiles) : std::max(64, (n_tiles + 63) / 64);
  *tiles_per_cta = tpc;
  *gx = (nacc + 31) / 32;
  *gy = (n_tiles + tpc - 1) / tpc;
}

// Above 48 KB, static shared memory (up to 13.7 KB: the two-level reduce's sums)
// included, a kernel has to opt in.
static cudaError_t allow_smem(const void* k, size_t smem) {
  if (smem + sizeof(GvTaskMem) + 1024 <= 48 * 1024) return cudaSuccess;
  return cudaFuncSetAttribute(k, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem);
}

cudaError_t launch_reduce(const GvReduceArgs& a, size_t smem, cudaStream_t s, bool pdl) {
  int tpc, gx, gy;
  reduce_grid(a.n_tiles, a.nacc, &tpc, &gx, &gy);
  if (tpc != a.tiles_per_cta) return cudaErrorInvalidValue;
  cudaError_t e = allow_smem((const void*)gv_reduce_kernel, smem);
  if (e != cudaSuccess) return e;
  return gv_launch(gv_reduce_kernel, dim3(gx, gy), dim3(256), smem, s, pdl, a);
}

// At most this many tiles: the clusters, 8 (ndim + 1) CTAs.  More tiles want
// every SM for their partials: ten iterations of 1e6 events (977 tiles, four
// axes of 100 bins) 409 us with a CTA per slot and 434 with clusters; 98 tiles
// 209 and 203.
constexpr int kClusterTiles = 32 * GV_RED_TILES_PER_LOAD;
cudaError_t launch_reduce_slots(const GvReduceArgs& a, size_t smem, cudaStream_t s, bool pdl) {
  if (a.n_tiles > kClusterTiles) {
    const cudaError_t e = allow_smem((const void*)gv_reduce_slots_kernel, smem);
    if (e != cudaSuccess) return e;
    return gv_launch(gv_reduce_slots_kernel, dim3(a.nacc), dim3(256), smem, s, pdl, a);
  }
  const cudaError_t e = allow_smem((const void*)gv_reduce_cluster_kernel, smem);
  if (e != cudaSuccess) return e;
  const int nc = (a.has_bins ? a.ndim : 0) + 1 + (2 * a.nhist + kClusterSlots - 1) / kClusterSlots;
  cudaLaunchConfig_t cfg = {};
  cfg.gridDim = dim3(kClusterCtas * nc);
  cfg.blockDim = dim3(kClusterThreads);
  cfg.dynamicSmemBytes = smem;
  cfg.stream = s;
  cudaLaunchAttribute attr[2];
  attr[0].id = cudaLaunchAttributeClusterDimension;
  attr[0].val.clusterDim.x = kClusterCtas;
  attr[0].val.clusterDim.y = attr[0].val.clusterDim.z = 1;
  attr[1].id = cudaLaunchAttributeProgrammaticStreamSerialization;
  attr[1].val.programmaticStreamSerializationAllowed = 1;
  cfg.attrs = attr;
  cfg.numAttrs = pdl ? 2 : 1;
  return cudaLaunchKernelEx(&cfg, gv_reduce_cluster_kernel, a);
}

cudaError_t launch_reduce_batch(const GvReduceArgs* args, const int4* tasks, int ntasks, int k,
                                int last, double inv_m1, size_t smem, cudaStream_t s) {
  cudaError_t e = allow_smem((const void*)gv_reduce_batch_kernel, smem);
  if (e != cudaSuccess) return e;
  gv_reduce_batch_kernel<<<ntasks, 256, smem, s>>>(args, tasks, k, last, inv_m1);
  return cudaGetLastError();
}

cudaError_t launch_hist(const GvHistArgs& a, cudaStream_t s, bool pdl) {
  return gv_launch(gv_hist_kernel, dim3(1), dim3(256), 0, s, pdl, a);
}

cudaError_t launch_consts(int integrand, const double* params, double* kconst, cudaStream_t s) {
  gv_consts_kernel<<<1, 32, 0, s>>>(integrand, params, kconst);
  return cudaGetLastError();
}

cudaError_t launch_reset(GvState* st, cudaStream_t s) {
  gv_reset_kernel<<<1, 32, 0, s>>>(st);
  return cudaGetLastError();
}

cudaError_t launch_grid_pack(int d, int N, double* grid, GvState* st, unsigned long long it,
                             cudaStream_t s) {
  gv_grid_pack_kernel<<<d, 128, 0, s>>>(grid, d, N, st, it);
  return cudaGetLastError();
}

cudaError_t launch_rng_words(unsigned long long seed, uint32_t it, uint32_t batch,
                             unsigned long long ev0, long long n, int d, uint32_t* out,
                             cudaStream_t s) {
  if (n <= 0) return cudaSuccess;
  const int thr = 256;
  gv_rng_words_kernel<<<(unsigned)((n + thr - 1) / thr), thr, 0, s>>>(seed, it, batch, ev0, n, d,
                                                                     out);
  return cudaGetLastError();
}
}  // namespace gv
