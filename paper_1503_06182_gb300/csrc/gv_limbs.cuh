// gv_limbs.cuh -- exact sums of a tile's weights and of their squares in
// 32-bit shared-memory limbs.
//
// A weight is w = m 2^h with an integer significand m (24 bits in the FP32
// form, 53 in the FP64 form).  Its square is cut into 22-bit digits at
// absolute positions: the digit of limb index i counts units of
// 2^(22 i - 2 GV_SQ_OFF).  The digits of one event are therefore the same for
// every bin it falls into, and adding the event to a bin is three (FP32) or
// four 32-bit shared atomics with no further arithmetic; 1024 events of a
// tile leave 10 bits of headroom.  A row of L limbs per bin covers the events
// whose limb index lies within L - 4 of the tile's largest (at L = 9: weights
// down to 2^-55 of the tile's largest); a tile with smaller weights takes
// them in further passes over a lower window, so no weight is lost, and the
// passes a tile takes depend on its events alone.
//
// Before this, every bin of a tile had its own exponent (an atomicMax per
// axis and event) and every event shifted and split its square once per axis:
// about 45 instructions per axis and event against 8 now, and the tile's own
// sums took 128-bit shifts, adds and shuffles in every thread; they now go to
// per-lane columns of limbs with the same digits.  Bound by instruction issue
// before and after.  One FP32 fill of 1e6 events alone, before and now:
// Drell-Yan (4 axes) 28.7 and 22.0 us, 685 and 506 instructions per event;
// NLO-shaped (13 axes) 97 and 50 us; with a 60-bin histogram 34.5 and 26.4 us;
// 3-jet (5 axes, 1e7 events) 336 and 237 us.
#pragma once
#include "gv_common.cuh"
#include "gv_slotsum.cuh"

#define GV_LIMB_BITS 22
#define GV_LIMB_MASK 0x3FFFFFu
#define GV_SQ_OFF 1144  // 11 x 104: keeps every limb index positive (h >= -1126)
#define GV_W21_OFF 1155 // 21 x 55: the histogram's 21-bit digits of w

// Limbs per bin: 9 up to 1024 bins in all (weights down to 2^-55 of the tile's
// largest in one pass); above, fewer, so that the largest shapes still fit
// shared memory.  Odd, so that consecutive bins start in different banks.  Plain
// fills of up to 512 bins have 13 (2^-99): on a grid adapted over 40 iterations
// nearly every tile has an event below 2^-55, and a second pass; ten iterations
// of 1e6 Drell-Yan events then take 382 us with 9 and 330 with 13, on a fresh
// grid 314 and 326, and three jets of 1e7 events 2.71 and 2.74 ms.  With a
// histogram (535 and 562 us) or strata (1033 and 1131) the room is better spent
// on a fourth CTA per SM.
__host__ __device__ inline int gv_limbs(int dN, bool plain) {
  return plain && dN <= 512 ? 13 : (dN <= 1024 ? 9 : (dN <= 2048 ? 7 : 5));
}
// Rows of the per-lane columns of w (22-bit digits) and limbs per histogram
// bin of w (21-bit digits).  The largest weight stands at most 11 (L - 4) + 31
// bits above the lowest 22-bit digit (+ 30 above a 21-bit one): digit 3 (4) for
// L <= 9, digit 5 (6) for L = 13; its 24 or 53 bits reach 1 (2) or 3 digits
// further.
__host__ __device__ constexpr int gv_lane_rows(bool f64, int L = 9) {
  return (f64 ? 7 : 5) + (L > 9 ? 2 : 0);
}
__host__ __device__ constexpr int gv_hist_w_limbs(bool f64, int L) {
  return (f64 ? 9 : 7) + (L > 9 ? 2 : 0);
}

struct u192 {
  unsigned long long l0, l1, l2;
};

__device__ __forceinline__ void add192(u192& r, const u192& x) {
  asm("add.cc.u64 %0, %0, %3;\n\t"
      "addc.cc.u64 %1, %1, %4;\n\t"
      "addc.u64 %2, %2, %5;"
      : "+l"(r.l0), "+l"(r.l1), "+l"(r.l2)
      : "l"(x.l0), "l"(x.l1), "l"(x.l2));
}

// Arithmetic shift right of a 192-bit two's complement value.
__device__ __forceinline__ u192 sar192(u192 v, int s) {
  const unsigned long long ext = (unsigned long long)((long long)v.l2 >> 63);
  if (s <= 0) return v;
  if (s >= 192) return {ext, ext, ext};
  while (s >= 64) {
    v.l0 = v.l1;
    v.l1 = v.l2;
    v.l2 = ext;
    s -= 64;
  }
  if (s > 0) {
    v.l0 = (v.l0 >> s) | (v.l1 << (64 - s));
    v.l1 = (v.l1 >> s) | (v.l2 << (64 - s));
    v.l2 = (unsigned long long)((long long)v.l2 >> s);
  }
  return v;
}

// Left shift by 0 <= s < 64 (callers keep the result below 2^190).
__device__ __forceinline__ u192 shl192(u192 v, int s) {
  if (s <= 0) return v;
  v.l2 = (v.l2 << s) | (v.l1 >> (64 - s));
  v.l1 = (v.l1 << s) | (v.l0 >> (64 - s));
  v.l0 <<= s;
  return v;
}

// Adds v to the 32-bit word at shared-memory address p + OFF (p as
// gv_shared_address gives it): one instruction, address offset included.
template <int OFF>
__device__ __forceinline__ void gv_red(unsigned p, unsigned v) {
  asm volatile("red.shared.add.u32 [%0+%2], %1;" ::"r"(p), "r"(v), "n"(OFF) : "memory");
}
// The same where v != 0, without a branch.
template <int OFF>
__device__ __forceinline__ void gv_red_nonzero(unsigned p, unsigned v) {
  asm volatile(
      "{\n\t"
      ".reg .pred nz;\n\t"
      "setp.ne.u32 nz, %1, 0;\n\t"
      "@nz red.shared.add.u32 [%0+%2], %1;\n\t"
      "}" ::"r"(p),
      "r"(v), "n"(OFF)
      : "memory");
}
__device__ __forceinline__ unsigned gv_shared_address(const void* p) {
  return (unsigned)__cvta_generic_to_shared(p);
}

// Limb index and residue of h: h + GV_SQ_OFF = 11 limb + rem, for
// 0 <= h + GV_SQ_OFF < 4096 (5958 = ceil(2^16 / 11)).
__device__ __forceinline__ int gv_limb_index(int h) {
  return (int)(((unsigned)(h + GV_SQ_OFF) * 5958u) >> 16);
}

// A significand and the exponent of its last bit.
template <typename Real>
struct GvSig;
template <>
struct GvSig<float> {
  static constexpr int H = 0;  // the square's digits are those of m^2 2^(2 (e2 + H))
  static constexpr int LOW = 0;  // digits of the square below those
  static constexpr int BITS = 24;
  unsigned m;
  int e2;
  bool neg;
};
template <>
struct GvSig<double> {
  static constexpr int H = 21;   // of floor(m^2 2^-42), 64 bits
  static constexpr int LOW = 2;  // the other 42 bits
  static constexpr int BITS = 53;
  unsigned long long m;
  int e2;
  bool neg;
};

// The digits of (M << 2 rem), M the square: l[i] at limb index limb + i.
// FP32: M < 2^48 is exact, and the fourth digit is zero except for rem = 10.
__device__ __forceinline__ void gv_square_digits(const GvSig<float>& w, int rem, unsigned (&l)[4]) {
  const unsigned long long M = (unsigned long long)w.m * w.m;
  const unsigned lo = (unsigned)M, hi = (unsigned)(M >> 32), s = 2u * (unsigned)rem;
  l[0] = (lo << s) & GV_LIMB_MASK;
  l[1] = __funnelshift_r(lo, hi, 22u - s) & GV_LIMB_MASK;
  l[2] = (__funnelshift_r(lo, hi, 24u) >> (20u - s)) & GV_LIMB_MASK;
  l[3] = rem == 10 ? hi >> 14 : 0u;
}
// FP64: the high 64 bits of the 106-bit square.
__device__ __forceinline__ void gv_square_digits(const GvSig<double>& w, int rem,
                                                 unsigned (&l)[4]) {
  const unsigned long long P = __umul64hi(w.m << 11, w.m << 11);
  const unsigned s = 2u * (unsigned)rem;
  l[0] = ((unsigned)P << s) & GV_LIMB_MASK;
  l[1] = __funnelshift_r((unsigned)P, (unsigned)(P >> 32), 22u - s) & GV_LIMB_MASK;
  l[2] = (unsigned)(P >> (44u - s)) & GV_LIMB_MASK;
  l[3] = (unsigned)(P >> 46) >> (20u - s);
}
// The low 42 bits: the two digits below l[0] and the bits of l[0] below s (zero
// there).  The tile's own sums take them, the bins do not (a bin drops digits of
// that size anyway).
__device__ __forceinline__ void gv_square_low(const GvSig<double>& w, int rem, unsigned (&l)[3]) {
  const unsigned long long q = (w.m * w.m & 0x3FFFFFFFFFFull) << (2u * (unsigned)rem + 2u);
  l[0] = (unsigned)q & GV_LIMB_MASK;
  l[1] = (unsigned)(q >> 22) & GV_LIMB_MASK;
  l[2] = (unsigned)(q >> 44);
}

// The window of one pass: the squares' limb indices [base, base + L - 4] (their
// digits reach base + L - 1), and the lowest digit of w in units of 22 and 21
// bits.
struct GvWindow {
  int base, wbase, hbase;
};
template <typename Real>
__device__ __forceinline__ GvWindow gv_window(int e2max, int L) {
  GvWindow v;
  v.base = gv_limb_index(e2max + GvSig<Real>::H) - (L - 4);
  const int t = 11 * v.base - GvSig<Real>::H;  // e2 + GV_SQ_OFF of the smallest weight taken
  v.wbase = (t + 2200) / 22 - 100;             // (t > -2200)
  v.hbase = (t + GV_W21_OFF - GV_SQ_OFF + 2100) / 21 - 100;
  return v;
}

// Adds one weight to the columns of its lane: the square's digits and those
// of w (shared-memory addresses of the digits' first rows, 128 bytes a row).
// A lane's column takes at most 32 events of a tile, so the top digit of w
// needs no mask.
__device__ __forceinline__ unsigned gv_signed_digit(unsigned d, int s) { return (d ^ s) - s; }
__device__ __forceinline__ void gv_lane_add_w(const GvSig<float>& w, unsigned lw, int wbase) {
  const unsigned t = (unsigned)(w.e2 + GV_SQ_OFF);
  const unsigned idx = (t * 2979u) >> 16;  // t / 22
  const unsigned sh = t - 22u * idx;
  const int s = w.neg ? -1 : 0;
  const unsigned p = lw + (idx - (unsigned)wbase) * 128u;
  gv_red<0>(p, gv_signed_digit((w.m << sh) & GV_LIMB_MASK, s));
  gv_red<128>(p, gv_signed_digit(w.m >> (22u - sh), s));
}
__device__ __forceinline__ void gv_lane_add_w(const GvSig<double>& w, unsigned lw, int wbase) {
  const unsigned t = (unsigned)(w.e2 + GV_SQ_OFF);
  const unsigned idx = (t * 2979u) >> 16;
  const unsigned sh = t - 22u * idx;
  const int s = w.neg ? -1 : 0;
  const unsigned p = lw + (idx - (unsigned)wbase) * 128u;
  gv_red<0>(p, gv_signed_digit(((unsigned)w.m << sh) & GV_LIMB_MASK, s));
  gv_red<128>(p, gv_signed_digit((unsigned)(w.m >> (22u - sh)) & GV_LIMB_MASK, s));
  gv_red<256>(p, gv_signed_digit((unsigned)(w.m >> (44u - sh)) & GV_LIMB_MASK, s));
  gv_red<384>(p, gv_signed_digit((unsigned)(w.m >> 45) >> (21u - sh), s));
}
// (p: the row of the lowest digit, LOW rows below l[0]'s)
__device__ __forceinline__ void gv_lane_add_square(const GvSig<float>& w, int rem,
                                                   const unsigned (&l)[4], unsigned p) {
  gv_red<0>(p, l[0]);
  gv_red<128>(p, l[1]);
  gv_red<256>(p, l[2]);
  gv_red_nonzero<384>(p, l[3]);
}
__device__ __forceinline__ void gv_lane_add_square(const GvSig<double>& w, int rem,
                                                   const unsigned (&l)[4], unsigned p) {
  unsigned low[3];
  gv_square_low(w, rem, low);
  gv_red<0>(p, low[0]);
  gv_red<128>(p, low[1]);
  gv_red<256>(p, l[0] | low[2]);
  gv_red<384>(p, l[1]);
  gv_red<512>(p, l[2]);
  gv_red<640>(p, l[3]);
}
// The square's digits into a bin's row at address p.
template <typename Real>
__device__ __forceinline__ void gv_bin_add_square(const unsigned (&l)[4], unsigned p) {
  gv_red<0>(p, l[0]);
  gv_red<4>(p, l[1]);
  gv_red<8>(p, l[2]);
  if constexpr (sizeof(Real) == 8)
    gv_red<12>(p, l[3]);
  else
    gv_red_nonzero<12>(p, l[3]);
}
// w in 21-bit signed digits into a histogram bin's limbs (address of the
// bin's row): |digit| < 2^21, so 1024 of them stay in 32 bits with either
// sign.
template <typename Real>
__device__ __forceinline__ void gv_hist_add_w(const GvSig<Real>& w, unsigned row, int hbase) {
  const unsigned t = (unsigned)(w.e2 + GV_W21_OFF);
  const unsigned idx = t / 21u;
  const unsigned sh = t - 21u * idx;
  const int s = w.neg ? -1 : 0;
  const unsigned long long m = w.m;
  const unsigned p = row + (idx - (unsigned)hbase) * 4u;
  gv_red<0>(p, gv_signed_digit((unsigned)(m << sh) & 0x1FFFFFu, s));
  gv_red<4>(p, gv_signed_digit((unsigned)(m >> (21u - sh)) & 0x1FFFFFu, s));
  gv_red<8>(p, gv_signed_digit((unsigned)(m >> (42u - sh)) & 0x1FFFFFu, s));
  if constexpr (sizeof(Real) == 8) gv_red<12>(p, gv_signed_digit((unsigned)(m >> (63u - sh)), s));
}

// Warp-collective total of a lane column's `rows` digits (at most 16) as a
// 128-bit integer, row 0 counting units of 2^p (bits below 1 truncated row by
// row): lane j takes row j's sum over the lanes, shifts it into place, and
// the warp adds the rows.  Lane 0 returns the total.
template <bool SIGNED>
__device__ __forceinline__ u128 gv_lane_total(const unsigned* col, int rows, int p) {
  const int lane = threadIdx.x & 31;
  long long mine = 0;
  // a row of unsigned digits adds up to less than 2^32: those below 2^-32 of a
  // unit are nothing
#pragma unroll 4
  for (int j = SIGNED ? 0 : max(0, (-32 - p) / GV_LIMB_BITS); j < rows; ++j) {
    const unsigned v = col[j * 32 + lane];
    long long s;
    if constexpr (SIGNED)
      s = (long long)__reduce_add_sync(0xffffffffu, v & 0xFFFFu) +
          ((long long)__reduce_add_sync(0xffffffffu, (int)v >> 16) << 16);
    else
      s = (long long)__reduce_add_sync(0xffffffffu, v);
    if (lane == j) mine = s;
  }
  const unsigned long long ext = (unsigned long long)(mine >> 63);
  const int sh = GV_LIMB_BITS * lane + p;
  u128 r = {0ull, 0ull};
  if (lane < rows) {
    if (sh >= 64)
      r.hi = sh < 128 ? (unsigned long long)mine << (sh - 64) : 0ull;
    else if (sh > 0)
      r = u128{(unsigned long long)mine << sh, (unsigned long long)(mine >> (64 - sh))};
    else
      r = u128{(unsigned long long)(mine >> (sh > -64 ? -sh : 63)), ext};
  }
#pragma unroll
  for (int m = 8; m > 0; m >>= 1) {
    const u128 o = {shfl_xor_u64(r.lo, m), shfl_xor_u64(r.hi, m)};
    r = add128(r, o);
  }
  return r;
}

// The same for the forward fill, whose passes may cut the events into windows of
// either row length: the rows from absolute digit index `cut` on (row 0 is index
// j0 + cut), exactly, in units of that digit; lower ones drop.  Every lane below
// 16 returns the total.
template <bool SIGNED>
__device__ __forceinline__ u192 gv_lane_sum(const unsigned* col, int rows, int j0) {
  const int lane = threadIdx.x & 31;
  long long mine = 0;
#pragma unroll 4
  for (int j = max(0, -j0); j < rows; ++j) {
    const unsigned v = col[j * 32 + lane];
    long long s;
    if constexpr (SIGNED)
      s = (long long)__reduce_add_sync(0xffffffffu, v & 0xFFFFu) +
          ((long long)__reduce_add_sync(0xffffffffu, (int)v >> 16) << 16);
    else
      s = (long long)__reduce_add_sync(0xffffffffu, v);
    if (lane == j) mine = s;
  }
  const unsigned long long ext = (unsigned long long)(mine >> 63);
  const int sh = GV_LIMB_BITS * (j0 + lane), q = sh >> 6, r = sh & 63;
  const unsigned long long lo = (unsigned long long)mine << r;
  const unsigned long long hi = r ? (unsigned long long)(mine >> (64 - r)) : ext;
  u192 v = {0ull, 0ull, 0ull};
  if (mine != 0)
    v = q == 0 ? u192{lo, hi, ext} : (q == 1 ? u192{0ull, lo, hi} : u192{0ull, 0ull, q == 2 ? lo : 0ull});
#pragma unroll
  for (int m = 8; m > 0; m >>= 1) {
    const u192 o = {shfl_xor_u64(v.l0, m), shfl_xor_u64(v.l1, m), shfl_xor_u64(v.l2, m)};
    add192(v, o);
  }
  return v;
}
// Where those totals are cut for a tile of scale E: 22 to 43 bits below a unit of
// 2^(2 E - GV_FB) (squares) or 2^(E - GV_FB).
__device__ __forceinline__ int gv_square_cut(int E) { return (2 * E - GV_FB + 2 * GV_SQ_OFF) / 22 - 1; }
__device__ __forceinline__ int gv_w_cut(int E) { return (E - GV_FB + GV_SQ_OFF + 2200) / 22 - 101; }

// A bin's partial: a 112-bit integer at a bit position (gv_slotsum.cuh).  Of a
// bin's sums of w^2 it holds the limb of the largest digit index at which any of
// the tile's events has a nonzero digit in the bin, and the three below it, each
// summed over all events: at least 66 bits, at most 99.  What the limbs further
// down would carry into these is dropped, up to one unit per event.  So the
// partial is a function of the bin's events, whatever windows of limbs took them.
struct GvPartial {
  unsigned long long lo, hi;
  int pos;  // 0: empty
};
__device__ __forceinline__ GvPartial gv_bin_partial(const unsigned* row, int L, int base) {
  // a square of at least 2^46 (FP64: 2^62) has its top digit above two others:
  // the top limb t is at least 2
  int t = L - 1;
  unsigned a = row[t], b = row[t - 1], c = row[t - 2], d = row[t - 3];
  while (a == 0u && t > 2) {
    --t;
    a = b;
    b = c;
    c = d;
    d = t > 2 ? row[t - 3] : 0u;
  }
  if (a == 0u) return GvPartial{0ull, 0ull, 0};
  const u128 x = add128(u128{(unsigned long long)d + ((unsigned long long)c << 22),
                             (unsigned long long)a << 2},
                        u128{(unsigned long long)b << 44, b >> 20});
  return GvPartial{x.lo, x.hi, 22 * (base + t - 3) - 2 * GV_SQ_OFF + GV_POS_OFF};
}
// x of the windows so far, and the limbs of a lower one that x's digits reach.
// (The lower window's events have no digit above x's: theirs end at two limbs
// above its first window, where the smallest top digit of that stands.)
__device__ __forceinline__ GvPartial gv_bin_partial_more(GvPartial x, const unsigned* row, int L,
                                                         int base) {
  const int j = (x.pos - GV_POS_OFF + 2 * GV_SQ_OFF) / 22 - base;  // x's lowest digit; j >= 0
  u128 r = {x.lo, x.hi};
#pragma unroll
  for (int i = 0; i < 4; ++i) {
    const unsigned long long v = j + i < L ? row[j + i] : 0u;
    const int sh = 22 * i;  // at most 66
    r = add128(r, sh < 64 ? u128{v << sh, sh ? v >> (64 - sh) : 0ull} : u128{0ull, v << (sh - 64)});
  }
  return GvPartial{r.lo, r.hi, x.pos};
}
// A histogram bin's partial of w: two's complement, from its row of signed 21-bit
// digits.
__device__ __forceinline__ GvPartial gv_hist_partial(const int* row, int rows, int hbase) {
  int t = rows - 1;
  int a = row[t];
  while (a == 0 && t > 0) a = row[--t];
  if (a == 0) return GvPartial{0ull, 0ull, 0};
  u192 v = {(unsigned long long)(long long)a, (unsigned long long)((long long)a >> 63), 0ull};
#pragma unroll
  for (int i = 1; i <= 3; ++i) {
    const long long q = t >= i ? (long long)row[t - i] : 0ll;
    v = shl192(v, 21);
    const unsigned long long ext = (unsigned long long)(q >> 63);
    add192(v, u192{(unsigned long long)q, ext, ext});
  }
  return GvPartial{v.l0, v.l1, 21 * (hbase + t - 3) - GV_W21_OFF + GV_POS_OFF};
}
// The sum of two (a later pass over lower weights): the lower one aligned to the
// higher one's unit, bits below it dropped.  (|value| < 2^95: no overflow.)
__device__ __forceinline__ GvPartial gv_hist_partial_add(GvPartial x, GvPartial y) {
  if (x.pos == 0) return y;
  if (y.pos == 0) return x;
  if (x.pos < y.pos) {
    const GvPartial t = x;
    x = y;
    y = t;
  }
  const u192 s = sar192(u192{y.lo, y.hi, (unsigned long long)((long long)y.hi >> 63)}, x.pos - y.pos);
  const u128 r = add128(u128{x.lo, x.hi}, u128{s.l0, s.l1});
  return GvPartial{r.lo, r.hi, x.pos};
}
