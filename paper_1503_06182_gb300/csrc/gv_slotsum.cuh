// gv_slotsum.cuh -- the sum of one slot's tile partials, the same bits in every
// order and grouping of the tiles.
//
// A partial is a signed 128-bit integer v at an absolute bit position: its value
// is v 2^(pos - GV_POS_OFF), 0 < pos < 2^16, |v| < 2^127 (pos = 0: none).  It is
// cut into five 32-bit digits at absolute multiples of 32 bits (the top one
// signed), and digits of one position add up in one 64-bit counter, without
// carries.  The counters are a window of GV_SLOT_WORDS positions: from one below
// the lowest digit of the highest partial (by pos / 32) to the top one.  A digit
// below the window is dropped whole.  Which digits are dropped so depends on the
// partials alone, and a counter on nothing else: threads, tile ranges and kernels
// may split the tiles as they like, and a batch's sums are a single context's bit
// for bit.  At least 32 bits below the lowest one of the largest partial are kept
// (98 or more below a bin's largest sum, 128 below the scale of the channels').
// At most 2^31 partials: a counter then stays below 2^63.
//
// Before, each thread kept one 128-bit integer at the largest exponent so far,
// with 20 spare bits, and shifted it down when a larger one came: bits were
// dropped from partial sums, and which ones was a matter of the order.  A partial
// costs 5 funnel shifts, 6 selects and 6 64-bit additions here (GvAcc), 8 selects,
// 8 shifts and 2 additions there.  Where a warp holds all partials of a slot, the
// window is known before the first addition, and the same sum is one 192-bit
// integer (GvAccFixed): with counters there, stages of few tiles took 1 to 2%
// more, so 1%.
#pragma once
#include <cstdint>
#ifdef __CUDA_ARCH__
#define GV_S_FN __device__ __forceinline__
#elif defined(__CUDACC__)
#define GV_S_FN __device__ __host__ inline
#else
#define GV_S_FN inline
#endif

#define GV_POS_OFF 2400   // keeps every position positive (2 E - GV_FB >= -2242)
#define GV_SLOT_WORDS 6

struct GvAcc {
  unsigned long long w[GV_SLOT_WORDS];  // signed counters of positions 32 (g - 1 + j)
  int g;                                // 0: nothing yet
};

GV_S_FN GvAcc acc_zero() {
  GvAcc a;
#pragma unroll
  for (int j = 0; j < GV_SLOT_WORDS; ++j) a.w[j] = 0ull;
  a.g = 0;
  return a;
}

// The upper word of (hi : lo) << r, 0 <= r < 32.
GV_S_FN unsigned acc_funnel(unsigned lo, unsigned hi, unsigned r) {
#ifdef __CUDA_ARCH__
  return __funnelshift_l(lo, hi, r);
#else
  return (unsigned)(((((unsigned long long)hi << 32) | lo) << r) >> 32);
#endif
}

// The window moved up to g >= a.g.
GV_S_FN void acc_raise(GvAcc& a, int g) {
  if (a.g != 0 && g - a.g < GV_SLOT_WORDS) {
    for (int m = g - a.g; m > 0; --m) {
#pragma unroll
      for (int j = 0; j + 1 < GV_SLOT_WORDS; ++j) a.w[j] = a.w[j + 1];
      a.w[GV_SLOT_WORDS - 1] = 0ull;
    }
    a.g = g;
  } else if (g > a.g) {
    a = acc_zero();
    a.g = g;
  }
}

// The five digits of the value with words v0 .. v3 (v3 signed), shifted by pos's
// residue; the top one signed.
struct GvDigits {
  unsigned d0, d1, d2, d3, d4;
};
GV_S_FN GvDigits acc_digits(unsigned v0, unsigned v1, unsigned v2, unsigned v3, int pos) {
  const unsigned r = (unsigned)pos & 31u;
  return GvDigits{v0 << r, acc_funnel(v0, v1, r), acc_funnel(v1, v2, r), acc_funnel(v2, v3, r),
                  acc_funnel(v3, (unsigned)((int)v3 >> 31), r)};
}
GV_S_FN unsigned long long acc_signed(unsigned d) {
  return (unsigned long long)(long long)(int)d;
}
// Adds the partial with words v0 .. v3 at pos > 0 whose lowest digit is o = a.g -
// pos / 32 below the window's second position: 0 or 1, the usual case,
GV_S_FN void acc_add_near(GvAcc& a, unsigned v0, unsigned v1, unsigned v2, unsigned v3, int pos,
                          int o) {
  const GvDigits d = acc_digits(v0, v1, v2, v3, pos);
  const bool u = o == 0;
  a.w[0] += u ? 0u : d.d0;
  a.w[1] += u ? d.d0 : d.d1;
  a.w[2] += u ? d.d1 : d.d2;
  a.w[3] += u ? d.d2 : d.d3;
  a.w[4] += u ? (unsigned long long)d.d3 : acc_signed(d.d4);
  a.w[5] += u ? acc_signed(d.d4) : 0ull;
}
// or more: digits below the window drop.
GV_S_FN void acc_add_far(GvAcc& a, unsigned v0, unsigned v1, unsigned v2, unsigned v3, int pos,
                         int o) {
  const GvDigits d = acc_digits(v0, v1, v2, v3, pos);
  unsigned long long e[5] = {d.d0, d.d1, d.d2, d.d3, acc_signed(d.d4)};
  for (int m = o < GV_SLOT_WORDS ? o - 1 : 5; m > 0; --m) {
#pragma unroll
    for (int j = 0; j < 4; ++j) e[j] = e[j + 1];
    e[4] = 0ull;
  }
#pragma unroll
  for (int j = 0; j < 5; ++j) a.w[j] += e[j];
}

// The same sum where the highest position is known before the first addition:
// the window's words as one 192-bit two's complement integer (up to 2^20
// partials).  Dropping the digits below the window is a shift of whole words.
struct GvAccFixed {
  unsigned w[GV_SLOT_WORDS];
};
GV_S_FN void acc_add_fixed(GvAccFixed& a, unsigned v0, unsigned v1, unsigned v2, unsigned v3,
                           int pos, int g) {
  const GvDigits d = acc_digits(v0, v1, v2, v3, pos);
  const unsigned sg = (unsigned)((int)d.d4 >> 31);
  const int o = g - (pos >> 5);
  const bool u = o == 0;
  unsigned x0 = u ? 0u : d.d0, x1 = u ? d.d0 : d.d1, x2 = u ? d.d1 : d.d2, x3 = u ? d.d2 : d.d3,
           x4 = u ? d.d3 : d.d4, x5 = u ? d.d4 : sg;
  if (o > 1) {
    const int m = o - 1;  // words to drop; more than four: all digits
    if (m & 1) x0 = x1, x1 = x2, x2 = x3, x3 = x4, x4 = x5, x5 = sg;
    if (m & 2) x0 = x2, x1 = x3, x2 = x4, x3 = x5, x4 = x5 = sg;
    if (m & 4) x0 = x4, x1 = x2 = x3 = x4 = x5 = sg;
    if (m > 4) x0 = x1 = x2 = x3 = x4 = x5 = 0u;
  }
#ifdef __CUDA_ARCH__
  asm("add.cc.u32 %0, %0, %6;\n\t"
      "addc.cc.u32 %1, %1, %7;\n\t"
      "addc.cc.u32 %2, %2, %8;\n\t"
      "addc.cc.u32 %3, %3, %9;\n\t"
      "addc.cc.u32 %4, %4, %10;\n\t"
      "addc.u32 %5, %5, %11;"
      : "+r"(a.w[0]), "+r"(a.w[1]), "+r"(a.w[2]), "+r"(a.w[3]), "+r"(a.w[4]), "+r"(a.w[5])
      : "r"(x0), "r"(x1), "r"(x2), "r"(x3), "r"(x4), "r"(x5));
#else
  const unsigned x[GV_SLOT_WORDS] = {x0, x1, x2, x3, x4, x5};
  unsigned long long c = 0ull;
  for (int j = 0; j < GV_SLOT_WORDS; ++j) {
    c += (unsigned long long)a.w[j] + x[j];
    a.w[j] = (unsigned)c;
    c >>= 32;
  }
#endif
}

// Counter j of b in a window at g >= b.g (b's counters at `stride` words).
GV_S_FN unsigned long long acc_word(const unsigned long long* b, int stride, int bg, int g, int j) {
  const int i = j + (g - bg);
  return bg != 0 && i < GV_SLOT_WORDS ? b[i * stride] : 0ull;
}

// Sign and magnitude of a 256-bit two's complement integer in units of 2^(32 (g -
// 1) - GV_POS_OFF): its leading 64 bits (bit 63 set, worth 2^(e - 63)) and whether
// anything lies below them.  False for zero.
GV_S_FN bool acc_leading(unsigned long long (&q)[4], int g, unsigned long long* window,
                         bool* sticky, int* e, bool* neg) {
  *neg = (long long)q[3] < 0;
  if (*neg) {
    unsigned long long c = 1ull;
#pragma unroll
    for (int j = 0; j < 4; ++j) {
      q[j] = ~q[j] + c;
      c = (c != 0ull && q[j] == 0ull) ? 1ull : 0ull;
    }
  }
  // the leading word, the next one, and whether anything lies below them
  const int i = q[3] ? 3 : (q[2] ? 2 : (q[1] ? 1 : 0));
  const unsigned long long h = i == 3 ? q[3] : (i == 2 ? q[2] : (i == 1 ? q[1] : q[0]));
  const unsigned long long n = i == 3 ? q[2] : (i == 2 ? q[1] : (i == 1 ? q[0] : 0ull));
  const bool low = (i == 3 && q[1] != 0ull) || (i >= 2 && q[0] != 0ull);
  if (h == 0ull) return false;
#ifdef __CUDA_ARCH__
  const int lz = __clzll((long long)h);
#else
  const int lz = __builtin_clzll(h);
#endif
  *window = lz ? (h << lz) | (n >> (64 - lz)) : h;
  *sticky = low || (n << lz) != 0ull;
  *e = 64 * i + 63 - lz + 32 * (g - 1) - GV_POS_OFF;
  return true;
}
// The same of the counters, after their carries.
GV_S_FN bool acc_window(const GvAcc& a, unsigned long long* window, bool* sticky, int* e,
                        bool* neg) {
  unsigned long long q[4];
  long long carry = 0;
#pragma unroll
  for (int j = 0; j < 3; ++j) {
    carry += (long long)a.w[2 * j];
    const unsigned lo = (unsigned)carry;
    carry >>= 32;
    carry += (long long)a.w[2 * j + 1];
    q[j] = ((unsigned long long)(unsigned)carry << 32) | lo;
    carry >>= 32;
  }
  q[3] = (unsigned long long)carry;
  return acc_leading(q, a.g, window, sticky, e, neg);
}
