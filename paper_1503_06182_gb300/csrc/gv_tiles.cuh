// gv_tiles.cuh -- how a stage's events are cut into tiles (host code, shared
// with the tests).
#pragma once
#include <algorithm>
#include <utility>
#include <vector>

#define GV_TILE 1024          // most events of a tile (see gv_tile_events)

// Arithmetic of an event: the FP64 pipe, FP32, or 64-bit significands on the
// integer pipes (gv_x64.cuh).
enum { GV_FORM_F64 = 0, GV_FORM_F32 = 1, GV_FORM_X64 = 2 };

// Events per tile of a stage of ncall events (plain forward stages, single or
// batched): 128 to GV_TILE, a function of the call count and the arithmetic
// alone, so that results do not depend on the launch shape.  One tile is one
// CTA: the size minimises the rounds of tiles over the 152 SMs times a tile's
// time, its events plus a fixed part (staging, zeroing, epilogue) worth t0
// events.  A smaller size has to save 4% of that: its tiles cost a batch, whose
// members share the SMs, more partials (64 members of 1e4 to 1e7 calls 20.5 ms
// with powers of two, 20.8 so; 20.9 if any saving counts).  Ten iterations with
// 128 and with 1024 events a tile: 1e4 calls of the FP64 NLO-shaped weight on
// 13 axes 297 and 619 us, of FP64 Drell-Yan 199 and 287, of FP32 Drell-Yan 159
// and 162.  Against the powers of two: an FP64 fit step of 1e5 calls (143 tiles
// of 704 instead of 98 of 1024) 585 and 495 us, the Gaussian on four axes 209
// and 197, ten iterations of 1e6 FP32 NLO events (1042 of 960) 750 and 727.
inline int gv_tile_events(long long ncall, int form) {
  const long long t0 = form == GV_FORM_F32 ? 256 : 96;
  long long best = 0;
  int T = GV_TILE;
  for (int t = GV_TILE; t >= 128; t -= 32) {
    const long long tiles = (ncall + t - 1) / t, cost = (tiles + 151) / 152 * (t + t0);
    if (best == 0 || 100 * cost < 96 * best) {
      best = cost;
      T = t;
    }
  }
  return T;
}

inline long long gv_tile_count(long long ncall, int form) {
  const int t = gv_tile_events(ncall, form);
  return (ncall + t - 1) / t;
}

// The most tiles of any stage of at most ncall events: what a workspace for
// ncall events has room for, so that it serves every smaller stage too.  The
// count is no monotone function of the calls: 1e5 FP64 calls are 143 tiles,
// 77824 are 152.  It grows until a tile size t needs another round of the SMs,
// at multiples of 152 t events, so the largest count below ncall stands at such
// a multiple.  From 25 rounds on no size saves 4% of the largest one's (a round
// is less), and the count is ncall / GV_TILE.  The 1600 multiples below that are
// listed once.
inline long long gv_most_tiles(long long ncall, int form) {
  using Ends = std::vector<std::pair<long long, long long>>;
  const auto list = [](int f) {
    Ends v;
    for (int t = 128; t <= GV_TILE; t += 32)
      for (long long n = 152ll * t; n <= 24ll * 152 * GV_TILE; n += 152ll * t)
        v.push_back({n, gv_tile_count(n, f)});
    std::sort(v.begin(), v.end());
    for (size_t i = 1; i < v.size(); ++i) v[i].second = std::max(v[i].second, v[i - 1].second);
    return v;
  };
  static const Ends ends[2] = {list(GV_FORM_X64), list(GV_FORM_F32)};
  const Ends& v = ends[form == GV_FORM_F32];
  long long most = gv_tile_count(ncall, form);
  const auto it = std::upper_bound(v.begin(), v.end(), std::make_pair(ncall, 1ll << 62));
  if (it != v.begin()) most = std::max(most, (it - 1)->second);
  return most;
}
