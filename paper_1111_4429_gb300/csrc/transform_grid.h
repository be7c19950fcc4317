// The grid a product transform runs on (host code: no CUDA).
#pragma once
#include <stdint.h>

#include <algorithm>

namespace bgw {

// Line lengths that have kernels.
constexpr int kSupportedN[] = {8, 10, 12, 16, 20, 24, 30, 32, 36, 40, 48, 50, 60, 64};

// What one evaluation asks of its grid: `points` = max|Gv| + max|Gc| +
// max|Geps| + 1 over the axes, and the box [lo, hi] that holds every
// component of the three lists.
struct GridNeed {
  int points = 0;
  int lo = 0, hi = 0;
};

// A grid of s points serves when no kept coefficient aliases (s >= points)
// and every list lies in [-s/2, s/2), as the caller's n was checked for: a
// list wider than that would fold two of its vectors onto one slot (an
// epsilon list wider than the bands' products, or bands of one sphere far
// wider than the other's, even though nothing kept aliases).
inline bool grid_serves(int s, const GridNeed& g) { return s >= g.points && g.lo >= -(s / 2) && g.hi < s - s / 2; }

// Whether the pair transform's low-band lines run on a grid of s points: every
// kept frequency in the outer quarters, [-s/4, s/4).
inline bool grid_lowband(int s, int ng, const int32_t* geps) {
  if (s % 4) return false;
  for (int i = 0; i < 3 * ng; ++i)
    if (geps[i] < -(s / 4) || geps[i] >= s / 4) return false;
  return true;
}

// Any grid that serves gives the coefficients of the product itself, so the
// transforms run on the smallest such supported grid instead of the caller's
// (often a density grid, near twice the size needed).  4096 pairs, us a call in
// FP32 / FP64 (FP64 from 38 points on: 1024 pairs), spheres that need 8 points, 8^3
// 39 / 142, 16^3 67 / 716; need 14, 16^3 79 / 803, 20^3 117 / 1902; need 22, 24^3 203
// / 3379, 32^3 318 / 6905; need 31, 32^3 491 / 8535, 36^3 563 / 12793; need 38, 40^3
// 762 / 4856, 48^3 1024 / 7360; need 45, 48^3 2053 / 9159, 60^3 2161 / 17336.  A grid
// without the low-band lines is still the faster one (12 against 16, 20 against
// 24, 24 against 32, 36 against 40, 48 against 60) but for three: 30 (441 / 8387; 32:
// 361 / 7388), 50 in FP32 (need 49, N_G 2109 2071, 7153 2470; 60: 1902, 2231; FP64
// 11254 against 15557), and 60 where 64 has them (3895 / 19736 against 3037 / 18224).
inline int transform_grid(int n, const GridNeed& g, int ng, const int32_t* geps, bool fp32) {
  int m = n;
  for (int s : kSupportedN)
    if (grid_serves(s, g)) {
      m = std::min(m, s);
      break;
    }
  const int up = m == 30 ? 32 : m == 50 && fp32 ? 60 : m == 60 ? 64 : m;
  if (up > m && up <= n && !grid_lowband(m, ng, geps) && grid_lowband(up, ng, geps)) m = up;
  return m;
}

}  // namespace bgw
