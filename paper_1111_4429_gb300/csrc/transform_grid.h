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

// Any grid that serves gives the coefficients of the product itself, so the
// transforms run on the smallest such supported grid instead of the caller's
// (often a density grid, near twice the size needed).  Measured per pair
// (y,x passes + z pass, us): spheres that need 30 points, FP32 40^3 0.139,
// 32^3 0.080; FP64 3.70 and 1.71; spheres that need 44, FP32 60^3 0.553,
// 48^3 0.266.  The smallest is the fastest but for 30, where 32 allows the
// low-band lines (every kept frequency in [-8, 8)): FP32 0.096 against 0.080,
// FP64 1.93 against 1.71.  Lines of 36 and 50 points without the low band
// still beat low-band lines of 40 and 60.
inline int transform_grid(int n, const GridNeed& g, int ng, const int32_t* geps) {
  int m = n;
  for (int s : kSupportedN)
    if (grid_serves(s, g)) {
      m = std::min(m, s);
      break;
    }
  if (m == 30 && n >= 32) {
    for (int i = 0; i < 3 * ng; ++i)
      if (geps[i] < -8 || geps[i] >= 8) return m;
    m = 32;
  }
  return m;
}

}  // namespace bgw
