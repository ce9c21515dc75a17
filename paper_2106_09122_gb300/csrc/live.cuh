// Columns of a scene grid that can be non-zero ("live").  A scene pixel beyond
// the last library radius has a zero PSF, so dense storage of a wide grid is
// mostly zero columns (56 % at 12 of 16 lambda/D half width, 97 % at 64), and
// the products read only the live ones.  A pixel counts as live when, in half
// pixels X = 2 ix - (N - 1), Y = 2 iy - (N - 1), X^2 + Y^2 <= R2 with
// R2 = floor((2 r_last / S)^2 (1 + 1e-9)): integers, so host and device agree
// exactly, and a superset of the columns that the build fills (its FP64 test
// r <= r_last errs by some 1e-15).
#pragma once

#include <math.h>
#include <stdint.h>

constexpr int kLiveGroup = 32;  // split storage: liveness per 32 columns (64 bytes of a row)

inline long long live_r2(double r_last, double S) {
  if (r_last < 0.0) return -1;
  const double t = 2.0 * r_last / S, v = t * t * (1.0 + 1e-9);
  return v < 1099511627776.0 ? (long long)v : 1ll << 40;  // (2 N)^2 < 2^40: everything is live
}

// Live pixels [a, b) of scene row iy (a == b: none).
__host__ __device__ inline void live_row(int N, long long R2, int iy, int &a, int &b) {
  const long long Y = 2ll * iy - (N - 1), v = R2 - Y * Y;
  a = b = 0;
  if (v < 0) return;
  long long w = (long long)sqrt((double)v);
  while (w * w > v) --w;
  while ((w + 1) * (w + 1) <= v) ++w;
  const long long lo = N - 1 - w, hi = N - 1 + w;  // |2 ix - (N - 1)| <= w
  a = lo <= 0 ? 0 : (int)((lo + 1) / 2);
  b = hi >= 2ll * (N - 1) ? N : (int)(hi / 2) + 1;
  if (a >= b) a = b = 0;
}
