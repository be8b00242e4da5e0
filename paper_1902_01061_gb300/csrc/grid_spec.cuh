// Geometry of the uniform grid of the exact grid searches: plain arithmetic,
// for the device and for a host compiler (no CUDA headers).
#pragma once
#include <cmath>
#include <cstddef>
#include <cstdint>

#ifndef __CUDACC__
#define SCGR_HD inline
#else
#define SCGR_HD __host__ __device__ inline
#endif

namespace scgr {

// Uniform grid of the exact grid searches (on the device): origin, cell edge,
// cells per axis and in all, the cloud's largest extent.
struct GridSpec {
  float o[3];
  float h, inv_h, extent;
  int g[3];
  int ncell;
};
constexpr int GRID_CELLS_PER_POINT = 4;           // at most this many cells per point
constexpr int64_t GRID_MAX_CELLS = 1ll << 30;     // and in all: cell numbers are 32-bit
constexpr float GRID_MIN_EXTENT = 1e-30f;         // a smaller box is one cell: its reciprocals would overflow

SCGR_HD int64_t grid_most_cells(int64_t n) {
  const int64_t c = GRID_CELLS_PER_POINT * n;
  return c < GRID_MAX_CELLS ? c : GRID_MAX_CELLS;
}
// Entries of a cloud's cell counts: its most cells, one more, and a reserve of 64.
inline size_t grid_start_entries(int64_t n) { return (size_t)grid_most_cells(n) + 64 + 1; }

// Grid of a cloud from its box: cell edge h = sqrt(8 A / n), A the box's
// surface area (about 8 points per occupied cell on a surface sample), at most
// grid_most_cells(n) cells and 2^16 + 1 per axis.
SCGR_HD void make_grid_spec(const float* lo, const float* hi, int n, GridSpec* out) {
  float e[3], emax = 0.f;
  for (int a = 0; a < 3; ++a) {
    e[a] = hi[a] - lo[a];
    emax = fmaxf(emax, e[a]);
  }
  // in units of the largest extent, so that no product overflows
  const bool point = !(emax >= GRID_MIN_EXTENT);
  const float ie = point ? 0.f : 1.f / emax;
  const float x = e[0] * ie, y = e[1] * ie, z = e[2] * ie;
  const float A = 2.f * (x * y + y * z + z * x);
  float h = fmaxf(sqrtf(8.f * A / (float)n), fmaxf(8.f / (float)n, 1.f / 65536.f));
  const int64_t most = grid_most_cells(n);
  int g[3];
  auto cells = [&](float v) {
    const int c = (int)ceilf(v / h + 1e-4f);
    return c > 1 ? c : 1;
  };
  // one cell once h passes the largest extent, after some 60 steps at most
  for (;;) {
    g[0] = cells(x);
    g[1] = cells(y);
    g[2] = cells(z);
    if (h > 2.f || (int64_t)g[0] * g[1] <= most / g[2]) break;
    h *= 1.25f;
  }
  h = point ? 1.f : h * emax;
  out->h = h;
  out->inv_h = 1.f / h;
  out->extent = emax;
  for (int a = 0; a < 3; ++a) {
    out->o[a] = lo[a];
    out->g[a] = g[a];
  }
  out->ncell = g[0] * g[1] * g[2];
}

}  // namespace scgr
