// Exact k-nearest neighbours and nearest-point queries through a uniform grid.
//
// The result is that of a brute-force search: the first k of the (key, index)
// order.  Points are counting-sorted into cells (the order inside a cell is
// arbitrary, so candidates are compared by (key, index) rather than relying on
// scan order).  A query scans a cube of cells around its own and grows it
// until the k-th key is certified: every unscanned point lies at least dout
// from the query, dout the distance to the boundary of the scanned cube less
// a margin for the float32 cell arithmetic, and the k-th key is below dout^2.
//
// Several clouds are built and searched per launch (blockIdx.y: the reference
// and the template of a registration, or every cloud of a batch).  The grid's
// geometry is computed on the device, so nothing waits for the host; arrays
// are sized for the most cells a grid may have (GRID_CELLS_PER_POINT).
#include <cfloat>
#include <climits>
#include <cmath>

#include "common.cuh"

namespace scgr {

constexpr unsigned FULL = 0xffffffffu;

// ---- statistics and geometry --------------------------------------------------

// Sum over the block of NV doubles per thread (256 threads, fixed order);
// valid in thread 0.
template <int NV>
__device__ __forceinline__ void block_sum_warps(double (&v)[NV], double (*sh)[NV]) {
#pragma unroll
  for (int off = 16; off > 0; off >>= 1)
#pragma unroll
    for (int q = 0; q < NV; ++q) v[q] += __shfl_down_sync(FULL, v[q], off);
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
  if (lane == 0)
#pragma unroll
    for (int q = 0; q < NV; ++q) sh[warp][q] = v[q];
  __syncthreads();
  if (threadIdx.x < 32) {
#pragma unroll
    for (int q = 0; q < NV; ++q) v[q] = lane < RED_THREADS / 32 ? sh[lane][q] : 0.0;
#pragma unroll
    for (int off = RED_THREADS / 64; off > 0; off >>= 1)
#pragma unroll
      for (int q = 0; q < NV; ++q) v[q] += __shfl_down_sync(FULL, v[q], off);
  }
}

// Blocks of a cloud's reductions: two points per thread of each block, at
// most CLOUD_PARTS.
__host__ __device__ inline int cloud_parts(int n) {
  const int b = (n + 2 * RED_THREADS - 1) / (2 * RED_THREADS);
  return b < CLOUD_PARTS ? b : CLOUD_PARTS;
}

// Pass 1: coordinate sums (float64) and the bounding box of each block's points.
__global__ void __launch_bounds__(RED_THREADS) cloud_sums_kernel(const CloudSet cs, double* __restrict__ part,
                                                                 float* __restrict__ bpart) {
  __shared__ double sh[RED_THREADS / 32][3];
  __shared__ float shb[RED_THREADS / 32][6];
  const GridCloud& g = cs[blockIdx.y];
  const int nb = cloud_parts(g.n);
  if ((int)blockIdx.x >= nb) return;
  double v[3] = {0.0, 0.0, 0.0};
  float b[6] = {FLT_MAX, FLT_MAX, FLT_MAX, FLT_MAX, FLT_MAX, FLT_MAX};  // min, -max
  for (int i = blockIdx.x * RED_THREADS + threadIdx.x; i < g.n; i += nb * RED_THREADS) {
    const float4 c = g.P[i];
    v[0] += c.x; v[1] += c.y; v[2] += c.z;
    b[0] = fminf(b[0], c.x); b[1] = fminf(b[1], c.y); b[2] = fminf(b[2], c.z);
    b[3] = fminf(b[3], -c.x); b[4] = fminf(b[4], -c.y); b[5] = fminf(b[5], -c.z);
  }
#pragma unroll
  for (int off = 16; off > 0; off >>= 1)
#pragma unroll
    for (int q = 0; q < 6; ++q) b[q] = fminf(b[q], __shfl_down_sync(FULL, b[q], off));
  if ((threadIdx.x & 31) == 0)
#pragma unroll
    for (int q = 0; q < 6; ++q) shb[threadIdx.x >> 5][q] = b[q];
  block_sum_warps<3>(v, sh);  // synchronises: shb is written
  const size_t o = (size_t)blockIdx.y * CLOUD_PARTS + blockIdx.x;
  if (threadIdx.x == 0)
#pragma unroll
    for (int q = 0; q < 3; ++q) part[o * 6 + q] = v[q];
  if (threadIdx.x < 6) {
    float m = shb[0][threadIdx.x];
#pragma unroll
    for (int w = 1; w < RED_THREADS / 32; ++w) m = fminf(m, shb[w][threadIdx.x]);
    bpart[o * 6 + threadIdx.x] = m;
  }
}

// One block per cloud: its mean, box and grid.
__global__ void __launch_bounds__(RED_THREADS) cloud_mean_kernel(const CloudSet cs, const double* __restrict__ part,
                                                                 const float* __restrict__ bpart) {
  static_assert(CLOUD_PARTS <= RED_THREADS, "one partial per thread");
  __shared__ double sh[RED_THREADS / 32][3];
  __shared__ float shb[RED_THREADS / 32][6];
  const GridCloud& g = cs[blockIdx.y];
  const int nb = cloud_parts(g.n);
  const size_t o = (size_t)blockIdx.y * CLOUD_PARTS + threadIdx.x;
  double v[3] = {0.0, 0.0, 0.0};
  float b[6] = {FLT_MAX, FLT_MAX, FLT_MAX, FLT_MAX, FLT_MAX, FLT_MAX};
  if ((int)threadIdx.x < nb) {
#pragma unroll
    for (int q = 0; q < 3; ++q) v[q] = part[o * 6 + q];
#pragma unroll
    for (int q = 0; q < 6; ++q) b[q] = bpart[o * 6 + q];
  }
#pragma unroll
  for (int off = 16; off > 0; off >>= 1)
#pragma unroll
    for (int q = 0; q < 6; ++q) b[q] = fminf(b[q], __shfl_down_sync(FULL, b[q], off));
  if ((threadIdx.x & 31) == 0)
#pragma unroll
    for (int q = 0; q < 6; ++q) shb[threadIdx.x >> 5][q] = b[q];
  block_sum_warps<3>(v, sh);
  if (threadIdx.x == 0 && g.mean) {
    const double in = 1.0 / (double)g.n;
#pragma unroll
    for (int q = 0; q < 3; ++q) g.mean[q] = v[q] * in;
  }
  if (threadIdx.x == 32) {  // its own warp: runs beside the mean's float64
    float lo[3], hi[3];
    for (int q = 0; q < 3; ++q) {
      float a = shb[0][q], c = shb[0][3 + q];
      for (int w = 1; w < RED_THREADS / 32; ++w) {
        a = fminf(a, shb[w][q]);
        c = fminf(c, shb[w][3 + q]);
      }
      lo[q] = a;
      hi[q] = -c;
    }
    make_grid_spec(lo, hi, g.n, g.spec);
  }
}

// Pass 2: scatter sums about the mean (where the cloud wants them), and the
// cell counters cleared.
__global__ void __launch_bounds__(RED_THREADS) cloud_scatter_kernel(const CloudSet cs, double* __restrict__ part) {
  __shared__ double sh[RED_THREADS / 32][6];
  const GridCloud& g = cs[blockIdx.y];
  const int nb = cloud_parts(g.n);
  if ((int)blockIdx.x >= nb) return;
  if (g.start) {
    const int cells = g.spec->ncell + 1;
    for (int c = blockIdx.x * RED_THREADS + threadIdx.x; c < cells; c += nb * RED_THREADS) g.start[c] = 0;
  }
  if (!g.scatter) return;
  const double m0 = g.mean[0], m1 = g.mean[1], m2 = g.mean[2];
  double v[6] = {0.0, 0.0, 0.0, 0.0, 0.0, 0.0};
  for (int i = blockIdx.x * RED_THREADS + threadIdx.x; i < g.n; i += nb * RED_THREADS) {
    const float4 c = g.P[i];
    const double dx = c.x - m0, dy = c.y - m1, dz = c.z - m2;
    v[0] += dx * dx; v[1] += dx * dy; v[2] += dx * dz;
    v[3] += dy * dy; v[4] += dy * dz; v[5] += dz * dz;
  }
  block_sum_warps<6>(v, sh);
  if (threadIdx.x == 0) {
    const size_t o = (size_t)blockIdx.y * CLOUD_PARTS + blockIdx.x;
#pragma unroll
    for (int q = 0; q < 6; ++q) part[o * 6 + q] = v[q];
  }
}

// One block: cloud y's scatter matrix and the largest eigenvalue of scatter / n.
__device__ void cloud_lmax(const GridCloud& g, int y, const double* __restrict__ part) {
  __shared__ double sh[RED_THREADS / 32][6];
  if (!g.scatter) return;
  const int nb = cloud_parts(g.n);
  const size_t o = (size_t)y * CLOUD_PARTS + threadIdx.x;
  double v[6] = {0.0, 0.0, 0.0, 0.0, 0.0, 0.0};
  if ((int)threadIdx.x < nb)
#pragma unroll
    for (int q = 0; q < 6; ++q) v[q] = part[o * 6 + q];
  block_sum_warps<6>(v, sh);
  if (threadIdx.x != 0) return;
  const double S[9] = {v[0], v[1], v[2], v[1], v[3], v[4], v[2], v[4], v[5]};
  double C[9];
  const double in = 1.0 / (double)g.n;
#pragma unroll
  for (int q = 0; q < 9; ++q) {
    g.scatter[q] = S[q];
    C[q] = S[q] * in;
  }
  *g.lmax = sym3_max_eigenvalue(C);
}
__global__ void __launch_bounds__(RED_THREADS) cloud_lmax_kernel(const CloudSet cs, const double* __restrict__ part) {
  cloud_lmax(cs[blockIdx.y], blockIdx.y, part);
}

// ---- counting sort into cells ---------------------------------------------------

// Cell of coordinate v on an axis (clamped to the grid, so v may lie outside
// the box).  Float32: v - o and the product round, so a point may sit up to
// about 4e-7 of the distance v - o beyond its cell's faces; the certification
// below allows for it.
__device__ __forceinline__ int cell_coord(float v, float o, float inv_h, int g) {
  return (int)fminf(fmaxf(floorf((v - o) * inv_h), 0.f), (float)(g - 1));
}

// First sorted position of cell c (c = ncell: the number of points): the
// count scan keeps a block-local part per cell and one offset per block.
__device__ __forceinline__ int cell_start(const GridCloud& g, int c) { return g.start[c] + g.tot[c / SCAN_B]; }

// The cell of every point and its rank of arrival there.  Block 0 of a cloud
// finishes the cloud's statistics meanwhile (a float64 latency chain).
__global__ void __launch_bounds__(256) cell_count_kernel(const CloudSet cs, const double* __restrict__ part) {
  static_assert(RED_THREADS == 256, "cloud_lmax runs in one of these blocks");
  const GridCloud& g = cs[blockIdx.y];
  if (blockIdx.x == 0) {
    cloud_lmax(g, blockIdx.y, part);
    return;
  }
  const int i = (blockIdx.x - 1) * 256 + threadIdx.x;
  if (i >= g.n) return;
  const GridSpec& sp = *g.spec;
  const float4 c = g.P[i];
  const int cx = cell_coord(c.x, sp.o[0], sp.inv_h, sp.g[0]);
  const int cy = cell_coord(c.y, sp.o[1], sp.inv_h, sp.g[1]);
  const int cz = cell_coord(c.z, sp.o[2], sp.inv_h, sp.g[2]);
  const int cell = (cz * sp.g[1] + cy) * sp.g[0] + cx;
  g.cell[i] = make_int2(cell, atomicAdd(g.start + cell, 1));
}

// Exclusive scan of the counts in place, over blocks of SCAN_B cells (the
// entry ncell included, so that it becomes the number of points).
constexpr int SCAN_T = 256;
constexpr int SCAN_PER = SCAN_B / SCAN_T;

__device__ __forceinline__ int block_scan_excl(int v, int* shw, int nwarps, int* total) {
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
  int inc = v;
#pragma unroll
  for (int off = 1; off < 32; off <<= 1) {
    const int u = __shfl_up_sync(FULL, inc, off);
    if (lane >= off) inc += u;
  }
  if (lane == 31) shw[warp] = inc;
  __syncthreads();
  if (warp == 0) {
    int w = lane < nwarps ? shw[lane] : 0;
#pragma unroll
    for (int off = 1; off < 32; off <<= 1) {
      const int u = __shfl_up_sync(FULL, w, off);
      if (lane >= off) w += u;
    }
    shw[lane] = w;
  }
  __syncthreads();
  *total = shw[nwarps - 1];
  return inc - v + (warp > 0 ? shw[warp - 1] : 0);
}

__global__ void __launch_bounds__(SCAN_T) scan_local_kernel(const CloudSet cs) {
  __shared__ int sh[SCAN_B + SCAN_B / 32];  // padded: thread t reads 16 entries in a row
  __shared__ int shw[32];
  const GridCloud& g = cs[blockIdx.y];
  const int cells = g.spec->ncell + 1;
  const int base = blockIdx.x * SCAN_B;
  if (base >= cells) return;
  for (int t = threadIdx.x; t < SCAN_B; t += SCAN_T) sh[t + t / 32] = base + t < cells ? g.start[base + t] : 0;
  __syncthreads();
  int sum = 0;
#pragma unroll
  for (int u = 0; u < SCAN_PER; ++u) {
    const int t = threadIdx.x * SCAN_PER + u;
    sum += sh[t + t / 32];
  }
  int total;
  int run = block_scan_excl(sum, shw, SCAN_T / 32, &total);
#pragma unroll
  for (int u = 0; u < SCAN_PER; ++u) {
    const int t = threadIdx.x * SCAN_PER + u;
    const int v = sh[t + t / 32];
    sh[t + t / 32] = run;
    run += v;
  }
  __syncthreads();
  for (int t = threadIdx.x; t < SCAN_B && base + t < cells; t += SCAN_T) g.start[base + t] = sh[t + t / 32];
  // a grid of one block needs no second pass
  if (threadIdx.x == 0) g.tot[blockIdx.x] = cells <= SCAN_B ? 0 : total;
}

__global__ void __launch_bounds__(1024) scan_blocks_kernel(const CloudSet cs) {
  __shared__ int shw[32];
  const GridCloud& g = cs[blockIdx.y];
  const int nb = (g.spec->ncell + SCAN_B) / SCAN_B;
  if (nb <= 1) return;
  int carry = 0;
  for (int b0 = 0; b0 < nb; b0 += 1024) {
    const int b = b0 + threadIdx.x;
    const int v = b < nb ? g.tot[b] : 0;
    int total;
    const int ex = block_scan_excl(v, shw, 32, &total);
    if (b < nb) g.tot[b] = carry + ex;
    carry += total;
    __syncthreads();
  }
}

// Points in cell order, the index in w.
__global__ void __launch_bounds__(256) cell_scatter_kernel(const CloudSet cs) {
  const GridCloud& g = cs[blockIdx.y];
  const int i = blockIdx.x * 256 + threadIdx.x;
  if (i >= g.n) return;
  const int2 cr = g.cell[i];
  float4 c = g.P[i];
  c.w = __int_as_float(g.base + i);
  g.sorted[cell_start(g, cr.x) + cr.y] = c;
}

// ---- queries ---------------------------------------------------------------------

// Squared distance of the (key, index) order.  FUSED = false: (dx*dx + dy*dy)
// + dz*dz, each operation rounded on its own.  FUSED = true: the sums fused with
// the products they add, as the assembler does in the packed brute-force search
// that served clouds below KNN_FUSED_KEY points and batches before; near ties
// fall as they fell there (its last n % 4 candidates apart, which it keyed one by
// one without fusing).
template <bool FUSED>
__device__ __forceinline__ float grid_key(float4 q, float4 c) {
  const float dx = __fsub_rn(q.x, c.x), dy = __fsub_rn(q.y, c.y), dz = __fsub_rn(q.z, c.z);
  if (FUSED) return __fmaf_rn(dz, dz, __fmaf_rn(dx, dx, __fmul_rn(dy, dy)));
  return __fadd_rn(__fadd_rn(__fmul_rn(dx, dx), __fmul_rn(dy, dy)), __fmul_rn(dz, dz));
}

// (key, index) as one integer that sorts like the pair (keys are >= +0).
__device__ __forceinline__ u64 pack_cand(float key, float w) {
  return ((u64)__float_as_uint(key) << 32) | __float_as_uint(w);
}
__device__ __forceinline__ float cand_key(u64 c) { return __uint_as_float((unsigned)(c >> 32)); }
constexpr u64 NO_CAND = ~0ull;

// Distance from q to what lies outside the cube of cells within s of cell
// cc[] (cell edge h): the nearest face that has cells behind it, less the
// margin of the float32 cell arithmetic.  INFINITY: nothing is outside.
__device__ __forceinline__ float outside_distance(const float (&q)[3], const float* o, float h, const int (&cc)[3],
                                                  const int (&g)[3], int s, float extent) {
  float d = INFINITY;
#pragma unroll
  for (int a = 0; a < 3; ++a) {
    const float v = q[a] - o[a];
    const float margin = 1e-6f * fmaxf(extent, fabsf(v));
    if (cc[a] - s > 0) d = fminf(d, v - (float)(cc[a] - s) * h - margin);
    if (cc[a] + s < g[a] - 1) d = fminf(d, (float)(cc[a] + s + 1) * h - v - margin);
  }
  return d;
}
__device__ __forceinline__ bool certified(float key, float dout) {
  return dout > 0.f && key < dout * dout * (1.f - 1e-5f);  // false for a NaN key (no candidate)
}

// Sorted positions [b, b + len) of cells x0..x1 (clamped) of the grid's row (y, z).
__device__ __forceinline__ void row_cells(const GridCloud& g, const int (&n)[3], int x0, int x1, int y, int z, int& b,
                                          int& len) {
  b = len = 0;
  x0 = max(x0, 0);
  x1 = min(x1, n[0] - 1);
  if (x0 > x1) return;
  const int c = (z * n[1] + y) * n[0];
  b = cell_start(g, c + x0);
  len = cell_start(g, c + x1 + 1) - b;
}
// The same for any row; len 0 where it is outside the grid.
__device__ __forceinline__ void row_range(const GridCloud& g, const int (&n)[3], int x0, int x1, int y, int z, int& b,
                                          int& len) {
  b = len = 0;
  if (y >= 0 && y < n[1] && z >= 0 && z < n[2]) row_cells(g, n, x0, x1, y, z, b, len);
}

// The rows of cells inside the grid of the cube within s of cell cc.
__device__ __forceinline__ int cube_rows(const int (&cc)[3], const int (&n)[3], int s) {
  return (min(cc[1] + s, n[1] - 1) - max(cc[1] - s, 0) + 1) * (min(cc[2] + s, n[2] - 1) - max(cc[2] - s, 0) + 1);
}
__device__ __forceinline__ void cube_row(const int (&cc)[3], const int (&n)[3], int s, int r, int& y, int& z) {
  const int y0 = max(cc[1] - s, 0), ey = min(cc[1] + s, n[1] - 1) - y0 + 1;
  z = max(cc[2] - s, 0) + r / ey;
  y = y0 + r % ey;
}

__device__ __forceinline__ int warp_incl_scan(int v) {
  const int lane = threadIdx.x & 31;
#pragma unroll
  for (int off = 1; off < 32; off <<= 1) {
    const int u = __shfl_up_sync(FULL, v, off);
    if (lane >= off) v += u;
  }
  return v;
}
// Lane l's ranges have running lengths incl; the sorted position of the t-th
// point of all of them (t below the total; other t give some valid lane's).
__device__ __forceinline__ int flat_position(int incl, int b, int len, int t) {
  int r = 0;
#pragma unroll
  for (int st = 16; st > 0; st >>= 1) {
    const int v = __shfl_sync(FULL, incl, r + st - 1);
    if (v <= t) r += st;
  }
  const int first = __shfl_sync(FULL, b - (incl - len), r);
  return first + t;
}

__device__ __forceinline__ u64 umin64(u64 a, u64 b) { return a < b ? a : b; }
__device__ __forceinline__ u64 umax64(u64 a, u64 b) { return a < b ? b : a; }

// Ascending bitonic sort / merge of one value per lane.
__device__ __forceinline__ u64 warp_sort(u64 v) {
  const int lane = threadIdx.x & 31;
#pragma unroll
  for (int size = 2; size <= 32; size <<= 1)
#pragma unroll
    for (int st = size >> 1; st > 0; st >>= 1) {
      const u64 o = __shfl_xor_sync(FULL, v, st);
      const bool up = (lane & size) == 0 || size == 32;
      v = ((lane & st) == 0) == up ? umin64(v, o) : umax64(v, o);
    }
  return v;
}
__device__ __forceinline__ u64 warp_merge(u64 v) {  // v bitonic
  const int lane = threadIdx.x & 31;
#pragma unroll
  for (int st = 16; st > 0; st >>= 1) {
    const u64 o = __shfl_xor_sync(FULL, v, st);
    v = (lane & st) == 0 ? umin64(v, o) : umax64(v, o);
  }
  return v;
}

// One warp per query (in cell order, so that neighbouring warps read the same
// cells).  A cube's cells are rows of consecutive cells, i.e. ranges of
// sorted points: each lane looks up one range, the ranges are flattened over
// the lanes and 32 candidates are keyed at a time.
//
// Only candidates closer than what the cube certifies (dout) can settle the
// query, so the others are dropped at once.  If at least k remain they hold
// the answer: a threshold near the wanted count cuts them to a warp's width
// (their number grows like the threshold, an area, so interpolation finds it
// in one or two steps) and each candidate's rank is the number of smaller
// ones.  If fewer than k remain the cube grows.  A cube with more candidates
// than the buffer holds goes to knn_stream.
// Bound: issue slots and the look-ups' latency.  1M + 1M points, k = 16: 2.2 ms
// for both clouds (12.2 ms with a sorted list of 16 per query that every
// candidate was inserted into); 5,003 + 4,801 points: 43 us (brute force: 350).
//
// Two warps a block: queries differ in length and a block keeps its warps'
// places until the last is done (8 warps: 32 of 64 warps active on average).
// 1M + 1M points, the whole descriptor pass: 8 warps and 5 blocks an SM 3406
// us, 4 and 10 3223, 2 and 20 3225, 2 and 24 (40 registers) 3121; with rows
// inside the grid only 3067.  A batch's
// table entries are chunks of queries that 8 warps share.
constexpr int QUERY_WARPS = 2, QUERY_BLOCKS = 24;
constexpr int QUERY_TABLE_WARPS = 8, QUERY_TABLE_BLOCKS = 5;
constexpr int QUERY_CAP = 256;  // candidates a warp keeps
constexpr int QUERY_PER = QUERY_CAP / 32;

// The search without a limit on the candidates: those below the k-th key so
// far wait in the buffer, 32 of them are sorted across the lanes and merged
// into the warp's sorted list of the best 32.
template <bool FUSED>
__device__ __noinline__ void knn_stream(const GridCloud& g, float4 q, const float (&q3)[3], const int (&cc)[3],
                                        const int (&n3)[3], int k, u64* buf) {
  const int lane = threadIdx.x & 31;
  const GridSpec& sp = *g.spec;
  u64 best = NO_CAND, thr = NO_CAND;
  int cnt = 0;
  auto flush = [&]() {
    __syncwarp();
    const u64 v = warp_sort(lane < cnt ? buf[lane] : NO_CAND);
    const u64 rest = lane + 32 < cnt ? buf[lane + 32] : NO_CAND;
    best = warp_merge(umin64(best, __shfl_sync(FULL, v, 31 - lane)));
    thr = __shfl_sync(FULL, best, k - 1);
    __syncwarp();
    buf[lane] = rest;
    cnt = cnt > 32 ? cnt - 32 : 0;
  };
  // The cube's rows inside the grid: two entries a row, its parts on either side
  // of the cube scanned so far (the whole row in the first where that one does not
  // reach it).  A grid a few cells thick has few rows however far the cube goes.
  // It grows by a cell, from 16 on by a sixteenth, so that a query across a gap
  // of s cells takes some 16 log s steps (growing by a quarter from the start,
  // 100,000 points, k = 24: 7% more time of all queries, for those that need 5 cells).
  for (int done = -1;;) {
    const int s = max(1, done + 1 + (done >> 4));
    const unsigned nr = 2u * (unsigned)cube_rows(cc, n3, s);
    for (unsigned r0 = 0; r0 < nr; r0 += 32) {
      const unsigned r = r0 + lane;
      int b = 0, len = 0;
      if (r < nr) {
        int y, z;
        cube_row(cc, n3, s, (int)(r >> 1), y, z);
        const bool inner = abs(y - cc[1]) <= done && abs(z - cc[2]) <= done;
        const int x0 = r & 1 ? (inner ? cc[0] + done + 1 : n3[0]) : cc[0] - s;
        const int x1 = inner && !(r & 1) ? cc[0] - done - 1 : cc[0] + s;
        row_cells(g, n3, x0, x1, y, z, b, len);
      }
      const int incl = warp_incl_scan(len);
      const int total = __shfl_sync(FULL, incl, 31);
      for (int t0 = 0; t0 < total; t0 += 32) {
        const int pos = flat_position(incl, b, len, t0 + lane);
        u64 cand = NO_CAND;
        if (t0 + lane < total) {
          const float4 c = g.sorted[pos];
          cand = pack_cand(grid_key<FUSED>(q, c), c.w);
        }
        const bool pass = cand < thr;
        const unsigned m = __ballot_sync(FULL, pass);
        if (pass) buf[cnt + __popc(m & ((1u << lane) - 1))] = cand;
        cnt += __popc(m);
        if (cnt >= 32) flush();
      }
    }
    if (cnt > 0) flush();
    const float dout = outside_distance(q3, sp.o, sp.h, cc, n3, s, sp.extent);
    if (dout == INFINITY || certified(cand_key(thr), dout)) break;
    done = s;
  }
  if (lane < k) g.knn[(size_t)__float_as_int(q.w) * k + lane] = (int32_t)(unsigned)best;
}

template <bool FUSED>
__device__ __forceinline__ void knn_query(const GridCloud& g, int t, int k, u64* buf) {
  const int lane = threadIdx.x & 31;
  const GridSpec& sp = *g.spec;
  const int n3[3] = {sp.g[0], sp.g[1], sp.g[2]};
  const float4 q = g.sorted[t];
  const float q3[3] = {q.x, q.y, q.z};
  int cc[3];
#pragma unroll
  for (int a = 0; a < 3; ++a) cc[a] = cell_coord(q3[a], sp.o[a], sp.inv_h, n3[a]);
  const int keep = k <= 24 ? 32 : 64;  // candidates to rank, at most
  for (int s = 1; s <= 32; s += s < 4 ? 1 : s >> 1) {
    const float dout = outside_distance(q3, sp.o, sp.h, cc, n3, s, sp.extent);
    float lim = dout > 0.f ? dout * dout * (1.f - 1e-5f) : 0.f;  // INFINITY where the cube covers the grid
    const int rows = cube_rows(cc, n3, s);  // at most 57 x 57
    const int y0 = max(cc[1] - s, 0), z0 = max(cc[2] - s, 0), ey = min(cc[1] + s, n3[1] - 1) - y0 + 1;
    int cnt = 0;
    __syncwarp();
    for (int r0 = 0; r0 < rows && cnt <= QUERY_CAP; r0 += 32) {
      const int r = r0 + lane;
      int b = 0, len = 0;
      if (r < rows) {
        // a float quotient, at least 1 / (2 ey) from a whole number
        const int dz = (int)__fdividef((float)r + 0.5f, (float)ey);
        row_cells(g, n3, cc[0] - s, cc[0] + s, y0 + r - dz * ey, z0 + dz, b, len);
      }
      const int incl = warp_incl_scan(len);
      const int total = __shfl_sync(FULL, incl, 31);
      for (int t0 = 0; t0 < total && cnt <= QUERY_CAP; t0 += 32) {
        const int pos = flat_position(incl, b, len, t0 + lane);
        float key = INFINITY, id = 0.f;
        if (t0 + lane < total) {
          const float4 c = g.sorted[pos];
          key = grid_key<FUSED>(q, c);
          id = c.w;
        }
        const unsigned m = __ballot_sync(FULL, key < lim);
        const int at = cnt + __popc(m & ((1u << lane) - 1));
        if (key < lim && at < QUERY_CAP) buf[at] = pack_cand(key, id);
        cnt += __popc(m);
      }
    }
    if (cnt > QUERY_CAP) break;
    if (cnt < k) {
      if (lim == INFINITY) break;
      continue;
    }
    __syncwarp();
    if (cnt > keep) {
      u64 c[QUERY_PER];
      float top = 0.f;
#pragma unroll
      for (int j = 0; j < QUERY_PER; ++j) {
        c[j] = j * 32 + lane < cnt ? buf[j * 32 + lane] : NO_CAND;
        if (j * 32 + lane < cnt) top = fmaxf(top, cand_key(c[j]));
      }
      if (lim == INFINITY) {
#pragma unroll
        for (int off = 16; off > 0; off >>= 1) top = fmaxf(top, __shfl_xor_sync(FULL, top, off));
        lim = top;
      }
      // a threshold below which k to `keep` candidates lie
      float lo = 0.f, hi = lim, nlo = 0.f, nhi = (float)cnt;
      const float want = 0.5f * (float)(k + keep);
      bool found = false;
      for (int it = 0; it < 24; ++it) {
        const float f = fminf(fmaxf(__fdividef(want - nlo, nhi - nlo), 0.1f), 0.9f);
        const float mid = fmaf(hi - lo, f, lo);
        int below = 0;
#pragma unroll
        for (int j = 0; j < QUERY_PER; ++j)
          if (j * 32 < cnt) below += __popc(__ballot_sync(FULL, cand_key(c[j]) < mid));  // NO_CAND: NaN, not below
        if (below < k) {
          lo = mid;
          nlo = (float)below;
        } else if (below > keep) {
          hi = mid;
          nhi = (float)below;
        } else {
          lim = mid;
          found = true;
          break;
        }
      }
      if (!found) break;
      __syncwarp();
      cnt = 0;
#pragma unroll
      for (int j = 0; j < QUERY_PER; ++j) {
        const bool in = cand_key(c[j]) < lim;
        const unsigned m = __ballot_sync(FULL, in);
        if (in) buf[cnt + __popc(m & ((1u << lane) - 1))] = c[j];
        cnt += __popc(m);
      }
      __syncwarp();
    }
    // ranks in the (key, index) order: the number of smaller candidates
    int32_t* out = g.knn + (size_t)__float_as_int(q.w) * k;
    if (lane == 0) buf[cnt] = NO_CAND;  // read in pairs (cnt <= QUERY_CAP - 1 here: keep < QUERY_CAP)
    __syncwarp();
    const u64 c0 = lane < cnt ? buf[lane] : NO_CAND;
    int r0 = 0;
    for (int j = 0; j < cnt; j += 2) {
      const ulonglong2 o = *reinterpret_cast<const ulonglong2*>(buf + j);
      r0 += (o.x < c0 ? 1 : 0) + (o.y < c0 ? 1 : 0);
    }
    if (lane < cnt && r0 < k) out[r0] = (int32_t)(unsigned)c0;
    if (cnt > 32) {
      const u64 c1 = lane + 32 < cnt ? buf[lane + 32] : NO_CAND;
      int r1 = 0;
      for (int j = 0; j < cnt; j += 2) {
        const ulonglong2 o = *reinterpret_cast<const ulonglong2*>(buf + j);
        r1 += (o.x < c1 ? 1 : 0) + (o.y < c1 ? 1 : 0);
      }
      if (lane + 32 < cnt && r1 < k) out[r1] = (int32_t)(unsigned)c1;
    }
    return;
  }
  __syncwarp();
  knn_stream<FUSED>(g, q, q3, cc, n3, k, buf);
}

// Cloud blockIdx.y, one query per warp; or (a batch, whose clouds differ in
// size) the KNN_TABLE_CHUNK queries from table[b].y of cloud table[b].x.
template <bool FUSED, int WARPS, int BLOCKS>
__global__ void __launch_bounds__(WARPS * 32, BLOCKS)
    knn_query_kernel(const CloudSet cs, const int2* __restrict__ table, int k) {
  __shared__ __align__(16) u64 bufs[WARPS][QUERY_CAP];
  const int warp = threadIdx.x >> 5;
  if (!table) {
    const GridCloud& g = cs[blockIdx.y];
    const int t = blockIdx.x * WARPS + warp;
    if (t < g.n) knn_query<FUSED>(g, t, k, bufs[warp]);
    return;
  }
  const int2 e = table[blockIdx.x];
  const GridCloud& g = cs[e.x];
  const int end = min(g.n, e.y + KNN_TABLE_CHUNK);
  for (int t = e.y + warp; t < end; t += WARPS) {
    knn_query<FUSED>(g, t, k, bufs[warp]);
    __syncwarp();
  }
}

// ---- nearest gridded point of external queries -----------------------------------

// Whether each coarse cell (NEAREST_COARSE^3 fine cells) holds a point: counts.
__global__ void __launch_bounds__(256) coarse_count_kernel(const CloudSet cs, int* __restrict__ ccount) {
  const GridCloud& g = cs[0];
  const int n3[3] = {g.spec->g[0], g.spec->g[1], g.spec->g[2]};
  int m3[3];
#pragma unroll
  for (int a = 0; a < 3; ++a) m3[a] = (n3[a] + NEAREST_COARSE - 1) / NEAREST_COARSE;
  const int total = m3[0] * m3[1] * m3[2];
  for (int c = blockIdx.x * 256 + threadIdx.x; c < total; c += gridDim.x * 256) {
    const int x = c % m3[0] * NEAREST_COARSE, y = c / m3[0] % m3[1] * NEAREST_COARSE,
              z = c / (m3[0] * m3[1]) * NEAREST_COARSE;
    int cnt = 0;
    for (int r = 0; r < NEAREST_COARSE * NEAREST_COARSE; ++r) {
      int b, len;
      row_range(g, n3, x, x + NEAREST_COARSE - 1, y + r % NEAREST_COARSE, z + r / NEAREST_COARSE, b, len);
      cnt += len;
    }
    ccount[c] = cnt;
  }
}

// Counts of the cells of the next level (NEAREST_COARSE^3 coarse cells each),
// behind the coarse ones.
__global__ void __launch_bounds__(256) super_count_kernel(const CloudSet cs, int* __restrict__ ccount) {
  const GridCloud& g = cs[0];
  int m3[3], s3[3];
#pragma unroll
  for (int a = 0; a < 3; ++a) {
    m3[a] = (g.spec->g[a] + NEAREST_COARSE - 1) / NEAREST_COARSE;
    s3[a] = (m3[a] + NEAREST_COARSE - 1) / NEAREST_COARSE;
  }
  const int coarse = m3[0] * m3[1] * m3[2], total = s3[0] * s3[1] * s3[2];
  for (int c = blockIdx.x * 256 + threadIdx.x; c < total; c += gridDim.x * 256) {
    const int x0 = c % s3[0] * NEAREST_COARSE, y0 = c / s3[0] % s3[1] * NEAREST_COARSE,
              z0 = c / (s3[0] * s3[1]) * NEAREST_COARSE;
    int cnt = 0;
    for (int z = z0; z < min(z0 + NEAREST_COARSE, m3[2]); ++z)
      for (int y = y0; y < min(y0 + NEAREST_COARSE, m3[1]); ++y)
        for (int x = x0; x < min(x0 + NEAREST_COARSE, m3[0]); ++x) cnt += ccount[(z * m3[1] + y) * m3[0] + x];
    ccount[coarse + c] = cnt;
  }
}

// One warp per query.  First the cube of cells around it, as ranges of
// sorted points flattened over the lanes: enough for a query on the surface.
// A query that this does not certify searches shells of large cells (edge
// 4 * `coarse` fine cells; a query at distance D would otherwise visit about
// (1.7 D / h)^3 fine cells, nearly all empty): each lane tests one cell, empty
// ones and ones whose box lies beyond the best key are dropped, and the warp
// takes the others nearest first: of a large cell's 4^3 coarse cells it
// scans, again nearest first and two at a time, the rows of fine cells that the
// best key does not rule out (a far query is a chain of dependent look-ups: the
// fewer links, the shorter).  The
// result is the (key, index)-first point whatever the order of the cells and
// of the points in a cell.
// Bound: issue slots and the latency of the range look-ups; a query on the
// surface costs about two hundred warp instructions.  (Shells of coarse cells,
// interiors enumerated, 300,000 reference points, 250,007 queries: 823 us;
// now 566 us: 154 for the 231,563 queries within a cell edge of the surface, the
// rest for 18,444 farther ones, 20 to 200 us of chain each.)
// Two warps a block (4: 584 us a change mask, 8: 597, 2: 552); more blocks an SM
// by fewer registers cost more than they hide (2 and 20 blocks: 594).
constexpr int NEAREST_WARPS = 2;

__global__ void __launch_bounds__(NEAREST_WARPS * 32, 16)
    nearest_query_kernel(const CloudSet cs, int coarse, const int* __restrict__ ccount, const float* __restrict__ q3,
                         int nq, int32_t* __restrict__ idx_out, float* __restrict__ key_out) {
  const GridCloud& g = cs[0];
  const int lane = threadIdx.x & 31;
  const int t = blockIdx.x * NEAREST_WARPS + (threadIdx.x >> 5);
  if (t >= nq) return;
  const GridSpec& sp = *g.spec;
  const int n3[3] = {sp.g[0], sp.g[1], sp.g[2]};
  const float q[3] = {q3[3 * (size_t)t], q3[3 * (size_t)t + 1], q3[3 * (size_t)t + 2]};
  const float4 q4 = make_float4(q[0], q[1], q[2], 0.f);
  int cc[3];
  float v[3], margin[3];
#pragma unroll
  for (int a = 0; a < 3; ++a) {
    cc[a] = cell_coord(q[a], sp.o[a], sp.inv_h, n3[a]);
    v[a] = q[a] - sp.o[a];
    margin[a] = 1e-6f * fmaxf(sp.extent, fabsf(v[a]));
  }
  // the warp's best of the points of its lanes' ranges
  auto scan_ranges = [&](int b, int len) {
    const int incl = warp_incl_scan(len);
    const int cnt = __shfl_sync(FULL, incl, 31);
    u64 mine = NO_CAND;
    for (int t0 = 0; t0 < cnt; t0 += 64) {  // two loads in flight
      const int at0 = flat_position(incl, b, len, t0 + lane);
      const int at1 = t0 + 32 < cnt ? flat_position(incl, b, len, t0 + 32 + lane) : at0;
      float4 p0 = make_float4(NAN, NAN, NAN, 0.f), p1 = p0;
      if (t0 + lane < cnt) p0 = g.sorted[at0];
      if (t0 + 32 + lane < cnt) p1 = g.sorted[at1];
      if (t0 + lane < cnt) mine = umin64(mine, pack_cand(grid_key<false>(q4, p0), p0.w));
      if (t0 + 32 + lane < cnt) mine = umin64(mine, pack_cand(grid_key<false>(q4, p1), p1.w));
    }
#pragma unroll
    for (int off = 16; off > 0; off >>= 1) mine = umin64(mine, __shfl_xor_sync(FULL, mine, off));
    return mine;
  };
  int b = 0, len = 0;
  if (lane < 9) row_range(g, n3, cc[0] - 1, cc[0] + 1, cc[1] + lane % 3 - 1, cc[2] + lane / 3 - 1, b, len);
  u64 best = scan_ranges(b, len);
  float dout = outside_distance(q, sp.o, sp.h, cc, n3, 1, sp.extent);
  if (dout != INFINITY && !certified(cand_key(best), dout)) {
    // squared distance to a cell's box, less the margins, as bits that sort like it
    constexpr unsigned NO_CELL = ~0u;
    auto box_bits = [&](int x, int y, int z, float H) {
      const int xyz[3] = {x, y, z};
      float d2 = 0.f;
#pragma unroll
      for (int a = 0; a < 3; ++a) {
        const float below = (float)xyz[a] * H - v[a] - margin[a];
        const float above = v[a] - (float)(xyz[a] + 1) * H - margin[a];
        const float d = fmaxf(0.f, fmaxf(below, above));
        d2 = fmaf(d, d, d2);
      }
      return __float_as_uint(d2 * (1.f - 1e-5f));
    };
    // the same for a row of `coarse` fine cells
    auto row_d2 = [&](int x, int y, int z) {
      const int lo[3] = {x, y, z}, hi[3] = {x + coarse, y + 1, z + 1};
      float d2 = 0.f;
#pragma unroll
      for (int a = 0; a < 3; ++a) {
        const float below = (float)lo[a] * sp.h - v[a] - margin[a];
        const float above = v[a] - (float)hi[a] * sp.h - margin[a];
        const float d = fmaxf(0.f, fmaxf(below, above));
        d2 = fmaf(d, d, d2);
      }
      return d2 * (1.f - 1e-5f);
    };
    // the lane whose cell is nearest; -1 when none is left that the best key
    // (NaN: no candidate yet) does not rule out
    auto nearest_lane = [&](unsigned bits) {
      const unsigned m = __reduce_min_sync(FULL, bits);
      if (m == NO_CELL || __uint_as_float(m) > cand_key(best)) return -1;
      return __ffs(__ballot_sync(FULL, bits == m)) - 1;
    };
    constexpr int NC = NEAREST_COARSE;
    const float H = sp.h * (float)coarse, HS = H * (float)NC;
    int m3[3], s3[3];
#pragma unroll
    for (int a = 0; a < 3; ++a) {
      m3[a] = (n3[a] + coarse - 1) / coarse;
      s3[a] = (m3[a] + NC - 1) / NC;
      cc[a] /= coarse * NC;
    }
    // counts of the large cells, and (levels 2) of the coarse ones; levels 1 asks the fine cells themselves
    const bool fine = coarse == 1;
    const int* scount = fine ? ccount : ccount + m3[0] * m3[1] * m3[2];
    for (int s = 0;; ++s) {
      int lo[3], e[3];  // the cube's part inside the grid
#pragma unroll
      for (int a = 0; a < 3; ++a) {
        lo[a] = max(cc[a] - s, 0);
        e[a] = min(cc[a] + s, s3[a] - 1) - lo[a] + 1;
      }
      const int cube = e[0] * e[1] * e[2];
      for (int c0 = 0; c0 < cube; c0 += 32) {
        const int c = c0 + lane, yz = c / e[0];
        const int x = lo[0] + c - yz * e[0], y = lo[1] + yz % e[1], z = lo[2] + yz / e[1];
        unsigned d = NO_CELL;
        if (c < cube && max(abs(x - cc[0]), max(abs(y - cc[1]), abs(z - cc[2]))) == s &&
            scount[(z * s3[1] + y) * s3[0] + x] != 0)
          d = box_bits(x, y, z, HS);
        for (int src; (src = nearest_lane(d)) >= 0;) {
          if (lane == src) d = NO_CELL;
          const int X = __shfl_sync(FULL, x, src) * NC, Y = __shfl_sync(FULL, y, src) * NC,
                    Z = __shfl_sync(FULL, z, src) * NC;
          static_assert(NC * NC * NC == 64, "two coarse cells a lane");
          unsigned dc[2];
#pragma unroll
          for (int r = 0; r < 2; ++r) {
            const int u = r * 32 + lane, xc = X + u % NC, yc = Y + u / NC % NC, zc = Z + u / (NC * NC);
            dc[r] = NO_CELL;
            if (xc < m3[0] && yc < m3[1] && zc < m3[2]) {
              const int c1 = (zc * m3[1] + yc) * m3[0] + xc;
              if (fine ? cell_start(g, c1 + 1) > cell_start(g, c1) : ccount[c1] != 0) dc[r] = box_bits(xc, yc, zc, H);
            }
          }
          // two coarse cells at a time, 16 lanes each: a lane per row of fine cells
          for (;;) {
            int u2[2] = {-1, -1};
#pragma unroll
            for (int t = 0; t < 2; ++t) {
              const int sc = nearest_lane(min(dc[0], dc[1]));
              if (sc < 0) break;
              u2[t] = __shfl_sync(FULL, dc[0] <= dc[1] ? lane : lane + 32, sc);
              if (lane == sc) (u2[t] < 32 ? dc[0] : dc[1]) = NO_CELL;
            }
            if (u2[0] < 0) break;
            const int u = lane < 16 ? u2[0] : u2[1], row = lane & 15;
            b = len = 0;
            if (u >= 0 && row < coarse * coarse) {
              const int xf = (X + u % NC) * coarse, yf = (Y + u / NC % NC) * coarse + row % coarse,
                        zf = (Z + u / (NC * NC)) * coarse + row / coarse;
              if (!(row_d2(xf, yf, zf) > cand_key(best))) row_range(g, n3, xf, xf + coarse - 1, yf, zf, b, len);
            }
            best = umin64(best, scan_ranges(b, len));
          }
        }
      }
      dout = outside_distance(q, sp.o, HS, cc, s3, s, sp.extent);
      if (dout == INFINITY || certified(cand_key(best), dout)) break;
    }
  }
  // an infinite or NaN key (a query whose squared distances leave float32's
  // range) is no candidate, as in the brute-force search
  if (lane == 0) {
    const bool found = cand_key(best) < INFINITY;
    if (idx_out) idx_out[t] = found ? (int32_t)(unsigned)best : INT_MAX;
    if (key_out) key_out[t] = found ? cand_key(best) : INFINITY;
  }
}

// ---- launchers --------------------------------------------------------------------

static inline unsigned up(int64_t a, int64_t b) { return (unsigned)((a + b - 1) / b); }

size_t grid_tot_entries(int64_t n) { return grid_start_entries(n) / SCAN_B + 2; }

// Means, boxes and grids of the clouds; scatter matrices and largest
// covariance eigenvalues of those that ask for them.  part: nclouds x
// CLOUD_PARTS x 6 doubles, bpart the same of floats.  most: points of the
// largest cloud.
// sorted: launch_grid_sort of the same clouds and part follows, which finishes
// the scatter matrices.
cudaError_t launch_clouds(Launch L, const CloudSet& cs, int nclouds, int most, bool scatter, bool sorted, double* part,
                          float* bpart) {
  const dim3 grid(cloud_parts(most), nclouds), one(1, nclouds);
  cloud_sums_kernel<<<grid, RED_THREADS, 0, L.stream>>>(cs, part, bpart);
  cloud_mean_kernel<<<one, RED_THREADS, 0, L.stream>>>(cs, part, bpart);
  if (L.counter) *L.counter += 2;
  if (scatter || cs.many || cs.one[0].start) {  // scatter sums, cleared cell counts
    cloud_scatter_kernel<<<grid, RED_THREADS, 0, L.stream>>>(cs, part);
    if (L.counter) *L.counter += 1;
  }
  if (scatter && !sorted) {
    cloud_lmax_kernel<<<one, RED_THREADS, 0, L.stream>>>(cs, part);
    if (L.counter) *L.counter += 1;
  }
  return cudaGetLastError();
}

// Counting sort of the clouds' points into their cells (after launch_clouds).
cudaError_t launch_grid_sort(Launch L, const CloudSet& cs, int nclouds, int most, const double* part) {
  const dim3 pts(up(most, 256), nclouds);
  const unsigned nsb = up((int64_t)grid_start_entries(most), SCAN_B);
  cell_count_kernel<<<dim3(pts.x + 1, nclouds), 256, 0, L.stream>>>(cs, part);
  scan_local_kernel<<<dim3(nsb, nclouds), SCAN_T, 0, L.stream>>>(cs);
  if (L.counter) *L.counter += 2;
  if (nsb > 1) {
    scan_blocks_kernel<<<dim3(1, nclouds), 1024, 0, L.stream>>>(cs);
    if (L.counter) *L.counter += 1;
  }
  cell_scatter_kernel<<<pts, 256, 0, L.stream>>>(cs);
  if (L.counter) *L.counter += 1;
  return cudaGetLastError();
}

// k nearest neighbours of every point of the sorted clouds.  fused: the key
// form of clouds below the brute-force limit (grid_key).
cudaError_t launch_knn_grid(Launch L, const CloudSet& cs, int nclouds, int most, int k, bool fused) {
  const dim3 grid(up(most, QUERY_WARPS), nclouds);
  if (fused) knn_query_kernel<true, QUERY_WARPS, QUERY_BLOCKS><<<grid, QUERY_WARPS * 32, 0, L.stream>>>(cs, nullptr, k);
  else knn_query_kernel<false, QUERY_WARPS, QUERY_BLOCKS><<<grid, QUERY_WARPS * 32, 0, L.stream>>>(cs, nullptr, k);
  if (L.counter) *L.counter += 1;
  return cudaGetLastError();
}

// The same for a batch's clouds (device array), in the order of a table of
// (cloud, first query).  Batches keep the key rounding they had (grid_key).
cudaError_t launch_knn_grid_table(Launch L, const GridCloud* many, const int2* table, int nblocks, int k) {
  if (nblocks <= 0) return cudaSuccess;
  CloudSet cs{};
  cs.many = many;
  knn_query_kernel<true, QUERY_TABLE_WARPS, QUERY_TABLE_BLOCKS>
      <<<nblocks, QUERY_TABLE_WARPS * 32, 0, L.stream>>>(cs, table, k);
  if (L.counter) *L.counter += 1;
  return cudaGetLastError();
}

cudaError_t launch_coarse_count(Launch L, const CloudSet& cs, int64_t n, int* ccount) {
  const unsigned b = up((int64_t)grid_start_entries(n) / 16, 256);
  coarse_count_kernel<<<b < 608 ? b : 608, 256, 0, L.stream>>>(cs, ccount);
  super_count_kernel<<<b < 152 ? b : 152, 256, 0, L.stream>>>(cs, ccount);
  if (L.counter) *L.counter += 2;
  return cudaGetLastError();
}

// Nearest point of the sorted cloud cs[0] for each of nq queries.  levels 2:
// far queries descend through cells of 16 and of 4 fine cells that hold
// points; 1: through cells of 4 and fine cells that do.
cudaError_t launch_nearest_grid(Launch L, const CloudSet& cs, int levels, const int* ccount, const float* q3, int nq,
                                int32_t* idx_out, float* key_out) {
  if (nq <= 0) return cudaSuccess;
  nearest_query_kernel<<<up(nq, NEAREST_WARPS), NEAREST_WARPS * 32, 0, L.stream>>>(
      cs, levels == 1 ? 1 : NEAREST_COARSE, ccount, q3, nq, idx_out, key_out);
  if (L.counter) *L.counter += 1;
  return cudaGetLastError();
}

}  // namespace scgr
