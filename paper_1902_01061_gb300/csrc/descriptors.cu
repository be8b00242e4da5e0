// One-time descriptor pass (Sec. III-A, Sec. IV): input packing and
// validation, k-nearest neighbours, curvature, cloud statistics of the scale
// model (Sec. III-B), sigma of Eq. 3, and the records the force kernel reads.
#include <cmath>
#include <climits>

#include "common.cuh"
#include "pointsum.cuh"

namespace scgr {

constexpr double SQRT_LOG2E = 1.2011224087864498;  // sqrt(log2 e)

static inline cudaError_t after_launch(Launch L) {
  if (L.counter) ++*L.counter;
  return cudaGetLastError();
}

// ---- pack + validate ----------------------------------------------------
__global__ void pack_kernel(const float* __restrict__ xyz, int64_t n, float4* __restrict__ out,
                            int* __restrict__ err) {
  const int64_t i = blockIdx.x * (int64_t)blockDim.x + threadIdx.x;
  if (i >= n) return;
  float x = xyz[3 * i], y = xyz[3 * i + 1], z = xyz[3 * i + 2];
  // |x| <= 1e18 keeps every squared-distance key finite in float32
  const bool ok = isfinite(x) && isfinite(y) && isfinite(z) && fabsf(x) <= 1e18f &&
                  fabsf(y) <= 1e18f && fabsf(z) <= 1e18f;
  if (!ok) {
    atomicOr(err, ERR_NONFINITE);
    x = y = z = 0.f;
  }
  out[i] = make_float4(x, y, z, 0.f);
}

cudaError_t launch_pack(Launch L, const float* xyz, int64_t n, float4* out, int* err) {
  if (n <= 0) return cudaSuccess;
  const int tpb = 256;
  pack_kernel<<<(unsigned)((n + tpb - 1) / tpb), tpb, 0, L.stream>>>(xyz, n, out, err);
  return after_launch(L);
}

// ---- brute-force kNN ----------------------------------------------------
// Each thread owns one query and keeps its KC best (key, index) pairs sorted
// in registers.  Candidates are scanned in increasing index order, so a
// candidate whose key equals the current KC-th key never displaces it: ties
// go to the lower index.  The key is the float32 value
// (dx*dx + dy*dy) + dz*dz with every operation rounded on its own
// (__fmul_rn / __fadd_rn forbid contraction into fused multiply-adds).
constexpr int KNN_TPB = 128;
constexpr int KNN_TILE = 1024;

// Insert (key, idx) into the sorted list kd/ki of KC entries if it beats the
// KC-th key; a key equal to an entry stays behind it (candidates arrive in
// increasing index order, so ties keep the lower index first).
template <int KC>
__device__ __forceinline__ void knn_insert(float key, int idx, float* kd, int* ki) {
  if (key < kd[KC - 1]) {
    kd[KC - 1] = key;
    ki[KC - 1] = idx;
#pragma unroll
    for (int m = KC - 1; m > 0; --m) {
      if (kd[m] < kd[m - 1]) {
        const float tk = kd[m];
        kd[m] = kd[m - 1];
        kd[m - 1] = tk;
        const int ti = ki[m];
        ki[m] = ki[m - 1];
        ki[m - 1] = ti;
      }
    }
  }
}

__device__ __forceinline__ float knn_key(float4 q, float4 c) {
  const float dx = __fsub_rn(q.x, c.x);
  const float dy = __fsub_rn(q.y, c.y);
  const float dz = __fsub_rn(q.z, c.z);
  return __fadd_rn(__fadd_rn(__fmul_rn(dx, dx), __fmul_rn(dy, dy)), __fmul_rn(dz, dz));
}

// Candidates that beat the KC-th key wait in a short per-thread queue; the
// warp merges all queues into the sorted lists together once any queue could
// overflow.  Inserting at once costs a 16-step pass for the whole warp
// whenever a single lane improves; queueing lets the lanes share that cost.
// The merge applies the exact test against the live list in candidate
// order, so the result is the same as inserting at once.  Four candidates
// are keyed per step with packed .f32x2 arithmetic (the same per-operation
// rounding as the scalar key), and the warp skips the queue code unless one
// of its lanes has a hit among them.
constexpr int KNN_QL = 8;  // queue capacity
constexpr int KNN_U = 4;   // candidates per step (KNN_TILE is a multiple)

__device__ __forceinline__ u64 knn_key2(u64 qx, u64 qy, u64 qz, u64 cx, u64 cy, u64 cz) {
  const u64 dx = sub2(qx, cx), dy = sub2(qy, cy), dz = sub2(qz, cz);
  return add2(add2(mul2(dx, dx), mul2(dy, dy)), mul2(dz, dz));
}

// Scan candidates P[base .. base + n) in index order for one query q held by
// this thread; tile staging is shared by the block (all threads of the block
// must call this with the same base and n, so the warp votes are uniform).
// The tile is stored as three coordinate arrays.  Indices written are global.
template <int KC>
__device__ __forceinline__ void knn_scan(const float4* __restrict__ P, int64_t base, int n, float4 q, float* kd,
                                         int* ki, float* tile, float* qks, int* qis) {
  float* tx = tile;
  float* ty = tile + KNN_TILE;
  float* tz = tile + 2 * KNN_TILE;
#pragma unroll
  for (int m = 0; m < KC; ++m) {
    kd[m] = INFINITY;
    ki[m] = INT_MAX;
  }
  // this thread's queue: slot s at [s * KNN_TPB + threadIdx.x] (conflict-free)
  float* qk = qks + threadIdx.x;
  int* qi = qis + threadIdx.x;
  int qn = 0;
  float thr = INFINITY;
  const u64 qx = pk2(q.x, q.x), qy = pk2(q.y, q.y), qz = pk2(q.z, q.z);
  for (int t0 = 0; t0 < n; t0 += KNN_TILE) {
    const int cnt = min(KNN_TILE, n - t0);
    __syncthreads();
    for (int t = threadIdx.x; t < cnt; t += KNN_TPB) {
      const float4 c = P[base + t0 + t];
      tx[t] = c.x;
      ty[t] = c.y;
      tz[t] = c.z;
    }
    __syncthreads();
    const int idx0 = (int)(base + t0);
    int jj = 0;
    if (KC == 1) {
      for (; jj < cnt; ++jj) knn_insert<KC>(knn_key(q, make_float4(tx[jj], ty[jj], tz[jj], 0.f)), idx0 + jj, kd, ki);
      continue;
    }
    for (; jj + KNN_U <= cnt; jj += KNN_U) {
      const ulonglong2 X = *reinterpret_cast<const ulonglong2*>(tx + jj);
      const ulonglong2 Y = *reinterpret_cast<const ulonglong2*>(ty + jj);
      const ulonglong2 Z = *reinterpret_cast<const ulonglong2*>(tz + jj);
      float key[KNN_U];
      upk2(knn_key2(qx, qy, qz, X.x, Y.x, Z.x), key[0], key[1]);
      upk2(knn_key2(qx, qy, qz, X.y, Y.y, Z.y), key[2], key[3]);
      const bool hit = (key[0] < thr) | (key[1] < thr) | (key[2] < thr) | (key[3] < thr);
      if (__any_sync(0xffffffffu, hit)) {
#pragma unroll
        for (int u = 0; u < KNN_U; ++u) {
          if (key[u] < thr) {
            qk[qn * KNN_TPB] = key[u];
            qi[qn * KNN_TPB] = idx0 + jj + u;
            ++qn;
          }
        }
        if (__any_sync(0xffffffffu, qn > KNN_QL - KNN_U)) {
          for (int sl = 0; sl < qn; ++sl) knn_insert<KC>(qk[sl * KNN_TPB], qi[sl * KNN_TPB], kd, ki);
          qn = 0;
          thr = kd[KC - 1];
        }
      }
    }
    if (jj < cnt) {  // ragged end of the last tile: empty the queue, then insert directly
      for (int sl = 0; sl < qn; ++sl) knn_insert<KC>(qk[sl * KNN_TPB], qi[sl * KNN_TPB], kd, ki);
      qn = 0;
      for (; jj < cnt; ++jj) knn_insert<KC>(knn_key(q, make_float4(tx[jj], ty[jj], tz[jj], 0.f)), idx0 + jj, kd, ki);
      thr = kd[KC - 1];
    }
  }
  for (int sl = 0; sl < qn; ++sl) knn_insert<KC>(qk[sl * KNN_TPB], qi[sl * KNN_TPB], kd, ki);
}

template <int KC>
__global__ void __launch_bounds__(KNN_TPB, KC > 16 ? 2 : 4) knn_brute_kernel(const float4* __restrict__ P, int n,
                                                            int k, int32_t* __restrict__ out) {
  __shared__ __align__(16) float tile[3 * KNN_TILE];
  __shared__ float qks[KNN_QL * KNN_TPB];
  __shared__ int qis[KNN_QL * KNN_TPB];
  const int qi = blockIdx.x * KNN_TPB + threadIdx.x;
  const float4 q = P[qi < n ? qi : n - 1];
  float kd[KC];
  int ki[KC];
  knn_scan<KC>(P, 0, n, q, kd, ki, tile, qks, qis);
  if (qi < n) {
#pragma unroll
    for (int m = 0; m < KC; ++m)
      if (m < k) out[(int64_t)qi * k + m] = ki[m];
  }
}

// Nearest reference point of arbitrary query points (change detection):
// the same exact key and (key, index) order as the kNN, k = 1.
__global__ void __launch_bounds__(KNN_TPB) nearest_kernel(const float4* __restrict__ P, int n,
                                                          const float* __restrict__ q3, int nq,
                                                          int32_t* __restrict__ idx_out, float* __restrict__ key_out) {
  __shared__ __align__(16) float tile[3 * KNN_TILE];
  const int qi = blockIdx.x * KNN_TPB + threadIdx.x;
  const int qc = qi < nq ? qi : nq - 1;
  const float4 q = make_float4(q3[3 * (size_t)qc], q3[3 * (size_t)qc + 1], q3[3 * (size_t)qc + 2], 0.f);
  float kd[1];
  int ki[1];
  knn_scan<1>(P, 0, n, q, kd, ki, tile, nullptr, nullptr);
  if (qi < nq) {
    if (idx_out) idx_out[qi] = ki[0];
    if (key_out) key_out[qi] = kd[0];
  }
}

cudaError_t launch_nearest(Launch L, const float4* P, int n, const float* q3, int nq, int32_t* idx_out,
                           float* key_out) {
  if (nq <= 0) return cudaSuccess;
  nearest_kernel<<<(nq + KNN_TPB - 1) / KNN_TPB, KNN_TPB, 0, L.stream>>>(P, n, q3, nq, idx_out, key_out);
  return after_launch(L);
}

__global__ void threshold_kernel(const float* __restrict__ key, int nq, float thr2, uint8_t* __restrict__ mask,
                                 float* __restrict__ dist) {
  const int i = blockIdx.x * blockDim.x + threadIdx.x;
  if (i >= nq) return;
  const float k = key[i];
  mask[i] = k > thr2 ? 1 : 0;
  if (dist) dist[i] = sqrtf(k);
}

cudaError_t launch_threshold(Launch L, const float* key, int nq, float thr2, uint8_t* mask, float* dist) {
  if (nq <= 0) return cudaSuccess;
  threshold_kernel<<<(nq + 255) / 256, 256, 0, L.stream>>>(key, nq, thr2, mask, dist);
  return after_launch(L);
}

cudaError_t launch_knn(Launch L, const float4* P, int n, int k, int32_t* out) {
  const unsigned grid = (unsigned)((n + KNN_TPB - 1) / KNN_TPB);
  if (k <= 8) knn_brute_kernel<8><<<grid, KNN_TPB, 0, L.stream>>>(P, n, k, out);
  else if (k <= 16) knn_brute_kernel<16><<<grid, KNN_TPB, 0, L.stream>>>(P, n, k, out);
  else knn_brute_kernel<32><<<grid, KNN_TPB, 0, L.stream>>>(P, n, k, out);
  return after_launch(L);
}

constexpr int CURV_TPB = 128;  // points per block of the curvature kernels

// ---- sigma of Eq. 3 ----------------------------------------------------------
// The population std of the reference curvatures from per-block sums and
// squared deviations about the block's own mean (sigma_part), merged in a fixed
// order: M2 = sum_b [M2_b + n_b (mean_b - mean)^2], as accurate as a second pass
// over the points without reading them again.
__device__ __forceinline__ void sigma_part(double a, bool live, int n_block, double* __restrict__ part) {
  __shared__ double sh[2][CURV_TPB / 32];
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
  double v = live ? a : 0.0;
#pragma unroll
  for (int off = 16; off > 0; off >>= 1) v += __shfl_xor_sync(0xffffffffu, v, off);
  if (lane == 0) sh[0][warp] = v;
  __syncthreads();
  double sum = sh[0][0];
#pragma unroll
  for (int w = 1; w < CURV_TPB / 32; ++w) sum += sh[0][w];
  const double d = live ? a - sum / (double)n_block : 0.0;
  v = d * d;
#pragma unroll
  for (int off = 16; off > 0; off >>= 1) v += __shfl_xor_sync(0xffffffffu, v, off);
  if (lane == 0) sh[1][warp] = v;
  __syncthreads();
  if (threadIdx.x == 0) {
    double m2 = sh[1][0];
#pragma unroll
    for (int w = 1; w < CURV_TPB / 32; ++w) m2 += sh[1][w];
    part[2 * (size_t)blockIdx.x] = sum;
    part[2 * (size_t)blockIdx.x + 1] = m2;
  }
}

__global__ void __launch_bounds__(CURV_TPB) sigma_parts_kernel(const double* __restrict__ a64, int n,
                                                              double* __restrict__ part) {
  const int i = blockIdx.x * CURV_TPB + threadIdx.x;
  sigma_part(i < n ? a64[i] : 0.0, i < n, min(CURV_TPB, n - (int)blockIdx.x * CURV_TPB), part);
}

// sigma (the caller's, or the std, 1 below 1e-12, times sigma_scale) and the
// factor sqrt(log2 e) / sigma that the force records use.
__device__ __forceinline__ void finish_sigma(double sum_a, double sum_d2, int64_t n, double sigma_user,
                                             double sigma_scale, DevStats* st) {
  st->asum[0] = sum_a;
  double sigma = sigma_user;
  if (!(sigma > 0.0)) {
    const double sd = sqrt(sum_d2 / (double)n);
    sigma = sd >= 1e-12 ? sd : 1.0;
    if (sigma_scale != 1.0) sigma *= sigma_scale;
  }
  st->sigma = sigma;
  st->kscale = SQRT_LOG2E / sigma;
}

constexpr int SIGMA_T = 256;

__device__ __forceinline__ double sigma_block_sum(double v, double* sh) {
#pragma unroll
  for (int off = 16; off > 0; off >>= 1) v += __shfl_xor_sync(0xffffffffu, v, off);
  if ((threadIdx.x & 31) == 0) sh[threadIdx.x >> 5] = v;
  __syncthreads();
  v = sh[0];
#pragma unroll
  for (int w = 1; w < SIGMA_T / 32; ++w) v += sh[w];
  __syncthreads();
  return v;
}

__global__ void __launch_bounds__(SIGMA_T) sigma_finish_kernel(const double* __restrict__ part, int n,
                                                              double sigma_user, double sigma_scale, DevStats* st) {
  __shared__ double sh[SIGMA_T / 32];
  const int nb = (n + CURV_TPB - 1) / CURV_TPB;
  double v = 0.0;
  for (int b = threadIdx.x; b < nb; b += SIGMA_T) v += part[2 * (size_t)b];
  const double sum = sigma_block_sum(v, sh), mean = sum / (double)n;
  v = 0.0;
  for (int b = threadIdx.x; b < nb; b += SIGMA_T) {
    const double nbk = (double)min(CURV_TPB, n - b * CURV_TPB);
    const double d = part[2 * (size_t)b] - nbk * mean;  // n_b (mean_b - mean)
    v += fma(d * d, b < nb - 1 ? 1.0 / CURV_TPB : 1.0 / nbk, part[2 * (size_t)b + 1]);
  }
  const double d2 = sigma_block_sum(v, sh);
  if (threadIdx.x == 0) finish_sigma(sum, d2, n, sigma_user, sigma_scale, st);
}

size_t sigma_part_bytes(int64_t n) { return (size_t)((n + CURV_TPB - 1) / CURV_TPB) * 2 * sizeof(double); }

// From the parts that the curvature kernels wrote.
cudaError_t launch_sigma_finish(Launch L, const double* part, int n, double sigma_user, double sigma_scale,
                                DevStats* st) {
  sigma_finish_kernel<<<1, SIGMA_T, 0, L.stream>>>(part, n, sigma_user, sigma_scale, st);
  return after_launch(L);
}

// From curvatures of any origin.
cudaError_t launch_sigma(Launch L, const double* a64, int n, double sigma_user, double sigma_scale, double* part,
                         DevStats* st) {
  sigma_parts_kernel<<<(n + CURV_TPB - 1) / CURV_TPB, CURV_TPB, 0, L.stream>>>(a64, n, part);
  if (L.counter) ++*L.counter;
  return launch_sigma_finish(L, part, n, sigma_user, sigma_scale, st);
}

// (h, l) += x, h the rounded sum (two-sum)
__device__ __forceinline__ void two_sum_add(float& h, float& l, float x) {
  const float t = __fadd_rn(h, x);
  const float bv = __fsub_rn(t, h);
  l = __fadd_rn(l, __fadd_rn(__fsub_rn(h, __fsub_rn(t, bv)), __fsub_rn(x, bv)));
  h = t;
}

// ---- curvature ----------------------------------------------------------
// a = lambda_min / (lambda_1 + lambda_2 + lambda_3) of the 1/k covariance of
// the k neighbours; lambda_min clamped at 0; 0 for a zero trace.
//
// The offsets from the point itself are exact float pairs (two-difference),
// their sums and products float pairs too (two-sum, fma remainder); only the
// covariance, its polynomial and the last Newton steps are float64.  The pairs
// leave an error in a of 2^-50 to 2^-48 rms (k = 8 to 32; emulated on patches
// of random orientation), so a point flatter than CURV_FLAT, where that would
// show in a float32 result, has its covariance formed again in float64 about
// the neighbours' mean, and so has one whose offsets' squares leave float32's
// comfortable range.  (A smooth surface of 1M points, k = 16, has a about 3e-7;
// none of its points is that flat.)
// Bound: float64 issue (about 80 such instructions a point, each 64 cycles of
// a warp scheduler on GB300) and the gather of the neighbours.
constexpr double CURV_FLAT = 0x1p-26;

__device__ __noinline__ void covariance_float64(const float4* __restrict__ P, const int32_t* __restrict__ nb, int k,
                                                double* C) {
  double mx = 0, my = 0, mz = 0;
  for (int m = 0; m < k; ++m) {
    const float4 c = P[nb[m]];
    mx += c.x;
    my += c.y;
    mz += c.z;
  }
  mx /= k;
  my /= k;
  mz /= k;
  for (int q = 0; q < 9; ++q) C[q] = 0.0;
  for (int m = 0; m < k; ++m) {
    const float4 c = P[nb[m]];
    const double dx = c.x - mx, dy = c.y - my, dz = c.z - mz;
    C[0] += dx * dx; C[1] += dx * dy; C[2] += dx * dz;
    C[4] += dy * dy; C[5] += dy * dz; C[8] += dz * dz;
  }
  C[0] /= k; C[1] /= k; C[2] /= k; C[4] /= k; C[5] /= k; C[8] /= k;
  C[3] = C[1]; C[6] = C[2]; C[7] = C[5];
}

__device__ __forceinline__ double surface_variation(const double* C) {
  const double tr = C[0] + C[4] + C[8];
  return tr > 0.0 ? fmax(sym3_extreme_eigenvalue(C, false), 0.0) / tr : 0.0;
}

__device__ __forceinline__ double point_curvature(const float4* __restrict__ P, const int32_t* __restrict__ nb, int k,
                                                  int i) {
  const float4 q = P[i];
  const float qv[3] = {q.x, q.y, q.z};
  float sh[3] = {0.f, 0.f, 0.f}, sl[3] = {0.f, 0.f, 0.f};
  float ph[6] = {0.f, 0.f, 0.f, 0.f, 0.f, 0.f}, pl[6] = {0.f, 0.f, 0.f, 0.f, 0.f, 0.f};  // xx xy xz yy yz zz
#pragma unroll 4
  for (int m = 0; m < k; ++m) {
    const float4 c = P[nb[m]];
    const float cv[3] = {c.x, c.y, c.z};
    float h[3], l[3];
#pragma unroll
    for (int a = 0; a < 3; ++a) {
      h[a] = __fsub_rn(cv[a], qv[a]);
      const float bv = __fsub_rn(h[a], cv[a]);
      l[a] = __fsub_rn(__fsub_rn(cv[a], __fsub_rn(h[a], bv)), __fadd_rn(qv[a], bv));
      two_sum_add(sh[a], sl[a], h[a]);
      sl[a] = __fadd_rn(sl[a], l[a]);
    }
#pragma unroll
    for (int a = 0, f = 0; a < 3; ++a)
#pragma unroll
      for (int b = a; b < 3; ++b, ++f) {
        const float p = __fmul_rn(h[a], h[b]);
        const float r = __fmaf_rn(h[a], l[b], __fmaf_rn(l[a], h[b], __fmaf_rn(h[a], h[b], -p)));
        two_sum_add(ph[f], pl[f], p);
        pl[f] = __fadd_rn(pl[f], r);
      }
  }
  double C[9], a = 0.0;
  const float tr = ph[0] + ph[3] + ph[5];
  bool again = !(tr > 1e-18f && tr < 1e30f);
  if (!again) {
    const double ik = 1.0 / (double)k;
    double mu[3];
#pragma unroll
    for (int d = 0; d < 3; ++d) mu[d] = ((double)sh[d] + (double)sl[d]) * ik;
#pragma unroll
    for (int d = 0, f = 0; d < 3; ++d)
#pragma unroll
      for (int b = d; b < 3; ++b, ++f)
        C[d * 3 + b] = C[b * 3 + d] = fma((double)ph[f] + (double)pl[f], ik, -mu[d] * mu[b]);
    a = surface_variation(C);
    again = a < CURV_FLAT;
  }
  if (again) {
    covariance_float64(P, nb, k, C);
    a = surface_variation(C);
  }
  return a;
}

struct CurvatureIn {
  const float4* P;
  const int32_t* nbr;
  int n;
  double* a64;
  float* a32;
  double* part;  // sigma_part's output (NULL: not wanted)
};

// Both clouds of a registration in one launch (blockIdx.y).
__global__ void __launch_bounds__(CURV_TPB) curvature_kernel(const CurvatureIn c0, const CurvatureIn c1, int k) {
  const CurvatureIn& c = blockIdx.y == 0 ? c0 : c1;
  const int i = blockIdx.x * CURV_TPB + threadIdx.x;
  if ((int)blockIdx.x * CURV_TPB >= c.n) return;
  double a = 0.0;
  if (i < c.n) {
    a = point_curvature(c.P, c.nbr + (int64_t)i * k, k, i);
    c.a64[i] = a;
    c.a32[i] = (float)a;
  }
  if (c.part) sigma_part(a, i < c.n, min(CURV_TPB, c.n - (int)blockIdx.x * CURV_TPB), c.part);
}

cudaError_t launch_curvature2(Launch L, const float4* X, const int32_t* nx, int n, double* ax64, float* ax32,
                              double* xpart, const float4* Y, const int32_t* ny, int m, double* ay64, float* ay32,
                              int k) {
  const int most = n > m ? n : m;
  curvature_kernel<<<dim3((most + CURV_TPB - 1) / CURV_TPB, Y ? 2 : 1), CURV_TPB, 0, L.stream>>>(
      CurvatureIn{X, nx, n, ax64, ax32, xpart}, CurvatureIn{Y, ny, m, ay64, ay32, nullptr}, k);
  return after_launch(L);
}

// ---- radius neighbourhood curvature (Sec. IV) ----------------------------
// The neighbourhood of p is every point q of the cloud (p included) whose
// float32 key (dx*dx + dy*dy) + dz*dz, each operation rounded on its own,
// is <= float32(scale^2 * e), e the largest eigenvalue of the cloud's 1/n
// covariance (radius sqrt(e), Sec. IV).  Its 1/|N| covariance gives
// a = lambda_min / trace.
//
// One pass over the cloud sums the count, the members' offsets and the products
// of the offsets, so accurately that the covariance S2/k - m m^T keeps a small
// eigenvalue.  A float32 difference of two coordinates may round, so each
// coordinate is split exactly, x = xh + xl with xh a multiple of u = 2^-21 r (r
// up to a power of two, the bound on |d|): differences h of the xh are exact, and the
// covariance of the offsets h + xl is that of the points (they differ from q - p by
// the constant xl of p).  A sum is a pair (acc, lo): acc starts at c = 1.5 * 2^k, 2^k
// above twice what a run of 32 points can add, so t = fma(x, y, acc) stays in
// acc's binade, acc - t is exact, and so is acc's sum of such steps; lo collects
// fma(x, y, acc - t), the exact rest rounded once, and the products with xl.  lo is a
// plain float32 sum over a tile's lane (128 points): its rounding is the error, some
// 2^-42 of the bound B on |d|^2 per point; a float pair (two-sum) carries the totals.
//
// That error is relative to B, not to the neighbourhood, so where the smallest
// eigenvalue is below 2^-17 B (few, tight or very flat neighbours) the point's
// covariance is summed again in float64 by its warp (none of 20,011 sampled
// surface points at scale 1, at most 1 in 500 at scale 0.5 and 500 points; an
// exact plane: all).  Above it the relative error of the eigenvalue is at most about 2^-25
// (emulated: 20 to 1,500 members, 3e-8 at 2^-17 B, 5e-10 at 1e-3 B; with offsets rounded to
// float32 4e-6 and 7e-7).
//
// Bound: the FP32 pipe.  A pair costs 8 lane operations for the key, 4 for
// the offsets and the count, 36 for the nine sums and 15 for the xl terms:
// 2.0 pairs per clock per SM; a group of four points that no query of the
// warp reaches costs only the keys.  Large clouds come in Morton order
// (order.cu): a warp's queries and a run of 32 points are then compact, and a
// run whose box lies beyond the radius of the warp's box costs nothing.
// (20,011 + 17,611 points, scale 1, the whole descriptor pass: 30.2 ms with
// two passes of 12 float64 operations per member; 1.87 ms in index order, 0.66 ms
// in Morton order; 0.58 ms with offsets rounded to float32.)
//
// Members' offsets are scaled by a power of two that brings the bound on
// |d|^2 (the smaller of the squared radius and three squared box extents)
// near 1, so that no product overflows or underflows.
constexpr int RAD_TPB = 128;
constexpr int RAD_TILE = 256;
constexpr int RAD_RUN = 32;
constexpr int RAD_NS = 10;  // count, d (3), d d^T (6: xx xy xz yy yz zz)
constexpr float RAD_FLAT = 0x1p-17f;  // smallest eigenvalue / B below which the sums are repeated in float64

struct RadiusScale {
  float s;         // power of two applied to the offsets
  float r2;        // squared radius (not scaled)
  float B;         // bound on |d|^2, scaled
  float c1, c2;    // acc's starting value for the offsets and for their products
  float cu, small; // 1.5 * 2^23 u; coordinates below `small` are split, larger ones are multiples of u / 2
};
__device__ __forceinline__ RadiusScale radius_scale_of(const double* e_dev, double scale2, const GridSpec* spec) {
  const float r2 = (float)(scale2 * e_dev[0]);
  const float diag2 = 3.0003f * spec->extent * spec->extent;  // at least the box's squared diagonal
  const float B = fmaxf(fminf(r2, diag2), 1e-36f);
  const int h = min(60, max(-60, -(ilogbf(B) >> 1)));
  RadiusScale o;
  o.s = ldexpf(1.f, h);
  o.r2 = r2;
  const float Bs = (B * o.s) * o.s;
  o.B = Bs;
  const int e = (ilogbf(B) >> 1) + 1;  // r < 2^e
  o.cu = ldexpf(1.5f, e + 2);
  o.small = ldexpf(1.f, e + 1);
  // Bs < 2^(ilogb + 1), sqrt(Bs) < 2^((ilogb >> 1) + 1): 2^(k - 1) >= the
  // RAD_RUN / 2 = 16 terms of a lane
  o.c2 = 1.5f * ldexpf(1.f, ilogbf(Bs) + 6);
  o.c1 = 1.5f * ldexpf(1.f, (ilogbf(Bs) >> 1) + 6);
  return o;
}

// The multiple of u next to x (x itself where it is a multiple of u / 2): x - high is
// exact, and the difference of two within r of each other fits 23 bits.
__device__ __forceinline__ float radius_high(float x, const RadiusScale& sc) {
  return fabsf(x) < sc.small ? __fsub_rn(__fadd_rn(x, sc.cu), sc.cu) : x;
}

// (acc, lo) += x y in both lanes
__device__ __forceinline__ void split_fma2(u64& acc, u64& lo, u64 x, u64 y) {
  const u64 t = fma2(x, y, acc);
  lo = add2(lo, fma2(x, y, sub2(acc, t)));
  acc = t;
}
__device__ __forceinline__ void split_add2(u64& acc, u64& lo, u64 x) {
  const u64 t = add2(acc, x);
  lo = add2(lo, sub2(x, sub2(t, acc)));
  acc = t;
}
__device__ __forceinline__ float member_mask(float key, float r2) {
  float m;
  asm("set.le.f32.f32 %0, %1, %2;" : "=f"(m) : "f"(key), "f"(r2));
  return m;
}

// Covariance of points from their count, sum and sum of products.
__device__ __forceinline__ void covariance_of_sums(const double (&v)[RAD_NS], double* C) {
  const double ik = 1.0 / v[0];
  const double mx = v[1] * ik, my = v[2] * ik, mz = v[3] * ik;
  C[0] = fma(v[4], ik, -mx * mx); C[1] = fma(v[5], ik, -mx * my); C[2] = fma(v[6], ik, -mx * mz);
  C[4] = fma(v[7], ik, -my * my); C[5] = fma(v[8], ik, -my * mz); C[8] = fma(v[9], ik, -mz * mz);
  C[3] = C[1]; C[6] = C[2]; C[7] = C[5];
}

// Query i's sums over the points of tiles [t0, t1) of split blockIdx.y, written
// as doubles to part[split][sum][n] (in scaled coordinates).
__global__ void __launch_bounds__(RAD_TPB, 5)
    radius_sums_kernel(const float4* __restrict__ P, int n, const float* __restrict__ box,
                       const double* __restrict__ e_dev, double scale2, const GridSpec* __restrict__ spec,
                       int tiles_per_split, double* __restrict__ part) {
  __shared__ __align__(16) float tile[9][RAD_TILE];  // x, y, z; their high parts, scaled; their low parts, scaled
  const int i = blockIdx.x * RAD_TPB + threadIdx.x;
  const RadiusScale sc = radius_scale_of(e_dev, scale2, spec);
  const float4 q4 = P[i < n ? i : n - 1];
  const u64 q2x = pk2(q4.x, q4.x), q2y = pk2(q4.y, q4.y), q2z = pk2(q4.z, q4.z);
  const float hx = radius_high(q4.x, sc) * sc.s, hy = radius_high(q4.y, sc) * sc.s, hz = radius_high(q4.z, sc) * sc.s;
  const u64 h2x = pk2(hx, hx), h2y = pk2(hy, hy), h2z = pk2(hz, hz);
  float H[RAD_NS], Lo[RAD_NS];
#pragma unroll
  for (int f = 0; f < RAD_NS; ++f) H[f] = Lo[f] = 0.f;
  const int lane = threadIdx.x & 31;
  float qb[6] = {q4.x, q4.y, q4.z, -q4.x, -q4.y, -q4.z};  // the warp's box: min, -max
  if (box) {
#pragma unroll
    for (int off = 16; off > 0; off >>= 1)
#pragma unroll
      for (int f = 0; f < 6; ++f) qb[f] = fminf(qb[f], __shfl_xor_sync(0xffffffffu, qb[f], off));
  }
  const int t0 = blockIdx.y * tiles_per_split * RAD_TILE;
  const int t1 = min(n, t0 + tiles_per_split * RAD_TILE);
  for (int base = t0; base < t1; base += RAD_TILE) {
    // the runs of the tile that a query of the warp may reach
    unsigned todo = (1u << (RAD_TILE / RAD_RUN)) - 1;
    if (box) {
      bool reach = false;
      if (lane < RAD_TILE / RAD_RUN && base + lane * RAD_RUN < t1) {
        const float* b = box + 6 * (size_t)(base / RAD_RUN + lane);
        float d2 = 0.f;
#pragma unroll
        for (int f = 0; f < 3; ++f) {
          const float g = fmaxf(0.f, fmaxf(b[f] + qb[f + 3], qb[f] + b[f + 3]));
          d2 = fmaf(g, g, d2);
        }
        reach = !(d2 * (1.f - 1e-5f) > sc.r2);
      }
      todo = __ballot_sync(0xffffffffu, reach);
    }
    if (!__syncthreads_or((int)todo)) continue;
#pragma unroll
    for (int t = threadIdx.x; t < RAD_TILE; t += RAD_TPB) {
      // past the end: a point at NaN, whose key is never <= r2
      const float4 c = base + t < t1 ? P[base + t] : make_float4(NAN, NAN, NAN, 0.f);
      const float cv[3] = {c.x, c.y, c.z};
#pragma unroll
      for (int a = 0; a < 3; ++a) {
        const float high = base + t < t1 ? radius_high(cv[a], sc) : 0.f;
        tile[a][t] = cv[a];
        tile[3 + a][t] = high * sc.s;
        tile[6 + a][t] = base + t < t1 ? __fsub_rn(cv[a], high) * sc.s : 0.f;
      }
    }
    __syncthreads();
    u64 acc[RAD_NS], lo[RAD_NS];
    acc[0] = 0ull;
#pragma unroll
    for (int f = 1; f < RAD_NS; ++f) lo[f] = 0ull;
#pragma unroll 1
    for (; todo; todo &= todo - 1) {
      const int run = (__ffs(todo) - 1) * RAD_RUN;
#pragma unroll
      for (int f = 1; f < RAD_NS; ++f) acc[f] = f < 4 ? pk2(sc.c1, sc.c1) : pk2(sc.c2, sc.c2);
#pragma unroll 1
      for (int j = run; j < run + RAD_RUN; j += 4) {
        const ulonglong2 X = *reinterpret_cast<const ulonglong2*>(&tile[0][j]);
        const ulonglong2 Y = *reinterpret_cast<const ulonglong2*>(&tile[1][j]);
        const ulonglong2 Z = *reinterpret_cast<const ulonglong2*>(&tile[2][j]);
        u64 d[2][3], m[2];
        d[0][0] = sub2(X.x, q2x); d[0][1] = sub2(Y.x, q2y); d[0][2] = sub2(Z.x, q2z);
        d[1][0] = sub2(X.y, q2x); d[1][1] = sub2(Y.y, q2y); d[1][2] = sub2(Z.y, q2z);
        bool any = false;
#pragma unroll
        for (int h = 0; h < 2; ++h) {
          // packed products, scalar sums: ptxas fuses a packed add with the
          // packed product it adds, which would round the key once less
          float x0, x1, y0, y1, z0, z1;
          upk2(mul2(d[h][0], d[h][0]), x0, x1);
          upk2(mul2(d[h][1], d[h][1]), y0, y1);
          upk2(mul2(d[h][2], d[h][2]), z0, z1);
          const float k0 = __fadd_rn(__fadd_rn(x0, y0), z0), k1 = __fadd_rn(__fadd_rn(x1, y1), z1);
          any |= (k0 <= sc.r2) | (k1 <= sc.r2);
          m[h] = pk2(member_mask(k0, sc.r2), member_mask(k1, sc.r2));
        }
        if (!__any_sync(0xffffffffu, any)) continue;
#pragma unroll
        for (int h = 0; h < 2; ++h) {
          // of others than members the high parts' offsets are 0 and the low parts count 0 times
          auto offset = [&](int a, u64 q2) {
            float m0, m1, v0, v1;
            upk2(m[h], m0, m1);
            upk2(sub2(*reinterpret_cast<const u64*>(&tile[3 + a][j + 2 * h]), q2), v0, v1);
            return pk2(m0 != 0.f ? v0 : 0.f, m1 != 0.f ? v1 : 0.f);
          };
          const u64 x = offset(0, h2x), y = offset(1, h2y), z = offset(2, h2z);
          const u64 xl = *reinterpret_cast<const u64*>(&tile[6][j + 2 * h]);
          const u64 yl = *reinterpret_cast<const u64*>(&tile[7][j + 2 * h]);
          const u64 zl = *reinterpret_cast<const u64*>(&tile[8][j + 2 * h]);
          acc[0] = add2(acc[0], m[h]);
          split_add2(acc[1], lo[1], x);
          split_add2(acc[2], lo[2], y);
          split_add2(acc[3], lo[3], z);
          lo[1] = fma2(m[h], xl, lo[1]);
          lo[2] = fma2(m[h], yl, lo[2]);
          lo[3] = fma2(m[h], zl, lo[3]);
          split_fma2(acc[4], lo[4], x, x);
          split_fma2(acc[5], lo[5], x, y);
          split_fma2(acc[6], lo[6], x, z);
          split_fma2(acc[7], lo[7], y, y);
          split_fma2(acc[8], lo[8], y, z);
          split_fma2(acc[9], lo[9], z, z);
          lo[4] = fma2(x, add2(xl, xl), lo[4]);
          lo[5] = fma2(x, yl, fma2(y, xl, lo[5]));
          lo[6] = fma2(x, zl, fma2(z, xl, lo[6]));
          lo[7] = fma2(y, add2(yl, yl), lo[7]);
          lo[8] = fma2(y, zl, fma2(z, yl, lo[8]));
          lo[9] = fma2(z, add2(zl, zl), lo[9]);
        }
      }
#pragma unroll
      for (int f = 1; f < RAD_NS; ++f) {
        const float c = f < 4 ? sc.c1 : sc.c2;
        float a0, a1;
        upk2(acc[f], a0, a1);
        two_sum_add(H[f], Lo[f], (a0 - c) + (a1 - c));  // exact: multiples of acc's last place
      }
    }
    float b0, b1;
    upk2(acc[0], b0, b1);
    two_sum_add(H[0], Lo[0], b0 + b1);
#pragma unroll
    for (int f = 1; f < RAD_NS; ++f) {
      upk2(lo[f], b0, b1);
      two_sum_add(H[f], Lo[f], b0 + b1);
    }
  }
  if (i >= n) return;
#pragma unroll
  for (int f = 0; f < RAD_NS; ++f) part[((size_t)blockIdx.y * RAD_NS + f) * n + i] = (double)H[f] + (double)Lo[f];
}

// Point i's count, sums of offsets and of their products in float64, by one warp
// (all lanes call it; lane 2 f gets sum f).
__device__ __noinline__ double radius_sums_float64(const float4* __restrict__ P, int n, const float* __restrict__ box,
                                                   float r2, int i) {
  const int lane = threadIdx.x & 31;
  const float4 q = P[i];
  double v[16];
#pragma unroll
  for (int f = 0; f < 16; ++f) v[f] = 0.0;
  auto add = [&](const float4 c) {
    if (!(knn_key(c, q) <= r2)) return;
    const double x = (double)c.x - q.x, y = (double)c.y - q.y, z = (double)c.z - q.z;
    v[0] += 1.0; v[1] += x; v[2] += y; v[3] += z;
    v[4] = fma(x, x, v[4]); v[5] = fma(x, y, v[5]); v[6] = fma(x, z, v[6]);
    v[7] = fma(y, y, v[7]); v[8] = fma(y, z, v[8]); v[9] = fma(z, z, v[9]);
  };
  if (!box) {
    for (int j0 = lane; j0 < n; j0 += 32 * 8) {  // eight loads in flight
      float4 c[8];
#pragma unroll
      for (int u = 0; u < 8; ++u) c[u] = j0 + 32 * u < n ? P[j0 + 32 * u] : make_float4(NAN, NAN, NAN, 0.f);
#pragma unroll
      for (int u = 0; u < 8; ++u) add(c[u]);
    }
  }
  const int runs = box ? (n + RAD_RUN - 1) / RAD_RUN : 0;
  for (int b0 = 0; b0 < runs; b0 += 32) {
    // the runs of 32 points that the point may reach, a lane each
    bool reach = b0 + lane < runs;
    if (reach) {
      const float* b = box + 6 * (size_t)(b0 + lane);
      const float gx = fmaxf(0.f, fmaxf(b[0] - q.x, q.x + b[3])), gy = fmaxf(0.f, fmaxf(b[1] - q.y, q.y + b[4])),
                  gz = fmaxf(0.f, fmaxf(b[2] - q.z, q.z + b[5]));
      reach = !(fmaf(gz, gz, fmaf(gy, gy, gx * gx)) * (1.f - 1e-5f) > r2);
    }
    for (unsigned todo = __ballot_sync(0xffffffffu, reach); todo; todo &= todo - 1) {
      const int j = (b0 + __ffs(todo) - 1) * RAD_RUN + lane;
      if (j < n) add(P[j]);
    }
  }
  __syncwarp();
  warp_reduce16(v);
  return v[0];
}

// The splits' sums of a point added in order, its covariance (a power-of-two
// scaling leaves a = lambda_min / trace unchanged) and its curvature; in
// float64 from the points where the sums do not resolve it (RAD_FLAT).
__global__ void __launch_bounds__(CURV_TPB)
    radius_curvature_kernel(const double* __restrict__ part, int S, int n, const float4* __restrict__ P,
                            const float* __restrict__ box, const double* __restrict__ e_dev, double scale2,
                            const GridSpec* __restrict__ spec, double* __restrict__ a64, float* __restrict__ a32,
                            double* __restrict__ sigma_out) {
  const int i0 = blockIdx.x * CURV_TPB + threadIdx.x;
  const int i = min(i0, n - 1);
  const RadiusScale sc = radius_scale_of(e_dev, scale2, spec);
  double v[RAD_NS];
#pragma unroll
  for (int f = 0; f < RAD_NS; ++f) v[f] = part[(size_t)f * n + i];
  for (int s = 1; s < S; ++s) {
#pragma unroll
    for (int f = 0; f < RAD_NS; ++f) v[f] += part[((size_t)s * RAD_NS + f) * n + i];
  }
  double C[9];
  covariance_of_sums(v, C);
  double a = v[0] > 3.0 ? surface_variation(C) : 0.0;  // three points or fewer lie in a plane
  const bool again = i0 < n && v[0] > 3.0 && !(a * (C[0] + C[4] + C[8]) >= (double)(RAD_FLAT * sc.B));
  unsigned todo = __ballot_sync(0xffffffffu, again);
  if (todo) {
    for (; todo; todo &= todo - 1) {
      const int src = __ffs(todo) - 1;
      const double w = radius_sums_float64(P, n, box, sc.r2, __shfl_sync(0xffffffffu, i, src));
#pragma unroll
      for (int f = 0; f < RAD_NS; ++f) {
        const double t = __shfl_sync(0xffffffffu, w, 2 * f);
        if ((threadIdx.x & 31) == src) v[f] = t;
      }
    }
    if (again) {
      covariance_of_sums(v, C);
      a = surface_variation(C);
    }
  }
  if (i0 < n) {
    const int o = box ? __float_as_int(P[i].w) : i;
    a64[o] = a;
    a32[o] = (float)a;
  }
  if (sigma_out) sigma_part(a, i0 < n, min(CURV_TPB, n - (int)blockIdx.x * CURV_TPB), sigma_out);
}

// Splits of the cloud, so that a small one still gives every SM about eight
// blocks (at least one tile each); in order, where a block's work is the tiles
// near its queries, 32 (20,011 + 18,009 points, scale 1: 895 us with 8, 727
// with 16, 711 with 32; 40,000: 2731, 2180, 1860).
int radius_splits(int n, int num_sms, bool ordered) {
  const int blocks = (n + RAD_TPB - 1) / RAD_TPB, ntiles = (n + RAD_TILE - 1) / RAD_TILE;
  int S = ((ordered ? 32 : 8) * num_sms + blocks - 1) / blocks;
  if (S > ntiles) S = ntiles;
  const int tps = (ntiles + S - 1) / S;
  return (ntiles + tps - 1) / tps;
}
size_t radius_scratch_bytes(int n, int num_sms, bool ordered) {
  return (size_t)radius_splits(n, num_sms, ordered) * RAD_NS * n * sizeof(double);
}

// spec: the cloud's grid (launch_clouds; its extent); part: radius_scratch_bytes;
// box: the runs' boxes, with P in order and the index in w (launch_order), or
// NULL; sigma_out: sigma_part's output (NULL: not wanted).
cudaError_t launch_radius_curvature(Launch L, const float4* P, int n, const float* box, const double* e_dev,
                                    double scale2, const GridSpec* spec, int num_sms, double* part, double* a64,
                                    float* a32, double* sigma_out) {
  const int blocks = (n + RAD_TPB - 1) / RAD_TPB, ntiles = (n + RAD_TILE - 1) / RAD_TILE;
  const int S = radius_splits(n, num_sms, box != nullptr);
  radius_sums_kernel<<<dim3(blocks, S), RAD_TPB, 0, L.stream>>>(P, n, box, e_dev, scale2, spec, (ntiles + S - 1) / S,
                                                                part);
  radius_curvature_kernel<<<(n + CURV_TPB - 1) / CURV_TPB, CURV_TPB, 0, L.stream>>>(part, S, n, P, box, e_dev, scale2,
                                                                                   spec, a64, a32, sigma_out);
  if (L.counter) *L.counter += 2;
  return cudaGetLastError();
}

// ---- caller-supplied curvature --------------------------------------------
__global__ void check_curvature_kernel(const double* __restrict__ a64, int n, float* __restrict__ a32,
                                       int* __restrict__ err) {
  const int i = blockIdx.x * blockDim.x + threadIdx.x;
  if (i >= n) return;
  const double a = a64[i];
  if (!(a >= 0.0 && a <= 1.0)) atomicOr(err, ERR_NONFINITE);
  a32[i] = (float)a;
}

cudaError_t launch_check_curvature(Launch L, const double* a64, int n, float* a32, int* err) {
  check_curvature_kernel<<<(n + 255) / 256, 256, 0, L.stream>>>(a64, n, a32, err);
  return after_launch(L);
}

// ---- force-kernel records ----------------------------------------------
// s_ij = exp(-(aX - aY)^2 / sigma^2) = 2^(-(a_hat_X - a_hat_Y)^2) with
// a_hat = a * sqrt(log2 e) / sigma (Eq. 3).  In the mode g = aX aY s (Eq. 10)
// the factor aX enters the exponent as L = log2 aX (stored negated, -L >= 0)
// and aY multiplies the per-point sums; in the mode g = s, L = 0 and the aY
// factor is 1.  Reference coordinates are shifted by the reference mean so
// that |X'|^2 + |Y'|^2 - 2 X'.Y' loses little to cancellation.  The records
// are written tile-major as structure-of-arrays (FORCE_TJ points per tile).
// Padding records carry -L = +inf, so their weight is exactly 0.
__device__ __forceinline__ void write_x_record(int i, int n, const float4* __restrict__ X4,
                                               const double* __restrict__ aX64, int g_mode, const DevStats& st,
                                               float* __restrict__ Xr, float* __restrict__ XA) {
  const double kscale = st.kscale;
  const size_t t = (size_t)(i / FORCE_TJ), r = (size_t)(i % FORCE_TJ);
  float* xr = Xr + t * 4 * FORCE_TJ + r;
  float* xa = XA + t * 2 * FORCE_TJ + r;
  if (i < n) {
    const float4 c = X4[i];
    const float x = (float)((double)c.x - st.xbar[0]);
    const float y = (float)((double)c.y - st.xbar[1]);
    const float z = (float)((double)c.z - st.xbar[2]);
    const double nn = (double)x * x + (double)y * y + (double)z * z;
    xr[0] = x;
    xr[FORCE_TJ] = y;
    xr[2 * FORCE_TJ] = z;
    xr[3 * FORCE_TJ] = (float)nn;
    const double a = aX64[i];
    const float nL = g_mode == 1 ? (a > 0.0 ? (float)(-log2(a)) : INFINITY) : 0.f;
    xa[0] = (float)(a * kscale);
    xa[FORCE_TJ] = nL;
  } else {
    xr[0] = xr[FORCE_TJ] = xr[2 * FORCE_TJ] = xr[3 * FORCE_TJ] = 0.f;
    xa[0] = 0.f;
    xa[FORCE_TJ] = INFINITY;
  }
}

__device__ __forceinline__ void write_y_record(int i, int m, const float4* __restrict__ Y4,
                                               const double* __restrict__ aY64, const DevStats& st,
                                               float4* __restrict__ Y0r) {
  if (i < m) {
    const float4 c = Y4[i];
    Y0r[i] = make_float4(c.x, c.y, c.z, (float)(aY64[i] * st.kscale));
  } else {
    Y0r[i] = make_float4(0.f, 0.f, 0.f, 0.f);
  }
}

__global__ void records_kernel(const float4* __restrict__ X4, const double* __restrict__ aX64,
                               int n, int npad, const float4* __restrict__ Y4,
                               const double* __restrict__ aY64, int m, int mpad, int g_mode,
                               const DevStats* __restrict__ st, float* __restrict__ Xr,
                               float* __restrict__ XA, float4* __restrict__ Y0r) {
  const int i = blockIdx.x * blockDim.x + threadIdx.x;
  if (i < npad) write_x_record(i, n, X4, aX64, g_mode, *st, Xr, XA);
  if (i < mpad) write_y_record(i, m, Y4, aY64, *st, Y0r);
}

// Batched records: block (p, part) writes pair p's padded reference tiles and
// template slots (grid-strided over `part`).
__global__ void records_multi_kernel(const float4* __restrict__ X4, const double* __restrict__ aX64,
                                     const float4* __restrict__ Y4, const double* __restrict__ aY64,
                                     const BatchPair* __restrict__ pairs, int g_mode,
                                     const DevStats* __restrict__ st, float* __restrict__ Xr,
                                     float* __restrict__ XA, float4* __restrict__ Y0r) {
  const BatchPair bp = pairs[blockIdx.x];
  const DevStats& S = st[blockIdx.x];
  const int stride = blockDim.x * gridDim.y;
  const int npad = bp.ntiles * FORCE_TJ;
  for (int i = blockIdx.y * blockDim.x + threadIdx.x; i < npad; i += stride)
    write_x_record(i, (int)bp.n, X4 + bp.x0, aX64 + bp.x0, g_mode, S, Xr + (size_t)bp.xtile0 * 4 * FORCE_TJ,
                   XA + (size_t)bp.xtile0 * 2 * FORCE_TJ);
  for (int i = blockIdx.y * blockDim.x + threadIdx.x; i < bp.mpad; i += stride)
    write_y_record(i, (int)bp.m, Y4 + bp.y0, aY64 + bp.y0, S, Y0r + bp.ybase);
}

cudaError_t launch_records_multi(Launch L, const float4* X4, const double* aX64, const float4* Y4,
                                 const double* aY64, const BatchPair* pairs, int npairs, int g_mode,
                                 const DevStats* stats, float4* Xr, float2* XA, float4* Y0r) {
  records_multi_kernel<<<dim3(npairs, 8), 256, 0, L.stream>>>(X4, aX64, Y4, aY64, pairs, g_mode, stats,
                                                               reinterpret_cast<float*>(Xr),
                                                               reinterpret_cast<float*>(XA), Y0r);
  return after_launch(L);
}

// sigma of every pair of a batch: block p takes pair p's reference curvatures
// (mean, then squared deviations, in a fixed order).
__global__ void __launch_bounds__(SIGMA_T)
    sigma_multi_kernel(const double* __restrict__ aX64, const BatchPair* __restrict__ pairs, double sigma_user,
                       DevStats* __restrict__ out) {
  __shared__ double sh[SIGMA_T / 32];
  const BatchPair& bp = pairs[blockIdx.x];
  const double* a = aX64 + bp.x0;
  double v = 0.0;
  for (int64_t i = threadIdx.x; i < bp.n; i += SIGMA_T) v += a[i];
  const double sum = sigma_block_sum(v, sh), mean = sum / (double)bp.n;
  v = 0.0;
  for (int64_t i = threadIdx.x; i < bp.n; i += SIGMA_T) {
    const double d = a[i] - mean;
    v = fma(d, d, v);
  }
  const double d2 = sigma_block_sum(v, sh);
  if (threadIdx.x == 0) finish_sigma(sum, d2, bp.n, sigma_user, 1.0, out + blockIdx.x);
}

cudaError_t launch_sigma_multi(Launch L, const double* aX64, const BatchPair* pairs, int npairs, double sigma_user,
                               DevStats* out) {
  sigma_multi_kernel<<<npairs, SIGMA_T, 0, L.stream>>>(aX64, pairs, sigma_user, out);
  return after_launch(L);
}

cudaError_t launch_records(Launch L, const float4* X4, const double* aX64, int n, int npad,
                           const float4* Y4, const double* aY64, int m, int mpad, int g_mode,
                           const DevStats* stats, float4* Xr, float2* XA, float4* Y0r) {
  const int tpb = 256;
  const int tot = npad > mpad ? npad : mpad;
  records_kernel<<<(tot + tpb - 1) / tpb, tpb, 0, L.stream>>>(
      X4, aX64, n, npad, Y4, aY64, m, mpad, g_mode, stats, reinterpret_cast<float*>(Xr),
      reinterpret_cast<float*>(XA), Y0r);
  return after_launch(L);
}

}  // namespace scgr
