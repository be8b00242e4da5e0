// Points of both clouds in Morton order of a 32^3 grid over their box, for the
// radius neighbourhoods (descriptors.cu): consecutive points are close to one
// another, so runs of 32 have small boxes.  A stable radix sort (two passes of
// 8 bits) of a 15-bit key, free of atomics on the output: the order, and with it
// every later sum, is the same in every run.  Both clouds share each launch
// (blockIdx.y).
//
// Bound: launch latency and a block's chain of rounds (20,011 + 17,611 points:
// 28 us of kernels, seven launches).
#include "common.cuh"

namespace scgr {

constexpr int ORD_T = 256;
constexpr int ORD_ROUNDS = 4;
constexpr int ORD_BLOCK = ORD_T * ORD_ROUNDS;  // points per block
constexpr int ORD_SCAN_T = 1024;

__host__ __device__ inline int order_blocks(int n) { return (n + ORD_BLOCK - 1) / ORD_BLOCK; }

// bits 0..4 of v to bits 0, 3, 6, 9, 12
__device__ __forceinline__ unsigned spread3(unsigned v) {
  return (v & 1) | (v & 2) << 2 | (v & 4) << 4 | (v & 8) << 6 | (v & 16) << 8;
}
__device__ __forceinline__ unsigned order_key(float4 c, const GridSpec& sp) {
  const float inv = 32.f / sp.extent;  // an empty box: NaN or infinite products, clamped
  const unsigned x = (unsigned)fminf(fmaxf((c.x - sp.o[0]) * inv, 0.f), 31.f);
  const unsigned y = (unsigned)fminf(fmaxf((c.y - sp.o[1]) * inv, 0.f), 31.f);
  const unsigned z = (unsigned)fminf(fmaxf((c.z - sp.o[2]) * inv, 0.f), 31.f);
  return spread3(x) | spread3(y) << 1 | spread3(z) << 2;
}

// Pass 0 keys the points (and counts the low digit), pass 1 counts the high one.
template <int PASS>
__global__ void __launch_bounds__(ORD_T) order_count_kernel(const OrderClouds oc) {
  __shared__ int hist[256];
  const OrderCloud& c = oc.c[blockIdx.y];
  const int nb = order_blocks(c.n);
  if ((int)blockIdx.x >= nb) return;
  hist[threadIdx.x] = 0;
  __syncthreads();
#pragma unroll
  for (int r = 0; r < ORD_ROUNDS; ++r) {
    const int i = blockIdx.x * ORD_BLOCK + r * ORD_T + threadIdx.x;
    if (i < c.n) {
      unsigned k;
      if (PASS == 0) {
        k = order_key(c.P[i], *c.spec);
        c.key[0][i] = (unsigned short)k;
      } else {
        k = c.key[1][i];
      }
      atomicAdd(&hist[PASS == 0 ? (k & 255) : (k >> 8)], 1);
    }
  }
  __syncthreads();
  c.count[threadIdx.x * nb + blockIdx.x] = hist[threadIdx.x];
}

// One block per cloud: exclusive scan of the 256 x nb counts, digit-major.
__global__ void __launch_bounds__(ORD_SCAN_T) order_scan_kernel(const OrderClouds oc) {
  __shared__ int shw[32];
  const OrderCloud& c = oc.c[blockIdx.y];
  const int total = 256 * order_blocks(c.n);
  const int per = (total + ORD_SCAN_T - 1) / ORD_SCAN_T;
  const int b = threadIdx.x * per, e = min(total, b + per);
  int sum = 0;
  for (int i = b; i < e; ++i) sum += c.count[i];
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
  int inc = sum;
#pragma unroll
  for (int off = 1; off < 32; off <<= 1) {
    const int u = __shfl_up_sync(0xffffffffu, inc, off);
    if (lane >= off) inc += u;
  }
  if (lane == 31) shw[warp] = inc;
  __syncthreads();
  if (warp == 0) {
    int w = shw[lane];
#pragma unroll
    for (int off = 1; off < 32; off <<= 1) {
      const int u = __shfl_up_sync(0xffffffffu, w, off);
      if (lane >= off) w += u;
    }
    shw[lane] = w;
  }
  __syncthreads();
  int run = inc - sum + (warp > 0 ? shw[warp - 1] : 0);
  for (int i = b; i < e; ++i) {
    const int v = c.count[i];
    c.count[i] = run;
    run += v;
  }
}

// Stable scatter of one digit: rounds of 256 points in index order; in a round
// a point's place is its digit's base, the earlier warps' counts of that digit
// and the earlier lanes of its own warp.
template <int PASS>
__global__ void __launch_bounds__(ORD_T) order_scatter_kernel(const OrderClouds oc) {
  __shared__ int base[256];
  __shared__ int wc[ORD_T / 32][256];
  const OrderCloud& c = oc.c[blockIdx.y];
  const int nb = order_blocks(c.n);
  if ((int)blockIdx.x >= nb) return;
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
  base[threadIdx.x] = c.count[threadIdx.x * nb + blockIdx.x];
  for (int r = 0; r < ORD_ROUNDS; ++r) {
#pragma unroll
    for (int w = 0; w < ORD_T / 32; ++w) wc[w][threadIdx.x] = 0;
    __syncthreads();
    const int i = blockIdx.x * ORD_BLOCK + r * ORD_T + threadIdx.x;
    const bool live = i < c.n;
    const unsigned k = live ? c.key[PASS][i] : 0u;
    const int digit = live ? (int)(PASS == 0 ? (k & 255) : (k >> 8)) : 256;
    const unsigned same = __match_any_sync(0xffffffffu, digit);
    const int rank = __popc(same & ((1u << lane) - 1));
    if (live && rank == 0) wc[warp][digit] = __popc(same);
    __syncthreads();
    int run = base[threadIdx.x];
#pragma unroll
    for (int w = 0; w < ORD_T / 32; ++w) {
      const int v = wc[w][threadIdx.x];
      wc[w][threadIdx.x] = run;
      run += v;
    }
    base[threadIdx.x] = run;
    __syncthreads();
    if (live) {
      const int pos = wc[warp][digit] + rank;
      if (PASS == 0) {
        c.key[1][pos] = (unsigned short)k;
        c.perm[0][pos] = i;
      } else {
        c.perm[1][pos] = c.perm[0][i];
      }
    }
    __syncthreads();
  }
}

// The points in order, the index in w, and the boxes of the runs of 32.
__global__ void __launch_bounds__(ORD_T) order_gather_kernel(const OrderClouds oc) {
  const OrderCloud& c = oc.c[blockIdx.y];
  const int s = blockIdx.x * ORD_T + threadIdx.x;
  if (s - (int)(threadIdx.x & 31) >= c.n) return;
  float b[6] = {INFINITY, INFINITY, INFINITY, INFINITY, INFINITY, INFINITY};  // min, -max
  if (s < c.n) {
    const int i = c.perm[1][s];
    float4 p = c.P[i];
    b[0] = p.x; b[1] = p.y; b[2] = p.z;
    b[3] = -p.x; b[4] = -p.y; b[5] = -p.z;
    p.w = __int_as_float(i);
    c.sorted[s] = p;
  }
#pragma unroll
  for (int off = 16; off > 0; off >>= 1)
#pragma unroll
    for (int q = 0; q < 6; ++q) b[q] = fminf(b[q], __shfl_xor_sync(0xffffffffu, b[q], off));
  if ((threadIdx.x & 31) < 6) {
    const int q = threadIdx.x & 31;
    float v = b[0];
#pragma unroll
    for (int u = 1; u < 6; ++u) v = q == u ? b[u] : v;
    c.box[6 * (size_t)(s >> 5) + q] = v;
  }
}

static size_t order_count_entries(int64_t n) { return (size_t)256 * order_blocks((int)n); }

size_t order_bytes(int64_t n) {
  return (size_t)n * (sizeof(float4) + 2 * sizeof(int) + 2 * sizeof(unsigned short)) +
         order_count_entries(n) * sizeof(int) + (size_t)((n + 31) / 32) * 6 * sizeof(float);
}

// A cloud's arrays in one buffer of order_bytes.
OrderCloud order_cloud(void* buf, const float4* P, const GridSpec* spec, int64_t n) {
  OrderCloud o{};
  o.P = P;
  o.spec = spec;
  o.n = (int)n;
  o.sorted = (float4*)buf;
  o.box = (float*)(o.sorted + n);
  o.perm[0] = (int*)(o.box + (n + 31) / 32 * 6);
  o.perm[1] = o.perm[0] + n;
  o.count = o.perm[1] + n;
  o.key[0] = (unsigned short*)(o.count + order_count_entries(n));
  o.key[1] = o.key[0] + n;
  return o;
}

cudaError_t launch_order(Launch L, const OrderClouds& oc) {
  const int most = oc.c[0].n > oc.c[1].n ? oc.c[0].n : oc.c[1].n;
  const dim3 grid(order_blocks(most), 2), one(1, 2);
  order_count_kernel<0><<<grid, ORD_T, 0, L.stream>>>(oc);
  order_scan_kernel<<<one, ORD_SCAN_T, 0, L.stream>>>(oc);
  order_scatter_kernel<0><<<grid, ORD_T, 0, L.stream>>>(oc);
  order_count_kernel<1><<<grid, ORD_T, 0, L.stream>>>(oc);
  order_scan_kernel<<<one, ORD_SCAN_T, 0, L.stream>>>(oc);
  order_scatter_kernel<1><<<grid, ORD_T, 0, L.stream>>>(oc);
  order_gather_kernel<<<dim3((most + ORD_T - 1) / ORD_T, 2), ORD_T, 0, L.stream>>>(oc);
  if (L.counter) *L.counter += 7;
  return cudaGetLastError();
}

}  // namespace scgr
