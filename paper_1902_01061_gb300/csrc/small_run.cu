// Many iterations of a small registration in one launch.
//
// At 1,000 x 1,000 an iteration is a few microseconds of pair work; as a force
// launch and a combine-finalize launch it took 22 us, half of it launch
// latency, the trip of the split partials through memory and re-reading the
// records.  Here one thread-block cluster runs all iterations: every block
// keeps the whole reference in shared memory and owns a share of the template
// points, the blocks' 13 sums meet in the leader's shared memory (distributed
// shared memory), the leader's warp 0 forms the pose and writes the float32 map
// back to every block.  Two cluster barriers an iteration; the blocks of a
// cluster are co-scheduled by the hardware, and nothing waits on another launch.
//
// Bound: the leader's chain (13 sums across blocks, the pose update's float64)
// and then the pair rate of 16 SMs.  An iteration: 500 x 500 7.6 us (20.9 as
// two launches), 1,000 x 1,000 11.0 (22.7), 2,000 x 2,000 26.4 (28.4); with
// one template point per thread across all of a block's threads, instead of a
// warp per reference slice, 1,000 x 1,000 took 12.9.
#include <cooperative_groups.h>

#include "common.cuh"
#include "pair.cuh"
#include "pointsum.cuh"
#include "pose_update.cuh"

namespace cg = cooperative_groups;

namespace scgr {

constexpr int SMALL_THREADS = 512;
constexpr int SMALL_WARPS = SMALL_THREADS / 32;  // slices of the reference, one per warp
constexpr int SMALL_CLUSTER = 16;
constexpr int SMALL_RUN = 128;  // reference points per plain float32 sum (as the half-tile force pass)
constexpr int SMALL_MAX_P = 4;

struct SmallShared {
  DevPose ps;          // the leader's pose; the other blocks use its float32 map
  DevStats st;
  PosePre pre;
  PoseRate rate[2];
  double rows[SMALL_CLUSTER * SMALL_MAX_P][13];  // one per warp of points and block
  double cols[4][13];
  double tot[13];
  bool ok;
};

// P template points per lane: a block owns 32 P points, and each of its warps
// takes them against one slice of the reference (broadcast reads).
template <int PM, int P>
__global__ void __launch_bounds__(SMALL_THREADS, 1)
    small_run_kernel(const float* __restrict__ Xr, const float* __restrict__ XA, int npad,
                     const float4* __restrict__ Y0r, const float* __restrict__ aY32, int g_mode, int m, DevPose* pose,
                     const DevStats* __restrict__ stats, StepParams sp, float qexp, int iters, int* err) {
  constexpr int PC = 32 * P;
  extern __shared__ __align__(16) float sX[];  // [6][npad], then the slices' sums [SMALL_WARPS][PC]
  __shared__ SmallShared S;
  cg::cluster_group cluster = cg::this_cluster();
  const int rank = (int)cluster.block_rank();
  const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
  const bool leader = rank == 0;
  float4* part = reinterpret_cast<float4*>(sX + (size_t)6 * npad);

  for (int t = tid; t < npad / FORCE_TJ * 6 * (FORCE_TJ / 4); t += SMALL_THREADS) {
    const int tile = t / (6 * (FORCE_TJ / 4)), r = t / (FORCE_TJ / 4) % 6, j = t % (FORCE_TJ / 4);
    const float* src = r < 4 ? Xr + ((size_t)tile * 4 + r) * FORCE_TJ : XA + ((size_t)tile * 2 + r - 4) * FORCE_TJ;
    reinterpret_cast<float4*>(sX + (size_t)r * npad)[tile * (FORCE_TJ / 4) + j] = reinterpret_cast<const float4*>(src)[j];
  }
  if (tid < (int)(sizeof(DevPose) / 4)) reinterpret_cast<int*>(&S.ps)[tid] = reinterpret_cast<const int*>(pose)[tid];
  if (tid < (int)(sizeof(DevStats) / 4)) reinterpret_cast<int*>(&S.st)[tid] = reinterpret_cast<const int*>(stats)[tid];
  float4 y0[P];
#pragma unroll
  for (int q = 0; q < P; ++q) {
    const int i = rank * PC + q * 32 + lane;
    y0[q] = i < m ? Y0r[i] : make_float4(0.f, 0.f, 0.f, 0.f);
  }
  const int len = npad / SMALL_WARPS;
  cluster.sync();
  const int it0 = S.ps.it, E = S.ps.E;
  if (leader && warp == 1) pose_schedule(it0, E, sp, S.rate[0]);
  if (leader && warp == 2) pose_scale(S.ps.s, &S.st, sp, S.rate[0]);

  for (int it = 0; it < iters; ++it) {
    PoseRate& now = S.rate[it & 1];
    PoseRate& next = S.rate[(it + 1) & 1];
    const PointFrame fr(&S.ps);
    if (leader && warp >= SMALL_WARPS - 2) pose_pre(2 + (warp & 1), &S.ps, &S.st, sp, S.pre, now);
    {
      u64 mx[P], my[P], mz[P], ny[P], ah[P];
      float h[P][4], c[P][4];
#pragma unroll
      for (int q = 0; q < P; ++q) {
        float yx, yy, yz;
        template_point(y0[q], fr.A, fr.b, yx, yy, yz);
        const float n = fmaf(yz, yz, fmaf(yy, yy, yx * yx));
        mx[q] = pk2(-2.f * yx, -2.f * yx);
        my[q] = pk2(-2.f * yy, -2.f * yy);
        mz[q] = pk2(-2.f * yz, -2.f * yz);
        ny[q] = pk2(n, n);
        ah[q] = pk2(y0[q].w, y0[q].w);
#pragma unroll
        for (int v = 0; v < 4; ++v) h[q][v] = c[q][v] = 0.f;
      }
      const u64 nq = pk2(-qexp, -qexp);
      const float* x0 = sX + warp * len;
      for (int j0 = 0; j0 < len; j0 += SMALL_RUN) {
        u64 a[P][4];
#pragma unroll
        for (int q = 0; q < P; ++q)
#pragma unroll
          for (int v = 0; v < 4; ++v) a[q][v] = 0ull;
        const int j1 = min(len, j0 + SMALL_RUN);
        constexpr int UNR = P >= 4 ? 1 : P == 2 ? 2 : 4;
#pragma unroll UNR
        for (int j = j0; j < j1; j += 4) {
          const ulonglong2 X = *reinterpret_cast<const ulonglong2*>(x0 + j);
          const ulonglong2 Y = *reinterpret_cast<const ulonglong2*>(x0 + npad + j);
          const ulonglong2 Z = *reinterpret_cast<const ulonglong2*>(x0 + 2 * npad + j);
          const ulonglong2 N = *reinterpret_cast<const ulonglong2*>(x0 + 3 * npad + j);
          const ulonglong2 Av = *reinterpret_cast<const ulonglong2*>(x0 + 4 * npad + j);
          const ulonglong2 Lv = *reinterpret_cast<const ulonglong2*>(x0 + 5 * npad + j);
#pragma unroll
          for (int q = 0; q < P; ++q)
            pair2<PM>(X.x, Y.x, Z.x, N.x, Av.x, Lv.x, mx[q], my[q], mz[q], ny[q], ah[q], nq, a[q][0], a[q][1], a[q][2], a[q][3]);
#pragma unroll
          for (int q = 0; q < P; ++q)
            pair2<PM>(X.y, Y.y, Z.y, N.y, Av.y, Lv.y, mx[q], my[q], mz[q], ny[q], ah[q], nq, a[q][0], a[q][1], a[q][2], a[q][3]);
        }
#pragma unroll
        for (int q = 0; q < P; ++q)
#pragma unroll
          for (int v = 0; v < 4; ++v) {
            float l0, l1;
            upk2(a[q][v], l0, l1);
            kahan_add(h[q][v], c[q][v], l0 + l1);
          }
      }
#pragma unroll
      for (int q = 0; q < P; ++q)
        part[warp * PC + q * 32 + lane] =
            make_float4(h[q][0] - c[q][0], h[q][1] - c[q][1], h[q][2] - c[q][2], h[q][3] - c[q][3]);
    }
    __syncthreads();
    if (warp < P) {  // point `tid` of the block
      const int i = rank * PC + tid;
      const float4 y = i < m ? Y0r[i] : make_float4(0.f, 0.f, 0.f, 0.f);
      float acc[13];
#pragma unroll
      for (int q = 0; q < 13; ++q) acc[q] = 0.f;
      if (i < m) {
        const float4 fw = point_fw(part, (size_t)PC, SMALL_WARPS, tid, y, g_mode == 1 ? aY32[i] : 1.f, fr);
        point_acc(fw, y, fr, acc);
      }
      double w[16];
#pragma unroll
      for (int q = 0; q < 13; ++q) w[q] = (double)acc[q];
      w[13] = w[14] = w[15] = 0.0;
      warp_reduce16(w);
      const int q = warp_reduce16_slot(lane);
      double* row = cluster.map_shared_rank(&S.rows[0][0], 0) + (rank * P + warp) * 13;
      if ((lane & 1) == 0 && q < 13) row[q] = w[0];
    }
    cluster.sync();  // the rows are in the leader, every block has read its map
    if (leader) {
      constexpr int ROWS = SMALL_CLUSTER * P;
      // column sums: 8 chains (4 warps x 2 half warps) of ROWS / 8, then across
      if (warp < 4) {
        const int half = lane >> 4, q = lane & 15;
        double v = 0.0;
        if (q < 13)
#pragma unroll
          for (int r = 0; r < ROWS / 8; ++r) v += S.rows[r * 8 + warp * 2 + half][q];
        v += __shfl_xor_sync(WFULL, v, 16);
        if (lane < 13) S.cols[warp][lane] = v;
      }
      __syncthreads();
      if (warp == 0) {
        if (lane < 13) S.tot[lane] = ((S.cols[0][lane] + S.cols[1][lane]) + S.cols[2][lane]) + S.cols[3][lane];
        __syncwarp();
        const bool moved = pose_post(S.tot, &S.ps, &S.st, sp, S.pre, now, err);
        if (lane == 0) S.ok = moved;
        __syncwarp();
        // the float32 map (A, b, ych, ycl: 18 consecutive floats) to the other blocks
        constexpr int MAP = 18;
        static_assert(sizeof(((DevPose*)0)->A) + sizeof(((DevPose*)0)->b) + sizeof(((DevPose*)0)->ych) +
                              sizeof(((DevPose*)0)->ycl) == MAP * 4, "map layout");
        for (int e = lane; e < (SMALL_CLUSTER - 1) * MAP; e += 32)
          cluster.map_shared_rank(S.ps.A, 1 + e / MAP)[e % MAP] = S.ps.A[e % MAP];
      } else if (warp == 1) {  // beside it: the next iteration's schedule and scale
        pose_schedule(it0 + it + 1, E, sp, next);
      } else if (warp == 2) {
        pose_scale(now.sn, &S.st, sp, next);
      }
    }
    cluster.sync();
    if (leader && !S.ok) {  // the pose was kept, and so is its scale
      if (warp == 2) pose_scale(S.ps.s, &S.st, sp, next);
      __syncthreads();
    }
  }
  if (leader && tid < (int)(sizeof(DevPose) / 4)) reinterpret_cast<int*>(pose)[tid] = reinterpret_cast<const int*>(&S.ps)[tid];
}

static size_t small_smem(int npad, int P) {
  return (size_t)npad * 6 * sizeof(float) + (size_t)SMALL_WARPS * 32 * P * sizeof(float4);
}

template <int PM, int P>
static cudaError_t small_config(int npad, int* clusters, cudaLaunchConfig_t* cfg, cudaLaunchAttribute* at) {
  cudaError_t e = cudaFuncSetAttribute(small_run_kernel<PM, P>, cudaFuncAttributeMaxDynamicSharedMemorySize,
                                       (int)small_smem(SMALL_MAX_POINTS, P));
  if (e == cudaSuccess) e = cudaFuncSetAttribute(small_run_kernel<PM, P>, cudaFuncAttributeNonPortableClusterSizeAllowed, 1);
  if (e != cudaSuccess) return e;
  *cfg = cudaLaunchConfig_t{};
  cfg->gridDim = dim3(SMALL_CLUSTER);
  cfg->blockDim = dim3(SMALL_THREADS);
  cfg->dynamicSmemBytes = small_smem(npad, P);
  at->id = cudaLaunchAttributeClusterDimension;
  at->val.clusterDim.x = SMALL_CLUSTER;
  at->val.clusterDim.y = at->val.clusterDim.z = 1;
  cfg->attrs = at;
  cfg->numAttrs = 1;
  return clusters ? cudaOccupancyMaxActiveClusters(clusters, small_run_kernel<PM, P>, cfg) : cudaSuccess;
}

// Whether the device runs a cluster of this kernel (asked once per context).
bool small_run_available() {
  cudaLaunchConfig_t cfg;
  cudaLaunchAttribute at[1];
  int clusters = 0;
  if (small_config<2, SMALL_MAX_P>(SMALL_MAX_POINTS, &clusters, &cfg, at) != cudaSuccess) {
    cudaGetLastError();
    return false;
  }
  return clusters > 0;
}

template <int PM, int P>
static cudaError_t launch_small_p(Launch L, const float* Xr, const float* XA, int npad, const float4* Y0r,
                                  const float* aY32, int g_mode, int m, DevPose* pose, const DevStats* stats,
                                  StepParams sp, float qexp, int iters, int* err) {
  cudaLaunchConfig_t cfg;
  cudaLaunchAttribute at[1];
  cudaError_t e = small_config<PM, P>(npad, nullptr, &cfg, at);
  if (e != cudaSuccess) return e;
  cfg.stream = L.stream;
  if (L.counter) ++*L.counter;
  return cudaLaunchKernelEx(&cfg, small_run_kernel<PM, P>, Xr, XA, npad, Y0r, aY32, g_mode, m, pose, stats, sp, qexp,
                            iters, err);
}

template <int PM>
static cudaError_t launch_small_pm(Launch L, const float* Xr, const float* XA, int npad, const float4* Y0r,
                                   const float* aY32, int g_mode, int m, DevPose* pose, const DevStats* stats,
                                   StepParams sp, float qexp, int iters, int* err) {
  const auto launch = m <= SMALL_CLUSTER * 32   ? launch_small_p<PM, 1>
                      : m <= SMALL_CLUSTER * 64 ? launch_small_p<PM, 2>
                                                : launch_small_p<PM, 4>;
  return launch(L, Xr, XA, npad, Y0r, aY32, g_mode, m, pose, stats, sp, qexp, iters, err);
}

cudaError_t launch_small_run(Launch L, int pmode, const float4* Xr, const float2* XA, int npad, const float4* Y0r,
                             const float* aY32, int g_mode, int m, DevPose* pose, const DevStats* stats,
                             StepParams sp, float qexp, int iters, int* err) {
  const float* xr = reinterpret_cast<const float*>(Xr);
  const float* xa = reinterpret_cast<const float*>(XA);
  const auto launch = pmode == 2   ? launch_small_pm<2>
                      : pmode == 3 ? launch_small_pm<3>
                      : pmode == 4 ? launch_small_pm<4>
                                   : launch_small_pm<0>;
  return launch(L, xr, xa, npad, Y0r, aY32, g_mode, m, pose, stats, sp, qexp, iters, err);
}

}  // namespace scgr
