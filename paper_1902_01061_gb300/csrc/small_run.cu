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
#include <cooperative_groups.h>

#include "common.cuh"
#include "pair.cuh"
#include "pointsum.cuh"
#include "pose_update.cuh"

namespace cg = cooperative_groups;

namespace scgr {

constexpr int SMALL_FORCE = 512;                                // threads on the pairs
constexpr int SMALL_THREADS = SMALL_FORCE + 32 * POSE_PRE_WARPS;  // and the update's first half (leader)
constexpr int SMALL_CLUSTER = 16;
constexpr int SMALL_RUN = 128;  // reference points per plain float32 sum (as the half-tile force pass)
constexpr int SMALL_MAX_ROWS = 64;  // sums that meet in the leader: one per warp of points and block

struct SmallShared {
  DevPose ps;          // the leader's pose; the other blocks use its float32 map
  DevStats st;
  PosePre pre;
  PoseRate rate;
  double rows[SMALL_MAX_ROWS][13];
  double cols[8][13];
  double tot[13];
  float4 part[SMALL_FORCE];
};

// pc: template points per block (32, 64 or 128), so SMALL_FORCE / pc slices of
// the reference per point; a warp shares its slice (broadcast reads).
template <int PM>
__global__ void __launch_bounds__(SMALL_THREADS, 1)
    small_run_kernel(const float* __restrict__ Xr, const float* __restrict__ XA, int npad,
                     const float4* __restrict__ Y0r, const float* __restrict__ aY32, int g_mode, int m, int pc,
                     DevPose* pose, const DevStats* __restrict__ stats, StepParams sp, float qexp, int iters, int* err) {
  extern __shared__ __align__(16) float sX[];  // [6][npad]
  __shared__ SmallShared S;
  cg::cluster_group cluster = cg::this_cluster();
  const int rank = (int)cluster.block_rank(), nblk = (int)cluster.num_blocks();
  const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
  const bool leader = rank == 0;

  for (int t = tid; t < npad / FORCE_TJ * 6 * (FORCE_TJ / 4); t += SMALL_THREADS) {
    const int tile = t / (6 * (FORCE_TJ / 4)), r = t / (FORCE_TJ / 4) % 6, j = t % (FORCE_TJ / 4);
    const float* src = r < 4 ? Xr + ((size_t)tile * 4 + r) * FORCE_TJ : XA + ((size_t)tile * 2 + r - 4) * FORCE_TJ;
    reinterpret_cast<float4*>(sX + (size_t)r * npad)[tile * (FORCE_TJ / 4) + j] = reinterpret_cast<const float4*>(src)[j];
  }
  if (tid < (int)(sizeof(DevPose) / 4)) reinterpret_cast<int*>(&S.ps)[tid] = reinterpret_cast<const int*>(pose)[tid];
  if (tid < (int)(sizeof(DevStats) / 4)) reinterpret_cast<int*>(&S.st)[tid] = reinterpret_cast<const int*>(stats)[tid];
  const int p = tid % pc, sl = tid / pc, i = rank * pc + p;
  const float4 y0 = i < m ? Y0r[i] : make_float4(0.f, 0.f, 0.f, 0.f);
  const float ay = i < m && g_mode == 1 ? aY32[i] : 1.f;
  const int len = npad / (SMALL_FORCE / pc);
  cluster.sync();

  for (int it = 0; it < iters; ++it) {
    if (tid >= SMALL_FORCE) {
      if (leader) pose_pre(warp - SMALL_FORCE / 32, &S.ps, &S.st, sp, S.pre, S.rate);
    } else {
      const PointFrame fr(&S.ps);
      {
        float yx, yy, yz;
        template_point(y0, fr.A, fr.b, yx, yy, yz);
        const float n = fmaf(yz, yz, fmaf(yy, yy, yx * yx));
        const u64 mx = pk2(-2.f * yx, -2.f * yx), my = pk2(-2.f * yy, -2.f * yy), mz = pk2(-2.f * yz, -2.f * yz);
        const u64 ny = pk2(n, n), ah = pk2(y0.w, y0.w), nq = pk2(-qexp, -qexp);
        float h[4] = {0.f, 0.f, 0.f, 0.f}, c[4] = {0.f, 0.f, 0.f, 0.f};
        const float* x0 = sX + sl * len;
        for (int j0 = 0; j0 < len; j0 += SMALL_RUN) {
          u64 a[2][4];
#pragma unroll
          for (int u = 0; u < 2; ++u)
#pragma unroll
            for (int v = 0; v < 4; ++v) a[u][v] = 0ull;
          const int j1 = min(len, j0 + SMALL_RUN);
#pragma unroll 2
          for (int j = j0; j < j1; j += 4) {
            const ulonglong2 X = *reinterpret_cast<const ulonglong2*>(x0 + j);
            const ulonglong2 Y = *reinterpret_cast<const ulonglong2*>(x0 + npad + j);
            const ulonglong2 Z = *reinterpret_cast<const ulonglong2*>(x0 + 2 * npad + j);
            const ulonglong2 N = *reinterpret_cast<const ulonglong2*>(x0 + 3 * npad + j);
            const ulonglong2 Av = *reinterpret_cast<const ulonglong2*>(x0 + 4 * npad + j);
            const ulonglong2 Lv = *reinterpret_cast<const ulonglong2*>(x0 + 5 * npad + j);
            pair2<PM>(X.x, Y.x, Z.x, N.x, Av.x, Lv.x, mx, my, mz, ny, ah, nq, a[0][0], a[0][1], a[0][2], a[0][3]);
            pair2<PM>(X.y, Y.y, Z.y, N.y, Av.y, Lv.y, mx, my, mz, ny, ah, nq, a[1][0], a[1][1], a[1][2], a[1][3]);
          }
#pragma unroll
          for (int v = 0; v < 4; ++v) {
            float l0, l1;
            upk2(add2(a[0][v], a[1][v]), l0, l1);
            kahan_add(h[v], c[v], l0 + l1);
          }
        }
        S.part[sl * pc + p] = make_float4(h[0] - c[0], h[1] - c[1], h[2] - c[2], h[3] - c[3]);
      }
      asm volatile("bar.sync 1, %0;" ::"n"(SMALL_FORCE) : "memory");
      if (tid < pc) {  // whole warps
        float acc[13];
#pragma unroll
        for (int q = 0; q < 13; ++q) acc[q] = 0.f;
        const float4 fw = point_fw(S.part, (size_t)pc, SMALL_FORCE / pc, p, y0, ay, fr);
        if (i < m) point_acc(fw, y0, fr, acc);
        double w[16];
#pragma unroll
        for (int q = 0; q < 13; ++q) w[q] = (double)acc[q];
        w[13] = w[14] = w[15] = 0.0;
        warp_reduce16(w);
        const int q = warp_reduce16_slot(lane);
        double* row = cluster.map_shared_rank(&S.rows[0][0], 0) + (rank * (pc / 32) + warp) * 13;
        if ((lane & 1) == 0 && q < 13) row[q] = w[0];
      }
    }
    cluster.sync();  // the rows are in the leader, every block has read its map
    if (leader) {
      const int rows = nblk * (pc / 32);
      if (warp < 8 && lane < 13) {
        double v = 0.0;
        for (int r = warp; r < rows; r += 8) v += S.rows[r][lane];
        S.cols[warp][lane] = v;
      }
      __syncthreads();
      if (warp == 0) {
        if (lane < 13) {
          double v = S.cols[0][lane];
#pragma unroll
          for (int k = 1; k < 8; ++k) v += S.cols[k][lane];
          S.tot[lane] = v;
        }
        __syncwarp();
        pose_post(S.tot, &S.ps, &S.st, sp, S.pre, S.rate, err);
        __syncwarp();
        // the float32 map (A, b, ych, ycl: 18 consecutive floats) to the other blocks
        constexpr int MAP = 18;
        static_assert(sizeof(((DevPose*)0)->A) + sizeof(((DevPose*)0)->b) + sizeof(((DevPose*)0)->ych) +
                              sizeof(((DevPose*)0)->ycl) == MAP * 4, "map layout");
        for (int e = lane; e < (nblk - 1) * MAP; e += 32)
          cluster.map_shared_rank(S.ps.A, 1 + e / MAP)[e % MAP] = S.ps.A[e % MAP];
      }
    }
    cluster.sync();
  }
  if (leader && tid < (int)(sizeof(DevPose) / 4)) reinterpret_cast<int*>(pose)[tid] = reinterpret_cast<const int*>(&S.ps)[tid];
}

static int small_points(int m) {
  const int per = (m + SMALL_CLUSTER - 1) / SMALL_CLUSTER;
  return per <= 32 ? 32 : per <= 64 ? 64 : 128;
}

template <int PM>
static cudaError_t small_config(int npad, int* clusters, cudaLaunchConfig_t* cfg, cudaLaunchAttribute* at) {
  const size_t smem = (size_t)npad * 6 * sizeof(float);
  cudaError_t e = cudaFuncSetAttribute(small_run_kernel<PM>, cudaFuncAttributeMaxDynamicSharedMemorySize,
                                       SMALL_MAX_POINTS * 6 * (int)sizeof(float));
  if (e == cudaSuccess) e = cudaFuncSetAttribute(small_run_kernel<PM>, cudaFuncAttributeNonPortableClusterSizeAllowed, 1);
  if (e != cudaSuccess) return e;
  *cfg = cudaLaunchConfig_t{};
  cfg->gridDim = dim3(SMALL_CLUSTER);
  cfg->blockDim = dim3(SMALL_THREADS);
  cfg->dynamicSmemBytes = smem;
  at->id = cudaLaunchAttributeClusterDimension;
  at->val.clusterDim.x = SMALL_CLUSTER;
  at->val.clusterDim.y = at->val.clusterDim.z = 1;
  cfg->attrs = at;
  cfg->numAttrs = 1;
  return clusters ? cudaOccupancyMaxActiveClusters(clusters, small_run_kernel<PM>, cfg) : cudaSuccess;
}

// Whether the device runs a cluster of this kernel (asked once per context).
bool small_run_available() {
  cudaLaunchConfig_t cfg;
  cudaLaunchAttribute at[1];
  int clusters = 0;
  if (small_config<2>(SMALL_MAX_POINTS, &clusters, &cfg, at) != cudaSuccess) {
    cudaGetLastError();
    return false;
  }
  return clusters > 0;
}

template <int PM>
static cudaError_t launch_small_pm(Launch L, const float* Xr, const float* XA, int npad, const float4* Y0r,
                                   const float* aY32, int g_mode, int m, DevPose* pose, const DevStats* stats,
                                   StepParams sp, float qexp, int iters, int* err) {
  cudaLaunchConfig_t cfg;
  cudaLaunchAttribute at[1];
  cudaError_t e = small_config<PM>(npad, nullptr, &cfg, at);
  if (e != cudaSuccess) return e;
  cfg.stream = L.stream;
  if (L.counter) ++*L.counter;
  return cudaLaunchKernelEx(&cfg, small_run_kernel<PM>, Xr, XA, npad, Y0r, aY32, g_mode, m, small_points(m), pose,
                            stats, sp, qexp, iters, err);
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
