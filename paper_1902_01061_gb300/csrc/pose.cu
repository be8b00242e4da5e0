// Pose update in float64 (Eq. 5.5, Eq. 6, Eq. 8, Eq. 9, Eq. 12): one block
// reduces the per-block (F, W, T) partials in a fixed order, then one warp
// forms the step, the Kabsch rotation (the polar factor of C^ by Newton's
// iteration in float32 with float64 corrections, else in float64, or a
// one-sided Jacobi SVD in the reflection and near-singular cases), the
// scale, the composed pose and its re-orthonormalisation.  The pose never
// leaves the device, so a run of iterations is a plain sequence of launches.
#include <cmath>

#include "common.cuh"
#include "pointsum.cuh"
#include "pose_update.cuh"

namespace scgr {

// Derived float32 map and template mean for the current pose.
__device__ void refresh_pose(DevPose* ps, const DevStats* st) {
  for (int q = 0; q < 9; ++q) ps->A[q] = (float)(ps->s * ps->R[q]);
  for (int c = 0; c < 3; ++c) {
    ps->b[c] = (float)(ps->t[c] - st->xbar[c]);
    const double yb = ps->s * (st->ybar0[0] * ps->R[c] + st->ybar0[1] * ps->R[3 + c] +
                               st->ybar0[2] * ps->R[6 + c]) + ps->t[c];
    set_ybs(ps, c, yb - st->xbar[c]);
  }
}

__global__ void pose_init_kernel(DevPose* ps, const DevStats* st, int E) {
  if (threadIdx.x != 0 || blockIdx.x != 0) return;
  for (int q = 0; q < 9; ++q) ps->R[q] = (q % 4 == 0) ? 1.0 : 0.0;
  ps->t[0] = ps->t[1] = ps->t[2] = 0.0;
  ps->s = 1.0;
  ps->it = 0;
  ps->E = E;
  ps->degenerate = 0;
  refresh_pose(ps, st);
}

__global__ void pose_refresh_kernel(DevPose* ps, const DevStats* st) {
  if (threadIdx.x == 0 && blockIdx.x == 0) refresh_pose(ps, st);
}

cudaError_t launch_pose_init(Launch L, DevPose* pose, const DevStats* stats, int E) {
  pose_init_kernel<<<1, 32, 0, L.stream>>>(pose, stats, E);
  if (L.counter) ++*L.counter;
  return cudaGetLastError();
}

cudaError_t launch_pose_refresh(Launch L, DevPose* pose, const DevStats* stats) {
  pose_refresh_kernel<<<1, 32, 0, L.stream>>>(pose, stats);
  if (L.counter) ++*L.counter;
  return cudaGetLastError();
}

// Column sums of the per-block partials.  A float64 instruction costs about
// 65 cycles on GB300 whatever the number of active lanes, and dependent ones
// do not overlap, so the sums are arranged by the length of the dependent
// chain in one lane (lane q < 13 adds column q):
// * up to FINALIZE_WARP_ROWS rows, warp 0 adds them alone, in order;
// * up to FINALIZE_SPLIT_ROWS, each of the 8 warps adds every 8th row (warp
//   w: rows w, w + 8, ...) and warp 0 adds the 8 warp sums in order, a chain
//   of rows / 8 + 8 additions instead of rows;
// * beyond that, each thread adds its rows, and each warp two of the 13
//   columns of thread sums.
constexpr int FINALIZE_WARP_ROWS = 16;
constexpr int FINALIZE_SPLIT_ROWS = 512;

// Totals of nblocks rows of 13 partials (fixed order) by warps 0..7 while
// warps 8..11 form the update's first half, then the second half.
constexpr int FINALIZE_THREADS = RED_THREADS + 32 * POSE_PRE_WARPS;

struct FinalizeShared {
  double sh[13][RED_THREADS];
  double tot[13];
  PosePre pre;
  PoseRate rate;
};

__device__ void finalize_body(const double* __restrict__ blockpart, int nblocks, DevPose* ps,
                              const DevStats* __restrict__ st, StepParams sp, int* err, FinalizeShared& F) {
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
  constexpr int NW = RED_THREADS / 32;
  if (nblocks <= FINALIZE_SPLIT_ROWS) {
    // rows in turn by one warp, or every 8th row by each of 8 (FINALIZE_WARP_ROWS)
    const int nw = nblocks <= FINALIZE_WARP_ROWS ? 1 : NW;
    if (warp >= NW) {
      pose_pre(warp - NW, ps, st, sp, F.pre, F.rate);
    } else if (warp < nw && lane < 13) {
      double col = 0.0;
      for (int b = warp; b < nblocks; b += nw) col += blockpart[(size_t)b * 13 + lane];
      F.sh[lane][warp] = col;
    }
    __syncthreads();
    if (warp != 0) return;
    if (lane < 13) {
      double tot = F.sh[lane][0];
      for (int k = 1; k < nw; ++k) tot += F.sh[lane][k];
      F.tot[lane] = tot;
    }
    __syncwarp();
  } else {
    if (warp >= NW) {
      pose_pre(warp - NW, ps, st, sp, F.pre, F.rate);
    } else {
      double v[13];
#pragma unroll
      for (int q = 0; q < 13; ++q) v[q] = 0.0;
      for (int b = threadIdx.x; b < nblocks; b += RED_THREADS) {
#pragma unroll
        for (int q = 0; q < 13; ++q) v[q] += blockpart[(size_t)b * 13 + q];
      }
#pragma unroll
      for (int q = 0; q < 13; ++q) F.sh[q][threadIdx.x] = v[q];
    }
    // each warp adds the threads' sums of columns w, w + 8
    __syncthreads();
    if (warp < NW)
      for (int q = warp; q < 13; q += NW) {
        double t = 0.0;
#pragma unroll
        for (int k = 0; k < RED_THREADS / 32; ++k) t += F.sh[q][k * 32 + lane];
#pragma unroll
        for (int off = 16; off > 0; off >>= 1) t += __shfl_xor_sync(WFULL, t, off);
        if (lane == 0) F.tot[q] = t;
      }
    __syncthreads();
    if (warp != 0) return;
  }
  pose_post(F.tot, ps, st, sp, F.pre, F.rate, err);
}

// Combine and finalize in one block, for templates of at most
// FUSED_MAX_SLOTS padded slots (the latency regime of small problems).
// 1. FUSED_THREADS threads form the points' (f, W_i) from their split
//    partials (point_fw) into shared memory: a thread's points are
//    sequential trips to memory, so more threads than the sums below use
//    shorten that chain.
// 2. The first RED_THREADS threads add them up (thread t: points t,
//    t + RED_THREADS, ... in order, through point_acc), the order a
//    RED_THREADS-thread pass over the points would take.
// 3. The 13 sums are reduced per warp (float64) and across the warps in
//    order by warp 0, and warp 0 updates the pose.
// One launch per iteration instead of two, and no per-block partials.
constexpr int FUSED_THREADS = 512;

__global__ void __launch_bounds__(FUSED_THREADS, 1)
    combine_finalize_kernel(const float4* __restrict__ partial, int S, int mpad, int m,
                            const float4* __restrict__ Y0r, const float* __restrict__ aY32, int g_mode,
                            DevPose* ps, const DevStats* __restrict__ st, StepParams sp, int* err) {
  __shared__ __align__(16) float4 fws[FUSED_MAX_SLOTS];  // (f, W_i) per point
  __shared__ double sh[13][RED_THREADS / 32];
  __shared__ double tot[13];
  __shared__ PosePre pre;
  __shared__ PoseRate rate;
  static_assert(FUSED_THREADS >= FINALIZE_THREADS, "warps for the update's first half");
  const PointFrame fr(ps);
  for (int i = threadIdx.x; i < m; i += FUSED_THREADS)
    fws[i] = point_fw(partial, (size_t)mpad, S, i, Y0r[i], g_mode == 1 ? aY32[i] : 1.f, fr);
  __syncthreads();
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
  if (threadIdx.x >= RED_THREADS) {
    if (warp < FINALIZE_THREADS / 32) pose_pre(warp - RED_THREADS / 32, ps, st, sp, pre, rate);
  } else {
    float acc[13];
#pragma unroll
    for (int q = 0; q < 13; ++q) acc[q] = 0.f;
    for (int i = threadIdx.x; i < m; i += RED_THREADS) point_acc(fws[i], Y0r[i], fr, acc);
    double w[16];
#pragma unroll
    for (int q = 0; q < 13; ++q) w[q] = (double)acc[q];
    w[13] = w[14] = w[15] = 0.0;
    warp_reduce16(w);
    // even lanes hold quantities 0..15 after the reduction; 13..15 are padding
    if ((lane & 1) == 0) {
      const int q = warp_reduce16_slot(lane);
      if (q < 13) sh[q][warp] = w[0];
    }
  }
  __syncthreads();  // all of ps read: warp 0 updates the pose from here
  if (warp != 0) return;
  if (lane < 13) {
    double col = 0.0;
    for (int k = 0; k < RED_THREADS / 32; ++k) col += sh[lane][k];
    tot[lane] = col;
  }
  __syncwarp();
  pose_post(tot, ps, st, sp, pre, rate, err);
}

cudaError_t launch_combine_finalize(Launch L, const float4* partial, int S, int mpad, int m, const float4* Y0r,
                                    const float* aY32, int g_mode, DevPose* pose, const DevStats* stats,
                                    StepParams sp, int* err) {
  combine_finalize_kernel<<<1, FUSED_THREADS, 0, L.stream>>>(partial, S, mpad, m, Y0r, aY32, g_mode, pose, stats,
                                                             sp, err);
  if (L.counter) ++*L.counter;
  return cudaGetLastError();
}

__global__ void __launch_bounds__(FINALIZE_THREADS)
    finalize_kernel(const double* __restrict__ blockpart, int nblocks, DevPose* ps,
                    const DevStats* __restrict__ st, StepParams sp, int* err) {
  __shared__ FinalizeShared F;
  finalize_body(blockpart, nblocks, ps, st, sp, err, F);
}

// ---- p = 1: all iterations from fixed moments ------------------------------
// For p = 1 the per-point sums W_i = sum_j w_ij and S_i = sum_j w_ij X'_j do not
// depend on the pose, so the totals of an iteration are polynomials in the
// pose over 22 fixed sums: with a = aY, u_i = Y0_i - ybar0, A = s R, and
// Y'_i - ybar' = u_i A,
//   F = s1 - m1 A - m0 ybar',          s1 = sum a S, m1 = sum a W u, m0 = sum a W
//   T^T = A^T (N - M2 A - m1^T ybar'), N = sum u^T a S, M2 = sum a W u^T u
// and the total weight is m0.  One pass over the template forms the sums in
// float64; then one block runs every iteration.  (Equal to the per-iteration
// pass up to rounding: that one forms each f_i in float32.)
// Bound: the float64 chain of an iteration, about 4 us.  35,000 x 30,800, 200
// iterations, descriptors included: 1.34 ms (5.8 ms with a combine and a
// finalize launch per iteration).
constexpr int NFIXED = 22;  // m0, m1[3], M2[6] (xx xy xz yy yz zz), s1[3], N[9]
constexpr int FIXED_TPB = 256;

static int fixed_blocks(int m, int num_sms) {
  const int b = (m + FIXED_TPB - 1) / FIXED_TPB;
  return b < 2 * num_sms ? b : 2 * num_sms;
}
size_t fixed_part_bytes(int num_sms) { return (size_t)2 * num_sms * NFIXED * sizeof(double); }

__global__ void __launch_bounds__(FIXED_TPB)
    fixed_moments_kernel(const float4* __restrict__ partial, int S, int mpad, int m, const float4* __restrict__ Y0r,
                         const double* __restrict__ aY64, int g_mode, const DevStats* __restrict__ st,
                         double* __restrict__ part) {
  __shared__ double sh[FIXED_TPB / 32][NFIXED];
  double v[NFIXED];
#pragma unroll
  for (int q = 0; q < NFIXED; ++q) v[q] = 0.0;
  const double y0m[3] = {st->ybar0[0], st->ybar0[1], st->ybar0[2]};
  for (int i = blockIdx.x * FIXED_TPB + threadIdx.x; i < m; i += gridDim.x * FIXED_TPB) {
    const PointSums r = point_sums(partial, (size_t)mpad, S, i);
    const float4 y0 = Y0r[i];
    const double a = g_mode == 1 ? aY64[i] : 1.0;
    const double w = a * ((double)r.Wh - (double)r.Wc);
    const double u[3] = {(double)y0.x - y0m[0], (double)y0.y - y0m[1], (double)y0.z - y0m[2]};
    v[0] += w;
#pragma unroll
    for (int c = 0, f = 4; c < 3; ++c) {
      const double wu = w * u[c], s = a * ((double)r.Sh[c] - (double)r.Sc[c]);
      v[1 + c] += wu;
#pragma unroll
      for (int d = c; d < 3; ++d, ++f) v[f] = fma(wu, u[d], v[f]);
      v[10 + c] += s;
#pragma unroll
      for (int d = 0; d < 3; ++d) v[13 + 3 * d + c] = fma(u[d], s, v[13 + 3 * d + c]);
    }
  }
#pragma unroll
  for (int off = 16; off > 0; off >>= 1)
#pragma unroll
    for (int q = 0; q < NFIXED; ++q) v[q] += __shfl_down_sync(WFULL, v[q], off);
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
  if (lane == 0)
#pragma unroll
    for (int q = 0; q < NFIXED; ++q) sh[warp][q] = v[q];
  __syncthreads();
  if (threadIdx.x < NFIXED) {
    double t = sh[0][threadIdx.x];
#pragma unroll
    for (int w = 1; w < FIXED_TPB / 32; ++w) t += sh[w][threadIdx.x];
    part[(size_t)blockIdx.x * NFIXED + threadIdx.x] = t;
  }
}

// One block, all iterations.  Between two poses only three warps' short
// float64 chains (the totals, s^2 R^T S0 R, the mean and the corrected rotation)
// and warp 0's second half lie on the path; the schedule and the scale of the
// next iteration are formed beside the second half.  Each role has an SM
// scheduler (warp % 4) to itself as far as that goes.
constexpr int FIXED_RUN_THREADS = 256;

__global__ void __launch_bounds__(FIXED_RUN_THREADS)
    fixed_run_kernel(const double* __restrict__ part, int nb, DevPose* pose, const DevStats* __restrict__ stats,
                     StepParams sp, int iters, int* err) {
  __shared__ double mo[NFIXED];
  __shared__ double tot[13];
  __shared__ PosePre pre;
  __shared__ PoseRate rate[2];
  __shared__ bool ok;
  __shared__ DevPose ps;
  __shared__ DevStats st;
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
  for (int q = warp; q < NFIXED; q += FIXED_RUN_THREADS / 32) {
    double t = 0.0;
    for (int b = lane; b < nb; b += 32) t += part[(size_t)b * NFIXED + q];
#pragma unroll
    for (int off = 16; off > 0; off >>= 1) t += __shfl_xor_sync(WFULL, t, off);
    if (lane == 0) mo[q] = t;
  }
  if (threadIdx.x < sizeof(DevPose) / 4) reinterpret_cast<int*>(&ps)[threadIdx.x] = reinterpret_cast<const int*>(pose)[threadIdx.x];
  if (threadIdx.x < sizeof(DevStats) / 4) reinterpret_cast<int*>(&st)[threadIdx.x] = reinterpret_cast<const int*>(stats)[threadIdx.x];
  __syncthreads();
  // lane (row, col) of the totals' warp: rows 0..2 are (N - M2 A - m1^T ybar'), row 3 is F
  const int row = min(lane / 3, 3), col = lane < 12 ? lane % 3 : 2;
  constexpr int SYM[9] = {0, 1, 2, 1, 3, 4, 2, 4, 5};
  double P[3], N, U;
#pragma unroll
  for (int k = 0; k < 3; ++k) P[k] = row < 3 ? mo[4 + SYM[row * 3 + k]] : mo[1 + k];
  N = row < 3 ? mo[13 + row * 3 + col] : mo[10 + col];
  U = row < 3 ? mo[1 + row] : mo[0];
  if (threadIdx.x == 0) tot[3] = mo[0];
  const int it0 = ps.it, E = ps.E;
  if (warp == 4) pose_schedule(ps.it, ps.E, sp, rate[0]);
  if (warp == 5) pose_scale(ps.s, &st, sp, rate[0]);
  for (int it = 0; it < iters; ++it) {
    PoseRate& now = rate[it & 1];
    PoseRate& next = rate[(it + 1) & 1];
    if (warp == 2) pose_pre(2, &ps, &st, sp, pre, now);
    if (warp == 3) pose_pre(3, &ps, &st, sp, pre, now);
    if (warp == 1) {
      const double R = ps.R[lane3().q];  // entry (r, c) in lanes 0..8
      const double A = ps.s * R;
      const double ybs =
          fma(ps.s, fma(st.ybar0[2], ps.R[6 + col], fma(st.ybar0[1], ps.R[3 + col], st.ybar0[0] * ps.R[col])), ps.t[col]) -
          st.xbar[col];
      double v = fma(-U, ybs, N);
#pragma unroll
      for (int k = 0; k < 3; ++k) v = fma(-P[k], wget(A, k * 3 + col), v);
      // T[a][b] = sum_c K[c][a] A[c][b]: lane (a, b) in 0..8
      const int a = min(lane, 8) / 3, b = min(lane, 8) % 3;
      double T = wget(v, a) * wget(A, b);
      T = fma(wget(v, 3 + a), wget(A, 3 + b), T);
      T = fma(wget(v, 6 + a), wget(A, 6 + b), T);
      if (lane < 9) tot[4 + lane] = T;
      else if (lane < 12) tot[col] = v;
    }
    __syncthreads();
    if (warp == 0) {
      const bool moved = pose_post(tot, &ps, &st, sp, pre, now, err, false);
      if (lane == 0) ok = moved;
    } else if (warp == 5) {
      pose_schedule(it0 + it + 1, E, sp, next);
    } else if (warp == 6) {
      pose_scale(now.sn, &st, sp, next);
    }
    __syncthreads();
    if (!ok) {  // the pose was kept, and so is its scale
      if (warp == 6) pose_scale(ps.s, &st, sp, next);
      __syncthreads();
    }
  }
  if (threadIdx.x == 0) refresh_pose(&ps, &st);
  __syncthreads();
  if (threadIdx.x < sizeof(DevPose) / 4) reinterpret_cast<int*>(pose)[threadIdx.x] = reinterpret_cast<const int*>(&ps)[threadIdx.x];
}

cudaError_t launch_fixed_moments(Launch L, const float4* partial, int S, int mpad, int m, const float4* Y0r,
                                 const double* aY64, int g_mode, const DevStats* stats, int num_sms, double* part) {
  fixed_moments_kernel<<<fixed_blocks(m, num_sms), FIXED_TPB, 0, L.stream>>>(partial, S, mpad, m, Y0r, aY64, g_mode,
                                                                            stats, part);
  if (L.counter) ++*L.counter;
  return cudaGetLastError();
}

cudaError_t launch_fixed_run(Launch L, const double* part, int m, int num_sms, DevPose* pose, const DevStats* stats,
                             StepParams sp, int iters, int* err) {
  fixed_run_kernel<<<1, FIXED_RUN_THREADS, 0, L.stream>>>(part, fixed_blocks(m, num_sms), pose, stats, sp, iters, err);
  if (L.counter) ++*L.counter;
  return cudaGetLastError();
}

// One block per pair of a batch.
__global__ void __launch_bounds__(FINALIZE_THREADS)
    finalize_multi_kernel(const double* __restrict__ blockpart, const BatchPair* __restrict__ pairs,
                          DevPose* poses, const DevStats* __restrict__ stats, StepParams sp, int* err) {
  __shared__ FinalizeShared F;
  const BatchPair& bp = pairs[blockIdx.x];
  StepParams spp = sp;
  spp.M = (int)bp.m;
  finalize_body(blockpart + (size_t)bp.cblk0 * 13, bp.ncblk, poses + blockIdx.x, stats + blockIdx.x, spp, err, F);
}

cudaError_t launch_finalize_multi(Launch L, const double* blockpart, const BatchPair* pairs, int npairs,
                                  DevPose* poses, const DevStats* stats, StepParams sp, int* err) {
  finalize_multi_kernel<<<npairs, FINALIZE_THREADS, 0, L.stream>>>(blockpart, pairs, poses, stats, sp, err);
  if (L.counter) ++*L.counter;
  return cudaGetLastError();
}

__global__ void pose_init_multi_kernel(DevPose* poses, const DevStats* stats, int npairs, int E) {
  const int p = blockIdx.x * blockDim.x + threadIdx.x;
  if (p >= npairs) return;
  DevPose* ps = poses + p;
  for (int q = 0; q < 9; ++q) ps->R[q] = (q % 4 == 0) ? 1.0 : 0.0;
  ps->t[0] = ps->t[1] = ps->t[2] = 0.0;
  ps->s = 1.0;
  ps->it = 0;
  ps->E = E;
  ps->degenerate = 0;
  refresh_pose(ps, stats + p);
}

cudaError_t launch_pose_init_multi(Launch L, DevPose* poses, const DevStats* stats, int npairs, int E) {
  pose_init_multi_kernel<<<(npairs + 127) / 128, 128, 0, L.stream>>>(poses, stats, npairs, E);
  if (L.counter) ++*L.counter;
  return cudaGetLastError();
}

cudaError_t launch_finalize(Launch L, const double* blockpart, int nblocks, DevPose* pose,
                            const DevStats* stats, StepParams sp, int* err) {
  finalize_kernel<<<1, FINALIZE_THREADS, 0, L.stream>>>(blockpart, nblocks, pose, stats, sp, err);
  if (L.counter) ++*L.counter;
  return cudaGetLastError();
}

// moved = s Y0 R + t (Eq. 9), float64 arithmetic, float32 output [m][3]
__global__ void apply_kernel(const float4* __restrict__ Y4, int m, const DevPose* __restrict__ ps,
                             float* __restrict__ out) {
  const int i = blockIdx.x * blockDim.x + threadIdx.x;
  if (i >= m) return;
  const float4 y = Y4[i];
  for (int c = 0; c < 3; ++c) {
    const double v = ps->s * ((double)y.x * ps->R[c] + (double)y.y * ps->R[3 + c] +
                              (double)y.z * ps->R[6 + c]) + ps->t[c];
    out[(size_t)i * 3 + c] = (float)v;
  }
}

cudaError_t launch_apply(Launch L, const float4* Y4, int m, const DevPose* pose, float* out) {
  if (m <= 0) return cudaSuccess;
  apply_kernel<<<(m + 255) / 256, 256, 0, L.stream>>>(Y4, m, pose, out);
  if (L.counter) ++*L.counter;
  return cudaGetLastError();
}

}  // namespace scgr
