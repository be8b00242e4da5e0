// Shape-weighted potential and its adjoint (the differentiation form).
//
// U = sum_i sum_j g(s_ij) d_ij^(p+1) / (p+1) is the potential whose negative
// gradient with respect to Y_i is the force of Eq. 5 (descriptors fixed).
// With Y = s Y0 R(omega) + t (row vectors, R = exp([omega]_x)^T) the pose
// gradient follows from G_i = dU/dY_i = -f_i:
//   dU/dt = sum_i G_i,   dU/ds = sum_i G_i . (Y0_i R),
//   dU/dR = s sum_i Y0_i^T G_i,   dU/dY0_i = s G_i R^T,
// and for the axis-angle the SO(3) right Jacobian J_r: perturbing
// R_col(omega + delta) = R_col(omega) exp([J_r(omega) delta]_x) gives
// dU/domega = J_r(omega)^T w, where w is the axial vector of the skew part of
// B = (dU/dR) R_col (w_c = sum_ab eps_abc B_ab).
//
// U and the adjoint's per-point sums come from one pass over the pairs:
// w_ij = g d^(p-1) gives both w d^2 = g d^(p+1) for U and the sums of the force
// kernel (sum w, sum w X') for G_i; without gradients only U is summed.  Tiles
// are recomputed (no N x M storage), the chain-rule terms reduced in float64 in
// a fixed order.  The 3x3 algebra of the pose (Rodrigues' formula, J_r) is done
// by the host, which has pose7 and reads the totals anyway.
#include <cmath>

#include "common.cuh"
#include "pair.cuh"
#include "pointsum.cuh"

namespace scgr {

__device__ __forceinline__ void tpoint(const float4 y0, const float* A, const float* b, float& yx,
                                       float& yy, float& yz) {
  template_point(y0, A, b, yx, yy, yz);
}

// The pose of an evaluation and its float32 map (one warp).
__global__ void pose_from_host_kernel(const HostPose hp, DevPose* ps, const DevStats* __restrict__ st) {
  const int l = threadIdx.x;
  if (l < 9) {
    ps->R[l] = hp.R[l];
    ps->A[l] = (float)(hp.s * hp.R[l]);
  }
  if (l < 3) {
    ps->t[l] = hp.t[l];
    ps->b[l] = (float)(hp.t[l] - st->xbar[l]);
    const double yb = hp.s * (st->ybar0[0] * hp.R[l] + st->ybar0[1] * hp.R[3 + l] + st->ybar0[2] * hp.R[6 + l]) + hp.t[l];
    set_ybs(ps, l, yb - st->xbar[l]);
  }
  if (l == 0) {
    ps->s = hp.s;
    ps->it = 0;
    ps->E = 1;
    ps->degenerate = 0;
  }
}

// ---- the pair pass -----------------------------------------------------------

// Reference points (j, j+1) against one template point: U += w d^2, and with
// GRAD W += w, S += w X'.
template <int PM, bool GRAD>
__device__ __forceinline__ void potential_pair2(u64 xv, u64 yv, u64 zv, u64 nv, u64 av, u64 lv, u64 mx, u64 my, u64 mz,
                                                u64 ny, u64 ah, u64 nq, u64& U, u64& W, u64& Sx, u64& Sy, u64& Sz) {
  u64 d2 = add2(nv, ny);
  d2 = fma2(xv, mx, d2);
  d2 = fma2(yv, my, d2);
  d2 = fma2(zv, mz, d2);
  const u64 u = sub2(av, ah);
  const u64 ep = fma2(u, u, lv);
  float e0, e1, q0, q1;
  u64 w;
  if (PM == 0) {
    upk2(d2, q0, q1);
    upk2(fma2(nq, pk2(lg2_approx(fabsf(q0)), lg2_approx(fabsf(q1))), ep), e0, e1);
    w = pk2(ex2_neg(e0), ex2_neg(e1));
  } else {
    upk2(ep, e0, e1);
    w = pk2(ex2_neg(e0), ex2_neg(e1));
    if (PM == 2) {
      upk2(d2, q0, q1);
      w = mul2(w, pk2(sqrt_approx(fabsf(q0)), sqrt_approx(fabsf(q1))));
    } else if (PM == 3) {
      w = mul2(w, d2);
    }
  }
  U = fma2(w, d2, U);
  if (GRAD) {
    W = add2(W, w);
    Sx = fma2(w, xv, Sx);
    Sy = fma2(w, yv, Sy);
    Sz = fma2(w, zv, Sz);
  }
}

// Template points [blockIdx.x * P * POT_TPB, ...) against the reference tiles
// of split blockIdx.y, at pose *ps.  The block's sum of aY U goes to upart in
// float64; with GRAD the points' (sum w, sum w X') to partial[split][mpad].
// Bound and layout are the force kernel's: ex2 and sqrt on the special-function
// unit (10.6 pairs per clock per SM), 12 FP32 lane operations a pair with
// gradients, 8 without; packed pairs, broadcast tiles, Kahan sums across tiles.
// Value and gradients at 50,000 x 50,000, p = 2: this pass 1.1 ms, the whole call
// through autograd 1.38 ms (3.6 ms as two general-p passes and a float64 combine;
// 2.3 ms with this pass run twice, in forward and again in backward).
constexpr int POT_TPB = 128;

template <int P, int PM, bool GRAD>
__global__ void __launch_bounds__(POT_TPB)
    potential_tile_kernel(const float* __restrict__ Xr, const float* __restrict__ XA, int ntiles, int tiles_per_split,
                          const float4* __restrict__ Y0r, int mpad, int m, const float* __restrict__ aY32, int g_mode,
                          const DevPose* __restrict__ ps, float qexp, float4* __restrict__ partial,
                          double* __restrict__ upart) {
  constexpr int TJ = FORCE_TJ, Q4 = TJ / 4, NV = GRAD ? 5 : 1;
  __shared__ __align__(16) float sT[6][TJ];
  __shared__ double shu[POT_TPB / 32];
  const int i0 = blockIdx.x * (P * POT_TPB) + threadIdx.x;
  float A[9], b[3];
#pragma unroll
  for (int q = 0; q < 9; ++q) A[q] = ps->A[q];
#pragma unroll
  for (int q = 0; q < 3; ++q) b[q] = ps->b[q];
  u64 mx[P], my[P], mz[P], ny[P], ah[P];
  float h[P][NV], c[P][NV];
#pragma unroll
  for (int q = 0; q < P; ++q) {
    const float4 y0 = Y0r[i0 + q * POT_TPB];
    float x, y, z;
    tpoint(y0, A, b, x, y, z);
    const float n = fmaf(z, z, fmaf(y, y, x * x));
    mx[q] = pk2(-2.f * x, -2.f * x);
    my[q] = pk2(-2.f * y, -2.f * y);
    mz[q] = pk2(-2.f * z, -2.f * z);
    ny[q] = pk2(n, n);
    ah[q] = pk2(y0.w, y0.w);
#pragma unroll
    for (int v = 0; v < NV; ++v) h[q][v] = c[q][v] = 0.f;
  }
  const u64 nq = pk2(-qexp, -qexp);
  const int t0 = blockIdx.y * tiles_per_split, t1 = min(ntiles, t0 + tiles_per_split);
  for (int t = t0; t < t1; ++t) {
    __syncthreads();
    const float4* g4 = reinterpret_cast<const float4*>(Xr + (size_t)t * 4 * TJ);
    const float4* a4 = reinterpret_cast<const float4*>(XA + (size_t)t * 2 * TJ);
#pragma unroll
    for (int u = threadIdx.x; u < 6 * Q4; u += POT_TPB)
      *reinterpret_cast<float4*>(&sT[u / Q4][4 * (u % Q4)]) = u < 4 * Q4 ? g4[u] : a4[u - 4 * Q4];
    __syncthreads();
    u64 acc[P][5];
#pragma unroll
    for (int q = 0; q < P; ++q)
#pragma unroll
      for (int v = 0; v < 5; ++v) acc[q][v] = 0ull;
#pragma unroll 2
    for (int jq = 0; jq < TJ; jq += 4) {
      const ulonglong2 X = *reinterpret_cast<const ulonglong2*>(&sT[0][jq]);
      const ulonglong2 Y = *reinterpret_cast<const ulonglong2*>(&sT[1][jq]);
      const ulonglong2 Z = *reinterpret_cast<const ulonglong2*>(&sT[2][jq]);
      const ulonglong2 N = *reinterpret_cast<const ulonglong2*>(&sT[3][jq]);
      const ulonglong2 Av = *reinterpret_cast<const ulonglong2*>(&sT[4][jq]);
      const ulonglong2 Lv = *reinterpret_cast<const ulonglong2*>(&sT[5][jq]);
#pragma unroll
      for (int q = 0; q < P; ++q)
        potential_pair2<PM, GRAD>(X.x, Y.x, Z.x, N.x, Av.x, Lv.x, mx[q], my[q], mz[q], ny[q], ah[q], nq, acc[q][0],
                                  acc[q][1], acc[q][2], acc[q][3], acc[q][4]);
#pragma unroll
      for (int q = 0; q < P; ++q)
        potential_pair2<PM, GRAD>(X.y, Y.y, Z.y, N.y, Av.y, Lv.y, mx[q], my[q], mz[q], ny[q], ah[q], nq, acc[q][0],
                                  acc[q][1], acc[q][2], acc[q][3], acc[q][4]);
    }
#pragma unroll
    for (int q = 0; q < P; ++q)
#pragma unroll
      for (int v = 0; v < NV; ++v) {
        float l0, l1;
        upk2(acc[q][v], l0, l1);
        kahan_add(h[q][v], c[q][v], l0 + l1);
      }
  }
  double u = 0.0;
#pragma unroll
  for (int q = 0; q < P; ++q) {
    const int i = i0 + q * POT_TPB;
    if (i < m) u += (g_mode == 1 ? (double)aY32[i] : 1.0) * ((double)h[q][0] - (double)c[q][0]);
    if constexpr (GRAD)
      partial[(size_t)blockIdx.y * mpad + i] =
          make_float4(h[q][1] - c[q][1], h[q][2] - c[q][2], h[q][3] - c[q][3], h[q][4] - c[q][4]);
  }
#pragma unroll
  for (int off = 16; off > 0; off >>= 1) u += __shfl_down_sync(0xffffffffu, u, off);
  if ((threadIdx.x & 31) == 0) shu[threadIdx.x >> 5] = u;
  __syncthreads();
  if (threadIdx.x == 0) {
    double t = shu[0];
#pragma unroll
    for (int w = 1; w < POT_TPB / 32; ++w) t += shu[w];
    upart[(size_t)blockIdx.y * gridDim.x + blockIdx.x] = t;
  }
}

template <int PM>
static void launch_potential_pm(Launch L, const ForcePlan& fp, bool grad, const float* Xr, const float* XA, int ntiles,
                                const float4* Y0r, int mpad, int m, const float* aY32, int g_mode, const DevPose* ps,
                                float qexp, float4* partial, double* upart) {
  const dim3 grid(fp.iblocks, fp.splits);
  const auto k = fp.P == 2 ? (grad ? potential_tile_kernel<2, PM, true> : potential_tile_kernel<2, PM, false>)
                           : (grad ? potential_tile_kernel<1, PM, true> : potential_tile_kernel<1, PM, false>);
  k<<<grid, POT_TPB, 0, L.stream>>>(Xr, XA, ntiles, fp.tiles_per_split, Y0r, mpad, m, aY32, g_mode, ps, qexp, partial,
                                    upart);
}

// The pair pass of the potential under plan fp (1 or 2 points x 128 threads).
cudaError_t launch_potential(Launch L, const ForcePlan& fp, bool grad, const float4* Xr, const float2* XA, int ntiles,
                             const float4* Y0r, int mpad, int m, const float* aY32, int g_mode, const DevPose* ps,
                             float qexp, float4* partial, double* upart) {
  const float* xr = reinterpret_cast<const float*>(Xr);
  const float* xa = reinterpret_cast<const float*>(XA);
  const auto launch = fp.pmode == 1   ? launch_potential_pm<1>
                      : fp.pmode == 3 ? launch_potential_pm<3>
                      : fp.pmode == 0 ? launch_potential_pm<0>
                                      : launch_potential_pm<2>;
  launch(L, fp, grad, xr, xa, ntiles, Y0r, mpad, m, aY32, g_mode, ps, qexp, partial, upart);
  if (L.counter) ++*L.counter;
  return cudaGetLastError();
}

// Per point: G_i = -f_i from the split partials (added with Kahan
// compensation, the rest in float64); the template-coordinate gradient s G_i R^T;
// per-block chain-rule sums (sum G, sum G.(Y0 R), sum Y0^T G).
__global__ void __launch_bounds__(RED_THREADS)
    adjoint_combine_kernel(const float4* __restrict__ partial, int S, int mpad, int m,
                           const float4* __restrict__ Y0r, const double* __restrict__ aY64,
                           int g_mode, const DevPose* __restrict__ ps, float* __restrict__ grad_xyz,
                           double* __restrict__ blockpart) {
  __shared__ double sh[RED_THREADS / 32][16];
  const int i = blockIdx.x * RED_THREADS + threadIdx.x;
  double v[16];
#pragma unroll
  for (int q = 0; q < 16; ++q) v[q] = 0.0;
  if (i < m) {
    const PointSums r = point_sums(partial, (size_t)mpad, S, i);
    const double W = (double)r.Wh - (double)r.Wc;
    float A[9], b[3];
#pragma unroll
    for (int q = 0; q < 9; ++q) A[q] = ps->A[q];
#pragma unroll
    for (int q = 0; q < 3; ++q) b[q] = ps->b[q];
    const float4 y0 = Y0r[i];
    float y[3];
    tpoint(y0, A, b, y[0], y[1], y[2]);
    const double ay = g_mode == 1 ? aY64[i] : 1.0;
    const double Y0d[3] = {(double)y0.x, (double)y0.y, (double)y0.z};
    double R[9], G[3];
#pragma unroll
    for (int q = 0; q < 9; ++q) R[q] = ps->R[q];
    // G = dU/dY = -f = aY (Y' sum w - sum w X')
#pragma unroll
    for (int c = 0; c < 3; ++c) {
      G[c] = ay * fma((double)y[c], W, (double)r.Sc[c] - (double)r.Sh[c]);
      v[c] = G[c];
    }
    double gY[3];  // G R^T: dU/dY0 = s gY, and G.(Y0 R) = Y0 . gY
#pragma unroll
    for (int a = 0; a < 3; ++a) gY[a] = fma(G[2], R[a * 3 + 2], fma(G[1], R[a * 3 + 1], G[0] * R[a * 3]));
    v[3] = fma(Y0d[2], gY[2], fma(Y0d[1], gY[1], Y0d[0] * gY[0]));
#pragma unroll
    for (int a = 0; a < 3; ++a)
#pragma unroll
      for (int bb = 0; bb < 3; ++bb) v[4 + 3 * a + bb] = Y0d[a] * G[bb];
    if (grad_xyz) {
      const double s = ps->s;
#pragma unroll
      for (int a = 0; a < 3; ++a) grad_xyz[(size_t)i * 3 + a] = (float)(s * gY[a]);
    }
  }
  warp_reduce16(v);
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
  if ((lane & 1) == 0) sh[warp][warp_reduce16_slot(lane)] = v[0];
  __syncthreads();
  if (threadIdx.x < 13) {
    double t = sh[0][threadIdx.x];
#pragma unroll
    for (int w = 1; w < RED_THREADS / 32; ++w) t += sh[w][threadIdx.x];
    blockpart[(size_t)blockIdx.x * 13 + threadIdx.x] = t;
  }
}

// One block: out[0] = sum of nu doubles of upart, out[1 .. 13] = column sums of
// nb rows of blockpart (nb = 0: none), out[14] = the device error word; all in
// a fixed order.
constexpr int PF_T = 512;
__global__ void __launch_bounds__(PF_T)
    potential_finish_kernel(const double* __restrict__ upart, int64_t nu, const double* __restrict__ blockpart, int nb,
                            const int* __restrict__ err, double* __restrict__ out) {
  __shared__ double sh[PF_T / 32][14];
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
  double u = 0.0;
  for (int64_t q = threadIdx.x; q < nu; q += PF_T) u += upart[q];
#pragma unroll
  for (int off = 16; off > 0; off >>= 1) u += __shfl_xor_sync(0xffffffffu, u, off);
  double col = 0.0;
  if (lane < 13)
    for (int b = warp; b < nb; b += PF_T / 32) col += blockpart[(size_t)b * 13 + lane];
  if (lane < 13) sh[warp][1 + lane] = col;
  if (lane == 0) sh[warp][0] = u;
  __syncthreads();
  if (threadIdx.x < 14) {
    double t = sh[0][threadIdx.x];
    for (int w = 1; w < PF_T / 32; ++w) t += sh[w][threadIdx.x];
    out[threadIdx.x] = t;
  }
  if (threadIdx.x == 32) out[14] = (double)*err;
}

cudaError_t launch_potential_finish(Launch L, const double* upart, int64_t nu, const double* blockpart, int nb,
                                    const int* err, double* out) {
  potential_finish_kernel<<<1, PF_T, 0, L.stream>>>(upart, nu, blockpart, nb, err, out);
  if (L.counter) ++*L.counter;
  return cudaGetLastError();
}

// One block: fixed-order column sums of [nb][13] partials.
__global__ void __launch_bounds__(RED_THREADS) column_sum13_kernel(const double* __restrict__ part, int nb,
                                                                   double* __restrict__ out) {
  __shared__ double sh[13][RED_THREADS];
  double v[13];
#pragma unroll
  for (int q = 0; q < 13; ++q) v[q] = 0.0;
  for (int b = threadIdx.x; b < nb; b += RED_THREADS) {
#pragma unroll
    for (int q = 0; q < 13; ++q) v[q] += part[(size_t)b * 13 + q];
  }
  block_sum<13>(v, sh);
  if (threadIdx.x == 0) {
#pragma unroll
    for (int q = 0; q < 13; ++q) out[q] = v[q];
  }
}

// ---- vector-Jacobian product of the force field ---------------------------
// f_i depends on Y_i only (X fixed, descriptors fixed), so dF/dY is block
// diagonal with J_ii = -aY sum_j w_ij [I + (p - 1) r r^T / d^2], r = Y_i - X_j,
// w_ij = g d^(p-1).  grad_i = J_ii v_i (J_ii is symmetric).
//
// Per point only C = sum_j c_ij r r^T with c = w / d^2 = g d^(p-3) is
// accumulated: its trace is sum_j w (r r^T / d^2 has trace 1), so
// J = -aY [tr(C) I + (p - 1) C].  A coincident pair has r = 0 and adds
// nothing, as its w = 0 for p > 1 asks.  For p = 1, J = -aY (sum_j w) I with
// w = g also for coincident pairs, so that form sums w alone (C[0]).
//
// Bound: the FP32 pipe.  A pair costs 18 FP32 lane operations (3 differences,
// 3 for d^2, 2 for the exponent, 1 weight, 3 + 6 for the products and sums)
// and two special-function results (ex2 and rsqrt for p = 2): 126 / 18 = 7
// pairs per clock per SM, 2.2e12 pairs/s.  The layout is the force kernel's:
// reference tiles in shared memory read as 128-bit broadcasts, two reference
// points per packed .f32x2 instruction, P template points per thread (their
// independent chains hide the special-function latency), the reference range
// split over grid.y so that a small template still fills the GPU, and the
// tile sums added across tiles with Kahan compensation.  Measured on GB300 at
// 10,007 x 9,001, p = 2: 88 us a call (5.2 ms with one scalar thread per
// template point, no split, and exp2f, log2f and a division per pair); the
// error against float64 went from 2.5e-7 to 1.4e-7.
constexpr int VJP_TPB = 128;
constexpr int VJP_NC = 6;                 // C: xx xy xz yy yz zz
constexpr float VJP_D2_MIN = 1e-37f;      // keeps rsqrt and lg2 of d^2 = 0 finite (the products with r are 0)

// Reference points (j, j+1) against one template point.  PM = 1, 2, 3: p = PM;
// 0: general p, with c = 2^(e2 log2 d^2 - ep), e2 = (p - 3) / 2 (nq = -e2).
template <int PM>
__device__ __forceinline__ void vjp_pair2(u64 xv, u64 yv, u64 zv, u64 av, u64 lv, u64 yx, u64 yy, u64 yz, u64 ah,
                                          u64 nq, u64 (&C)[VJP_NC]) {
  const u64 u = sub2(av, ah);
  const u64 ep = fma2(u, u, lv);  // u^2 - L: the pose-free factor is 2^-ep
  float e0, e1;
  if (PM == 1) {
    upk2(ep, e0, e1);
    C[0] = add2(C[0], pk2(ex2_neg(e0), ex2_neg(e1)));
    return;
  }
  const u64 rx = sub2(yx, xv), ry = sub2(yy, yv), rz = sub2(yz, zv);
  u64 c;
  if (PM == 3) {
    upk2(ep, e0, e1);
    c = pk2(ex2_neg(e0), ex2_neg(e1));
  } else {
    float q0, q1;
    upk2(fma2(rz, rz, fma2(ry, ry, mul2(rx, rx))), q0, q1);
    q0 = fmaxf(q0, VJP_D2_MIN);
    q1 = fmaxf(q1, VJP_D2_MIN);
    if (PM == 2) {
      upk2(ep, e0, e1);
      c = mul2(pk2(ex2_neg(e0), ex2_neg(e1)), pk2(rsqrt_approx(q0), rsqrt_approx(q1)));
    } else {
      upk2(fma2(nq, pk2(lg2_approx(q0), lg2_approx(q1)), ep), e0, e1);
      c = pk2(ex2_neg(e0), ex2_neg(e1));
    }
  }
  const u64 cx = mul2(c, rx), cy = mul2(c, ry), cz = mul2(c, rz);
  C[0] = fma2(cx, rx, C[0]);
  C[1] = fma2(cx, ry, C[1]);
  C[2] = fma2(cx, rz, C[2]);
  C[3] = fma2(cy, ry, C[3]);
  C[4] = fma2(cy, rz, C[4]);
  C[5] = fma2(cz, rz, C[5]);
}

// grad_i = -aY [sum_w v + (p - 1) C v] in float64.
__device__ __forceinline__ void vjp_write(int i, const double (&C)[VJP_NC], double pm1, double ay,
                                          const float* __restrict__ v, float* __restrict__ grad) {
  const double W = pm1 == 0.0 ? C[0] : C[0] + C[3] + C[5];
  const double vx = v[3 * (size_t)i], vy = v[3 * (size_t)i + 1], vz = v[3 * (size_t)i + 2];
  double bx = 0.0, by = 0.0, bz = 0.0;
  if (pm1 != 0.0) {
    bx = pm1 * (C[0] * vx + C[1] * vy + C[2] * vz);
    by = pm1 * (C[1] * vx + C[3] * vy + C[4] * vz);
    bz = pm1 * (C[2] * vx + C[4] * vy + C[5] * vz);
  }
  grad[3 * (size_t)i] = (float)(-ay * (W * vx + bx));
  grad[3 * (size_t)i + 1] = (float)(-ay * (W * vy + by));
  grad[3 * (size_t)i + 2] = (float)(-ay * (W * vz + bz));
}

// Template points [blockIdx.x * P * VJP_TPB, ...) against the reference tiles
// of split blockIdx.y.  One split: the gradient is written here; several: the
// sums go to part[split][component][mpad] for vjp_combine_kernel.
template <int P, int PM>
__global__ void __launch_bounds__(VJP_TPB)
    force_vjp_kernel(const float* __restrict__ Xr, const float* __restrict__ XA, int ntiles, int tiles_per_split,
                     const float4* __restrict__ Y0r, int mpad, const double* __restrict__ aY64, int g_mode, int m,
                     const DevPose* __restrict__ ps, double pm1, const float* __restrict__ v,
                     float* __restrict__ grad, float* __restrict__ part) {
  constexpr int TJ = FORCE_TJ;
  constexpr int Q4 = TJ / 4;
  constexpr int NC = PM == 1 ? 1 : VJP_NC;
  __shared__ __align__(16) float sT[5][TJ];
  const int i0 = blockIdx.x * (P * VJP_TPB) + threadIdx.x;
  float A[9], b[3];
#pragma unroll
  for (int q = 0; q < 9; ++q) A[q] = ps->A[q];
#pragma unroll
  for (int q = 0; q < 3; ++q) b[q] = ps->b[q];
  u64 yx[P], yy[P], yz[P], ah[P];
#pragma unroll
  for (int q = 0; q < P; ++q) {
    const int i = i0 + q * VJP_TPB;
    const float4 y0 = Y0r[i < m ? i : m - 1];
    float x, y, z;
    tpoint(y0, A, b, x, y, z);
    yx[q] = pk2(x, x);
    yy[q] = pk2(y, y);
    yz[q] = pk2(z, z);
    ah[q] = pk2(y0.w, y0.w);
  }
  const float e2 = (float)(0.5 * (pm1 - 2.0));
  const u64 nq = pk2(-e2, -e2);
  float h[P][NC], k[P][NC];
#pragma unroll
  for (int q = 0; q < P; ++q)
#pragma unroll
    for (int c = 0; c < NC; ++c) h[q][c] = k[q][c] = 0.f;
  const int t0 = blockIdx.y * tiles_per_split;
  const int t1 = min(ntiles, t0 + tiles_per_split);
  for (int t = t0; t < t1; ++t) {
    __syncthreads();
    const float4* g4 = reinterpret_cast<const float4*>(Xr + (size_t)t * 4 * TJ);  // x, y, z (and |X'|^2, not used)
    const float4* a4 = reinterpret_cast<const float4*>(XA + (size_t)t * 2 * TJ);  // a_hat, -L
#pragma unroll
    for (int u = threadIdx.x; u < 5 * Q4; u += VJP_TPB)
      *reinterpret_cast<float4*>(&sT[u / Q4][4 * (u % Q4)]) = u < 3 * Q4 ? g4[u] : a4[u - 3 * Q4];
    __syncthreads();
    u64 C[P][VJP_NC];
#pragma unroll
    for (int q = 0; q < P; ++q)
#pragma unroll
      for (int c = 0; c < VJP_NC; ++c) C[q][c] = 0ull;
    constexpr int UNR = P == 1 ? 2 : 1;
#pragma unroll UNR
    for (int jq = 0; jq < TJ; jq += 4) {
      const ulonglong2 X = *reinterpret_cast<const ulonglong2*>(&sT[0][jq]);
      const ulonglong2 Y = *reinterpret_cast<const ulonglong2*>(&sT[1][jq]);
      const ulonglong2 Z = *reinterpret_cast<const ulonglong2*>(&sT[2][jq]);
      const ulonglong2 Av = *reinterpret_cast<const ulonglong2*>(&sT[3][jq]);
      const ulonglong2 Lv = *reinterpret_cast<const ulonglong2*>(&sT[4][jq]);
#pragma unroll
      for (int q = 0; q < P; ++q) {
        vjp_pair2<PM>(X.x, Y.x, Z.x, Av.x, Lv.x, yx[q], yy[q], yz[q], ah[q], nq, C[q]);
        vjp_pair2<PM>(X.y, Y.y, Z.y, Av.y, Lv.y, yx[q], yy[q], yz[q], ah[q], nq, C[q]);
      }
    }
#pragma unroll
    for (int q = 0; q < P; ++q)
#pragma unroll
      for (int c = 0; c < NC; ++c) {
        float l0, l1;
        upk2(C[q][c], l0, l1);
        kahan_add(h[q][c], k[q][c], l0 + l1);
      }
  }
#pragma unroll
  for (int q = 0; q < P; ++q) {
    const int i = i0 + q * VJP_TPB;
    if (i >= m) continue;
    if (gridDim.y == 1) {
      double C[VJP_NC];
#pragma unroll
      for (int c = 0; c < VJP_NC; ++c) C[c] = c < NC ? (double)h[q][c < NC ? c : 0] - (double)k[q][c < NC ? c : 0] : 0.0;
      vjp_write(i, C, pm1, g_mode == 1 ? aY64[i] : 1.0, v, grad);
    } else {
#pragma unroll
      for (int c = 0; c < NC; ++c) part[((size_t)blockIdx.y * NC + c) * mpad + i] = h[q][c] - k[q][c];
    }
  }
}

// The splits of one point added in order in float64, then its gradient.
__global__ void __launch_bounds__(VJP_TPB)
    vjp_combine_kernel(const float* __restrict__ part, int S, int nc, int mpad, const double* __restrict__ aY64,
                       int g_mode, int m, double pm1, const float* __restrict__ v, float* __restrict__ grad) {
  const int i = blockIdx.x * VJP_TPB + threadIdx.x;
  if (i >= m) return;
  double C[VJP_NC] = {0, 0, 0, 0, 0, 0};
  for (int s = 0; s < S; ++s) {
#pragma unroll
    for (int c = 0; c < VJP_NC; ++c)
      if (c < nc) C[c] += (double)part[((size_t)s * nc + c) * mpad + i];
  }
  vjp_write(i, C, pm1, g_mode == 1 ? aY64[i] : 1.0, v, grad);
}

// Splits of the reference range: enough blocks for about eight per SM (two
// waves of the four to five that are resident), at least one tile each, and at
// most 4 / nc times the force pass's splits by its own rule (force_splits), which
// keeps a block's run of tiles long enough to pay for its start (10,007 x 9,001,
// p = 2: 8 splits of 5 tiles, 1 point a thread 88 us; 20 of 2 tiles, 2 points 107
// us).  With few blocks even so, one template point per thread instead of two.  From the sizes
// alone, so that the same call gives the same bits whatever the context has held
// before and whatever knobs shape the force pass.
VjpPlan plan_vjp(int64_t m, int64_t npad, double p, int num_sms, int force_splits) {
  const int64_t want = 8 * (int64_t)num_sms, ntiles = npad / FORCE_TJ;
  VjpPlan v;
  v.nc = p == 1.0 ? 1 : VJP_NC;
  int64_t most = 4 * (int64_t)force_splits / v.nc;
  most = most < 1 ? 1 : most < ntiles ? most : ntiles;
  const int64_t b2 = (m + 2 * VJP_TPB - 1) / (2 * VJP_TPB), b1 = (m + VJP_TPB - 1) / VJP_TPB;
  v.P = b2 * most >= want ? 2 : 1;
  v.blocks = (int)(v.P == 2 ? b2 : b1);
  int64_t S = (want + v.blocks - 1) / v.blocks;
  if (S > most) S = most;
  v.tiles_per_split = (int)((ntiles + S - 1) / S);
  v.splits = (int)((ntiles + v.tiles_per_split - 1) / v.tiles_per_split);
  return v;
}
// Scratch of the splits' sums (one split needs none).
size_t vjp_part_bytes(const VjpPlan& v, int64_t mpad) {
  return v.splits > 1 ? (size_t)v.splits * v.nc * mpad * sizeof(float) : 0;
}

template <int PM>
static void launch_vjp_pm(Launch L, const VjpPlan& vp, const float* Xr, const float* XA, int ntiles, const float4* Y0r,
                          int mpad, const double* aY64, int g_mode, int m, const DevPose* ps, double pm1,
                          const float* v, float* grad, float* part) {
  const dim3 grid(vp.blocks, vp.splits);
  const auto k = vp.P == 2 ? force_vjp_kernel<2, PM> : force_vjp_kernel<1, PM>;
  k<<<grid, VJP_TPB, 0, L.stream>>>(Xr, XA, ntiles, vp.tiles_per_split, Y0r, mpad, aY64, g_mode, m, ps, pm1, v, grad,
                                    part);
  if (L.counter) ++*L.counter;
  if (vp.splits > 1) {
    vjp_combine_kernel<<<(m + VJP_TPB - 1) / VJP_TPB, VJP_TPB, 0, L.stream>>>(part, vp.splits, vp.nc, mpad, aY64,
                                                                              g_mode, m, pm1, v, grad);
    if (L.counter) ++*L.counter;
  }
}

cudaError_t launch_force_vjp(Launch L, const VjpPlan& vp, const float4* Xr, const float2* XA, int ntiles,
                             const float4* Y0r, int mpad, const double* aY64, int g_mode, int m, const DevPose* ps,
                             double p, const float* v, float* grad, float* part) {
  if (m <= 0) return cudaSuccess;
  const float* xr = reinterpret_cast<const float*>(Xr);
  const float* xa = reinterpret_cast<const float*>(XA);
  const auto launch = p == 1.0   ? launch_vjp_pm<1>
                      : p == 2.0 ? launch_vjp_pm<2>
                      : p == 3.0 ? launch_vjp_pm<3>
                                 : launch_vjp_pm<0>;
  launch(L, vp, xr, xa, ntiles, Y0r, mpad, aY64, g_mode, m, ps, p - 1.0, v, grad, part);
  return cudaGetLastError();
}

// ---- stored pair terms (comparison variant of the adjoint) -----------------
// Forward: every pair weight w_ij = g d^(p-1) is written to W[i][npad]
// (float32, M rows of the padded reference length; padding records carry
// weight 0) and the potential U = sum aY w d^2 / (p + 1) is summed per block.
// Backward: a block streams ST_RROWS rows back from HBM and forms the same
// per-point sums (sum w, sum w X') that the force kernel accumulates, so the
// adjoint reduction is shared.  Both passes move 16 bytes per thread access:
// a thread owns four consecutive reference points.
constexpr int ST_TPB = 256;
constexpr int ST_JB = 4 * ST_TPB;  // reference points per block column (npad is a multiple of it or of 256)

// Block (ST_ROWS template points x ST_JB reference points): the records are
// read once, each thread walks the block's template points and writes each
// row segment as one float4.
constexpr int ST_ROWS = 64;

__device__ __forceinline__ float st_ex2(float x) {
  float y;
  asm("ex2.approx.ftz.f32 %0, %1;" : "=f"(y) : "f"(x));
  return y;
}
__device__ __forceinline__ float st_lg2(float x) {
  float y;
  asm("lg2.approx.ftz.f32 %0, %1;" : "=f"(y) : "f"(x));
  return y;
}

// w = 2^-(u^2 - L) d^(p-1) with d^(p-1) = 2^(qexp log2 d^2), qexp = (p-1)/2.
__device__ __forceinline__ float st_weight(float d2, float ep, float qexp) {
  if (qexp == 0.f) return st_ex2(-ep);
  return st_ex2(fmaf(qexp, st_lg2(d2), -ep));  // d2 = 0: lg2 = -inf, weight 0
}

__global__ void __launch_bounds__(ST_TPB)
    store_pairs_kernel(const float* __restrict__ Xr, const float* __restrict__ XA, int npad, int m,
                       const float4* __restrict__ Y0r, const double* __restrict__ aY64, int g_mode,
                       const DevPose* __restrict__ ps, float qexp, float* __restrict__ Wst,
                       double* __restrict__ Upart) {
  __shared__ double sh[1][RED_THREADS];
  const int j0 = blockIdx.y * ST_JB + threadIdx.x * 4;
  const int i0 = blockIdx.x * ST_ROWS;
  float A[9], b[3];
#pragma unroll
  for (int q = 0; q < 9; ++q) A[q] = ps->A[q];
#pragma unroll
  for (int q = 0; q < 3; ++q) b[q] = ps->b[q];
  float4 x4 = make_float4(0.f, 0.f, 0.f, 0.f), y4 = x4, z4 = x4, a4 = x4;
  float4 l4 = make_float4(INFINITY, INFINITY, INFINITY, INFINITY);
  const bool live = j0 < npad;
  if (live) {
    const size_t t = (size_t)(j0 / FORCE_TJ), r = (size_t)(j0 % FORCE_TJ);
    const float* xr = Xr + t * 4 * FORCE_TJ + r;
    const float* xa = XA + t * 2 * FORCE_TJ + r;
    x4 = *reinterpret_cast<const float4*>(xr);
    y4 = *reinterpret_cast<const float4*>(xr + FORCE_TJ);
    z4 = *reinterpret_cast<const float4*>(xr + 2 * FORCE_TJ);
    a4 = *reinterpret_cast<const float4*>(xa);
    l4 = *reinterpret_cast<const float4*>(xa + FORCE_TJ);
  }
  const float xs[4] = {x4.x, x4.y, x4.z, x4.w}, ys[4] = {y4.x, y4.y, y4.z, y4.w};
  const float zs[4] = {z4.x, z4.y, z4.z, z4.w}, as[4] = {a4.x, a4.y, a4.z, a4.w};
  const float ls[4] = {l4.x, l4.y, l4.z, l4.w};
  // U terms are summed in FP32 over runs of 16 rows and the runs in FP64
  // (FP64 arithmetic per pair would cost more than the pair itself).
  double u[1] = {0.0};
  const int iend = min(m, i0 + ST_ROWS);
  for (int ib = i0; ib < iend; ib += 16) {
    float run = 0.f;
    const int ie = min(iend, ib + 16);
    for (int i = ib; i < ie; ++i) {
      const float4 y0 = Y0r[i];
      float yx, yy, yz;
      tpoint(y0, A, b, yx, yy, yz);
      const float ay = g_mode == 1 ? (float)aY64[i] : 1.f;
      float w[4];
#pragma unroll
      for (int k = 0; k < 4; ++k) {
        const float rx = yx - xs[k], ry = yy - ys[k], rz = yz - zs[k];
        const float d2 = fmaf(rz, rz, fmaf(ry, ry, rx * rx));
        const float uu = as[k] - y0.w;
        w[k] = st_weight(d2, fmaf(uu, uu, ls[k]), qexp);
        run = fmaf(ay * w[k], d2, run);
      }
      if (live) *reinterpret_cast<float4*>(Wst + (size_t)i * npad + j0) = make_float4(w[0], w[1], w[2], w[3]);
    }
    u[0] += (double)run;
  }
  block_sum<1>(u, sh);
  if (threadIdx.x == 0) Upart[(size_t)blockIdx.x * gridDim.y + blockIdx.y] = u[0];
}

// Backward from the stored weights: a block owns ST_RROWS template rows and
// each thread four consecutive reference points per step, so every weight is
// read once as part of a float4 (all ST_RROWS loads of a step are issued
// before they are used) and each reference record once per block.  The last
// block re-reads row m-1 for its missing rows and discards those sums.
constexpr int ST_RROWS = 8;

__global__ void __launch_bounds__(ST_TPB, 2)
    stored_rows_kernel(const float* __restrict__ Wst, int npad, int m, const float* __restrict__ Xr,
                       float4* __restrict__ partial) {
  __shared__ double red[ST_TPB / 32][ST_RROWS * 4];
  const int r0 = blockIdx.x * ST_RROWS;
  const int nr = min(ST_RROWS, m - r0);
  const float* rows[ST_RROWS];
#pragma unroll
  for (int r = 0; r < ST_RROWS; ++r) rows[r] = Wst + (size_t)min(r0 + r, m - 1) * npad;
  float acc[ST_RROWS][4];
#pragma unroll
  for (int r = 0; r < ST_RROWS; ++r) acc[r][0] = acc[r][1] = acc[r][2] = acc[r][3] = 0.f;
  for (int j0 = threadIdx.x * 4; j0 < npad; j0 += ST_JB) {
    float4 w4[ST_RROWS];
#pragma unroll
    for (int r = 0; r < ST_RROWS; ++r) w4[r] = *reinterpret_cast<const float4*>(rows[r] + j0);
    const size_t t = (size_t)(j0 / FORCE_TJ), q = (size_t)(j0 % FORCE_TJ);
    const float* xr = Xr + t * 4 * FORCE_TJ + q;
    const float4 x = *reinterpret_cast<const float4*>(xr);
    const float4 y = *reinterpret_cast<const float4*>(xr + FORCE_TJ);
    const float4 z = *reinterpret_cast<const float4*>(xr + 2 * FORCE_TJ);
#pragma unroll
    for (int r = 0; r < ST_RROWS; ++r) {
      const float4 w = w4[r];
      acc[r][0] += (w.x + w.y) + (w.z + w.w);
      acc[r][1] = fmaf(w.w, x.w, fmaf(w.z, x.z, fmaf(w.y, x.y, fmaf(w.x, x.x, acc[r][1]))));
      acc[r][2] = fmaf(w.w, y.w, fmaf(w.z, y.z, fmaf(w.y, y.y, fmaf(w.x, y.x, acc[r][2]))));
      acc[r][3] = fmaf(w.w, z.w, fmaf(w.z, z.z, fmaf(w.y, z.y, fmaf(w.x, z.x, acc[r][3]))));
    }
  }
  // block reduction: FP32 warp shuffles, then the warps' sums in FP64
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
#pragma unroll
  for (int r = 0; r < ST_RROWS; ++r)
#pragma unroll
    for (int c = 0; c < 4; ++c) {
      float v = acc[r][c];
      for (int off = 16; off > 0; off >>= 1) v += __shfl_down_sync(0xffffffffu, v, off);
      if (lane == 0) red[warp][r * 4 + c] = v;
    }
  __syncthreads();
  if (threadIdx.x < ST_RROWS * 4) {
    double v = 0.0;
    for (int w = 0; w < ST_TPB / 32; ++w) v += red[w][threadIdx.x];
    red[0][threadIdx.x] = v;
  }
  __syncthreads();
  if (threadIdx.x < nr)
    partial[r0 + threadIdx.x] = make_float4((float)red[0][threadIdx.x * 4], (float)red[0][threadIdx.x * 4 + 1],
                                            (float)red[0][threadIdx.x * 4 + 2], (float)red[0][threadIdx.x * 4 + 3]);
}

cudaError_t launch_store_pairs(Launch L, const float2* XA, const float4* Xr, int npad, const float4* Y0r,
                               const double* aY64, int g_mode, int m, const DevPose* ps, float qexp, float* Wst,
                               double* Upart) {
  const int nb = store_pairs_columns(npad);
  const int ib = (m + ST_ROWS - 1) / ST_ROWS;
  store_pairs_kernel<<<dim3(ib, nb), ST_TPB, 0, L.stream>>>(reinterpret_cast<const float*>(Xr),
                                                           reinterpret_cast<const float*>(XA), npad, m, Y0r, aY64,
                                                           g_mode, ps, qexp, Wst, Upart);
  if (L.counter) *L.counter += 1;
  return cudaGetLastError();
}

int store_pairs_columns(int npad) { return (npad + ST_JB - 1) / ST_JB; }
int store_pairs_row_blocks(int m) { return (m + ST_ROWS - 1) / ST_ROWS; }

cudaError_t launch_stored_rows(Launch L, const float* Wst, int npad, int m, const float4* Xr, float4* partial) {
  stored_rows_kernel<<<(m + ST_RROWS - 1) / ST_RROWS, ST_TPB, 0, L.stream>>>(Wst, npad, m,
                                                                            reinterpret_cast<const float*>(Xr), partial);
  if (L.counter) ++*L.counter;
  return cudaGetLastError();
}

cudaError_t launch_pose_from_host(Launch L, const HostPose& hp, DevPose* ps, const DevStats* st) {
  pose_from_host_kernel<<<1, 32, 0, L.stream>>>(hp, ps, st);
  if (L.counter) ++*L.counter;
  return cudaGetLastError();
}

cudaError_t launch_adjoint_combine(Launch L, const float4* partial, int S, int mpad, int m, const float4* Y0r,
                                   const double* aY64, int g_mode, const DevPose* ps, float* grad_xyz,
                                   double* blockpart) {
  adjoint_combine_kernel<<<(mpad + RED_THREADS - 1) / RED_THREADS, RED_THREADS, 0, L.stream>>>(
      partial, S, mpad, m, Y0r, aY64, g_mode, ps, grad_xyz, blockpart);
  if (L.counter) ++*L.counter;
  return cudaGetLastError();
}

cudaError_t launch_column_sum13(Launch L, const double* part, int nb, double* out) {
  column_sum13_kernel<<<1, RED_THREADS, 0, L.stream>>>(part, nb, out);
  if (L.counter) ++*L.counter;
  return cudaGetLastError();
}

}  // namespace scgr
