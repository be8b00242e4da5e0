// The pose update shared by the finalize kernels and the kernels that run many
// iterations in one launch (the library is built without relocatable device
// code, so shared device code lives in headers): 3x3 singular values and polar
// factors, warp-parallel 3x3 algebra, and the two halves of the update.
#pragma once
#include <cmath>

#include "common.cuh"

namespace scgr {

// A = U diag(S) V^T for a 3x3 A (row-major), S descending, U and V proper
// or improper orthogonal; one-sided Jacobi (Hestenes) rotations on columns.
__device__ inline void svd3(const double* Ain, double* U, double* S, double* V) {
  double a[3][3], v[3][3];
  for (int r = 0; r < 3; ++r)
    for (int c = 0; c < 3; ++c) {
      a[r][c] = Ain[r * 3 + c];
      v[r][c] = (r == c) ? 1.0 : 0.0;
    }
  for (int sweep = 0; sweep < 60; ++sweep) {
    double worst = 0.0;
    for (int pq = 0; pq < 3; ++pq) {
      const int p = pq == 2 ? 1 : 0;
      const int q = pq == 0 ? 1 : 2;
      double al = 0, be = 0, ga = 0;
      for (int k = 0; k < 3; ++k) {
        al += a[k][p] * a[k][p];
        be += a[k][q] * a[k][q];
        ga += a[k][p] * a[k][q];
      }
      if (ga == 0.0) continue;
      const double rel = fabs(ga) / sqrt(al * be);
      if (rel > worst) worst = rel;
      if (rel < 1e-16) continue;
      const double zeta = (be - al) / (2.0 * ga);
      double t;
      if (fabs(zeta) > 1e150) t = 0.5 / zeta;
      else t = (zeta >= 0 ? 1.0 : -1.0) / (fabs(zeta) + sqrt(1.0 + zeta * zeta));
      const double c = 1.0 / sqrt(1.0 + t * t);
      const double s = c * t;
      for (int k = 0; k < 3; ++k) {
        const double ap = a[k][p], aq = a[k][q];
        a[k][p] = c * ap - s * aq;
        a[k][q] = s * ap + c * aq;
        const double vp = v[k][p], vq = v[k][q];
        v[k][p] = c * vp - s * vq;
        v[k][q] = s * vp + c * vq;
      }
    }
    if (worst < 1e-15) break;
  }
  double sg[3];
  for (int p = 0; p < 3; ++p) sg[p] = sqrt(a[0][p] * a[0][p] + a[1][p] * a[1][p] + a[2][p] * a[2][p]);
  int o[3] = {0, 1, 2};
  for (int x = 0; x < 3; ++x)
    for (int y = 0; y < 2 - x; ++y)
      if (sg[o[y]] < sg[o[y + 1]]) {
        const int tmp = o[y];
        o[y] = o[y + 1];
        o[y + 1] = tmp;
      }
  double u[3][3];
  for (int c = 0; c < 3; ++c) {
    const int p = o[c];
    S[c] = sg[p];
    for (int r = 0; r < 3; ++r) {
      V[r * 3 + c] = v[r][p];
      u[r][c] = sg[p] > 0.0 ? a[r][p] / sg[p] : 0.0;
    }
  }
  // complete U where a singular value vanished (only the last two can)
  if (!(S[1] > 0.0)) {
    // pick any unit vector orthogonal to u0
    double e[3] = {0, 0, 0};
    const int ax = fabs(u[0][0]) < 0.577 ? 0 : (fabs(u[1][0]) < 0.577 ? 1 : 2);
    e[ax] = 1.0;
    const double d = e[0] * u[0][0] + e[1] * u[1][0] + e[2] * u[2][0];
    double n2 = 0;
    for (int r = 0; r < 3; ++r) {
      u[r][1] = e[r] - d * u[r][0];
      n2 += u[r][1] * u[r][1];
    }
    n2 = sqrt(n2);
    for (int r = 0; r < 3; ++r) u[r][1] /= n2;
  }
  if (!(S[2] > 0.0)) {
    u[0][2] = u[1][0] * u[2][1] - u[2][0] * u[1][1];
    u[1][2] = u[2][0] * u[0][1] - u[0][0] * u[2][1];
    u[2][2] = u[0][0] * u[1][1] - u[1][0] * u[0][1];
  }
  for (int r = 0; r < 3; ++r)
    for (int c = 0; c < 3; ++c) U[r * 3 + c] = u[r][c];
}

__device__ __forceinline__ double det3(const double* M) {
  return M[0] * (M[4] * M[8] - M[5] * M[7]) - M[1] * (M[3] * M[8] - M[5] * M[6]) +
         M[2] * (M[3] * M[7] - M[4] * M[6]);
}

// Nearest orthogonal matrix U V^T of R = U S V^T.
__device__ inline void polar3(const double* R, double* out) {
  double U[9], S[3], V[9];
  svd3(R, U, S, V);
  for (int r = 0; r < 3; ++r)
    for (int c = 0; c < 3; ++c)
      out[r * 3 + c] = U[r * 3] * V[c * 3] + U[r * 3 + 1] * V[c * 3 + 1] + U[r * 3 + 2] * V[c * 3 + 2];
}

// ---- warp-parallel 3x3 algebra -------------------------------------------
// GB300 issues an FP64 warp instruction at a small fraction of the FP32 rate
// whatever the number of active lanes, so the finalize step spreads its 3x3
// matrices over a warp: lane l < 9 owns entry (l / 3, l % 3) (lanes 9..31
// mirror entry 8; their results are never stored).  A 3x3 product is then 3
// FP64 instructions for the warp instead of 27 for one thread.  Every
// function here must be called by all 32 lanes of the warp together.
constexpr unsigned WFULL = 0xffffffffu;

struct Lane3 {
  int q, r, c;
};
__device__ __forceinline__ Lane3 lane3() {
  const int q = min((int)(threadIdx.x & 31), 8);
  return {q, q / 3, q % 3};
}
__device__ __forceinline__ double wget(double v, int idx) { return __shfl_sync(WFULL, v, idx); }

// (A B)_rc and (A^T B)_rc for lane-owned A and B
__device__ __forceinline__ double wmul(double a, double b, Lane3 L) {
  const double acc = wget(a, L.r * 3) * wget(b, L.c);
  return fma(wget(a, L.r * 3 + 2), wget(b, 6 + L.c), fma(wget(a, L.r * 3 + 1), wget(b, 3 + L.c), acc));
}
__device__ __forceinline__ double wmul_ta(double a, double b, Lane3 L) {
  const double acc = wget(a, L.r) * wget(b, L.c);
  return fma(wget(a, 6 + L.r), wget(b, 6 + L.c), fma(wget(a, 3 + L.r), wget(b, 3 + L.c), acc));
}

// Sum and maximum over lanes 0..8, the same value in every lane (lane 0's).
__device__ __forceinline__ float wsum9(float v) {
  if ((threadIdx.x & 31) >= 9) v = 0.f;
  for (int off = 16; off > 0; off >>= 1) v += __shfl_xor_sync(WFULL, v, off);
  return __shfl_sync(WFULL, v, 0);
}
__device__ __forceinline__ double wsum9d(double v) {
  if ((threadIdx.x & 31) >= 9) v = 0.0;
  for (int off = 16; off > 0; off >>= 1) v += __shfl_xor_sync(WFULL, v, off);
  return __shfl_sync(WFULL, v, 0);
}
__device__ __forceinline__ float wmax9(float v) {
  if ((threadIdx.x & 31) >= 9) v = 0.f;
  for (int off = 16; off > 0; off >>= 1) v = fmaxf(v, __shfl_xor_sync(WFULL, v, off));
  return __shfl_sync(WFULL, v, 0);
}

// 1/x for x > 0 in float64 from the float32 reciprocal and two Newton steps.
__device__ __forceinline__ double wrcp(double x) {
  double r = (double)(1.0f / (float)x);
  r = fma(r, fma(-x, r, 1.0), r);
  return fma(r, fma(-x, r, 1.0), r);
}

// Orthogonal polar factor Q of A (A = Q H, H symmetric positive definite)
// for det A > 0 by Newton's iteration X <- (g X + X^-T / g) / 2 with
// Frobenius-norm scaling g = (|X^-1| / |X|)^(1/2) while far from the limit
// (Higham, "Computing the polar decomposition -- with applications", 1986),
// in float64 with the 3x3 spread over the warp: Q's entry in each lane.
// X^-T is the cofactor matrix over the determinant.  The input is first
// scaled to unit Frobenius norm, which leaves the polar factor unchanged and
// keeps the FP32 norms below in range.  The scaling factor g and the stop
// test use FP32 sums: any positive weights (a X + b X^-T) / 2 keep the polar
// factor, so they only steer convergence; the last steps use a = b = 1
// exactly.  Returns false (the caller then takes the SVD) when det A <= 0,
// when |A|_F |A^-1|_F > 1e6, or when the iteration has not settled in 40
// steps.
__device__ inline bool polar_newton_warp(double A, Lane3 L, double& Q) {
  const double n2 = wsum9d(A * A);
  if (!(n2 > 0.0) || !isfinite(n2)) return false;
  double X = A * (1.0 / sqrt(n2));
  const int r1 = (L.r + 1) % 3, r2 = (L.r + 2) % 3, c1 = (L.c + 1) % 3, c2 = (L.c + 2) % 3;
  bool scale = true;
  for (int it = 0; it < 40; ++it) {
    double C = fma(-wget(X, r1 * 3 + c2), wget(X, r2 * 3 + c1), wget(X, r1 * 3 + c1) * wget(X, r2 * 3 + c2));
    const double det = fma(wget(X, 2), wget(C, 2), fma(wget(X, 1), wget(C, 1), wget(X, 0) * wget(C, 0)));
    if (!(det > 1e-30) || !isfinite(det)) return false;
    C *= wrcp(det);  // X^-T
    const float fx = (float)X, fc = (float)C;
    const float nx = wsum9(fx * fx), ny = wsum9(fc * fc);
    if (it == 0 && !(nx * ny <= 1e12f)) return false;
    const float g = scale ? sqrtf(sqrtf(ny / nx)) : 1.f;
    const double Xn = fma(0.5 * (double)g, X, (double)(0.5f / g) * C);
    const float dx = (float)(Xn - X), fn = (float)Xn;
    const float dd = wsum9(dx * dx), nn = wsum9(fn * fn);
    X = Xn;
    // stop once a step changed X by at most 1e-9 of its norm: Newton's
    // iteration converges quadratically there, so this iterate is within
    // about (1e-9)^2 of the polar factor, below float64 rounding
    if (dd <= 1e-18f * nn) break;
    scale = dd > 1e-4f * nn;
    if (it == 39) return false;
  }
  Q = X;
  return true;
}

__device__ __forceinline__ float fsqrt_approx(float x) {
  float y;
  asm("sqrt.approx.ftz.f32 %0, %1;" : "=f"(y) : "f"(x));
  return y;
}
// Sum of squares of nine values in a chain of three.
__device__ __forceinline__ float sq9(const float (&v)[9]) {
  const float p = fmaf(v[2], v[2], fmaf(v[1], v[1], v[0] * v[0]));
  const float q = fmaf(v[5], v[5], fmaf(v[4], v[4], v[3] * v[3]));
  const float r = fmaf(v[8], v[8], fmaf(v[7], v[7], v[6] * v[6]));
  return (p + q) + r;
}

// Float64 tests on the integer pipe (a float64 comparison costs as much as an
// addition): finite; positive and within [2^-100, 2^100); times 2^k for a
// normal value whose exponent stays in range (0 for zero).
__device__ __forceinline__ bool finite64(double v) { return (__double2hiint(v) & 0x7ff00000) != 0x7ff00000; }
__device__ __forceinline__ bool moderate64(double v) {
  const int h = __double2hiint(v);
  return h >= ((1023 - 100) << 20) && h < ((1023 + 100) << 20);
}
__device__ __forceinline__ double scale64(double v, int k) {
  const int h = __double2hiint(v);
  return (h & 0x7ff00000) == 0 ? 0.0 : __hiloint2double(h + (k << 20), __double2loint(v));
}

// Polar factor of A (lane-owned) with most of the work in float32.  On
// GB300 a float64 instruction costs about 65 cycles whatever the number of
// active lanes, and consecutive ones do not overlap, so the float64 work is
// kept to the few products that need it.  Every lane first runs the same
// scaled Newton iteration on its own float copy X of the 3x3, then two
// corrections against A itself bring the factor to float64 accuracy.  A
// correction writes the current factor as Q = R (I + S), R orthogonal and
// S = (Q^T Q - I) / 2 symmetric and small, forms B = Q^T A (float64), so
// that R^T A = (I - S) B to first order, and takes the small rotation w that
// makes R (I + [w]x)'s transpose times A symmetric: with H = (B + B^T) / 2
// and k = axial of the skew part of (I - S) B doubled, the symmetric-H
// identity [w]x H + H [w]x = [(tr(H) I - H) w]x gives (tr(H) I - H) w = k.
// Then Q <- Q + X ([w]x - S).  Only Q^T Q, Q^T A, B - B^T and the final
// sum are float64; the rest are small quantities whose float32 rounding is
// second order.  Each correction squares the error (float32's ~1e-7, then
// float64 rounding).  Returns false, and the caller takes polar_newton_warp,
// for inputs out of float32 range, det <= 0, a Frobenius condition estimate
// above 1e3, or a correction that does not shrink.
__device__ inline bool polar_float_refined_warp(double A, Lane3 L, double& Q) {
  const float fa = (float)A;
  float x[9];
#pragma unroll
  for (int k = 0; k < 9; ++k) x[k] = __shfl_sync(WFULL, fa, k);
  const float n2 = sq9(x);
  if (!(n2 > 1e-30f) || !isfinite(n2)) return false;
  const float inv = rsqrtf(n2);
#pragma unroll
  for (int k = 0; k < 9; ++k) x[k] *= inv;
  bool scale = true, done = false;
  for (int it = 0; it < 20 && !done; ++it) {
    float c[9];  // cofactors of X, then X^-T
    c[0] = x[4] * x[8] - x[5] * x[7];
    c[1] = x[5] * x[6] - x[3] * x[8];
    c[2] = x[3] * x[7] - x[4] * x[6];
    c[3] = x[2] * x[7] - x[1] * x[8];
    c[4] = x[0] * x[8] - x[2] * x[6];
    c[5] = x[1] * x[6] - x[0] * x[7];
    c[6] = x[1] * x[5] - x[2] * x[4];
    c[7] = x[2] * x[3] - x[0] * x[5];
    c[8] = x[0] * x[4] - x[1] * x[3];
    const float det = fmaf(x[2], c[2], fmaf(x[1], c[1], x[0] * c[0]));
    if (!(det > 1e-20f) || !isfinite(det)) return false;
    const float rd = __fdividef(1.f, det);
#pragma unroll
    for (int k = 0; k < 9; ++k) c[k] *= rd;
    float a = 0.5f, b = 0.5f;
    if (scale) {
      const float nx = sq9(x), ny = sq9(c);
      if (it == 0 && !(nx * ny <= 1e6f)) return false;
      // any positive weights keep the polar factor: an approximate fourth root
      const float g = fsqrt_approx(fsqrt_approx(__fdividef(ny, nx)));
      a = 0.5f * g;
      b = __fdividef(0.5f, g);
    }
    float d[9];
#pragma unroll
    for (int k = 0; k < 9; ++k) {
      const float xn = fmaf(a, x[k], b * c[k]);
      d[k] = xn - x[k];
      x[k] = xn;
    }
    const float dd = sq9(d), nn = sq9(x);
    done = dd <= 1e-10f * nn;
    scale = dd > 1e-4f * nn;
  }
  if (!done) return false;
  const int q = L.q;
  float mine = x[0];
#pragma unroll
  for (int k = 1; k < 9; ++k) mine = (q == k) ? x[k] : mine;
  // lanes 0..8 own Q^T Q, lanes 16..24 Q^T A: the two products share their
  // float64 instructions
  const int half = threadIdx.x & 16, e = min((int)(threadIdx.x & 15), 8), r = e / 3, c = e % 3;
  double Qd = (double)__shfl_sync(WFULL, mine, e);
  // A scaled by a power of two near 1 / ||A|| (exact), so that the 3x3
  // quantities below stay near unit size
  int e2 = 0;
  frexpf(sqrtf(n2), &e2);
  const double As = scale64(wget(A, e), -e2);
  const double I = (r == c) ? 1.0 : 0.0;
  for (int step = 0; step < 2; ++step) {
    const double Z = half ? As : Qd;
    double prod = wget(Qd, r) * wget(Z, half + c);
    prod = fma(wget(Qd, 3 + r), wget(Z, half + 3 + c), prod);
    prod = fma(wget(Qd, 6 + r), wget(Z, half + 6 + c), prod);
    const double tB = wget(prod, 16 + c * 3 + r);  // B^T, B = Q^T A
    const float of = (float)(prod - (half ? tB : I)), bf = (float)prod;  // E = Q^T Q - I, or K = B - B^T; B
    float sm[9], bm[9];
#pragma unroll
    for (int k = 0; k < 9; ++k) {
      sm[k] = 0.5f * __shfl_sync(WFULL, of, k);
      bm[k] = __shfl_sync(WFULL, bf, 16 + k);
    }
    const float k21 = __shfl_sync(WFULL, of, 23), k02 = __shfl_sync(WFULL, of, 18), k10 = __shfl_sync(WFULL, of, 19);
    // entries of S B for its skew part
    auto sb = [&](int rr, int cc) { return fmaf(sm[rr * 3 + 2], bm[6 + cc], fmaf(sm[rr * 3 + 1], bm[3 + cc], sm[rr * 3] * bm[cc])); };
    const float kp0 = k21 - (sb(2, 1) - sb(1, 2));
    const float kp1 = k02 - (sb(0, 2) - sb(2, 0));
    const float kp2 = k10 - (sb(1, 0) - sb(0, 1));
    // M = tr(H) I - H, H = (B + B^T) / 2
    const float tr = bm[0] + bm[4] + bm[8];
    const float m00 = tr - bm[0], m11 = tr - bm[4], m22 = tr - bm[8];
    const float m01 = -0.5f * (bm[1] + bm[3]), m02 = -0.5f * (bm[2] + bm[6]), m12 = -0.5f * (bm[5] + bm[7]);
    // adj(M) (symmetric) and det M
    const float a00 = m11 * m22 - m12 * m12, a01 = m02 * m12 - m01 * m22, a02 = m01 * m12 - m02 * m11;
    const float a11 = m00 * m22 - m02 * m02, a12 = m01 * m02 - m00 * m12, a22 = m00 * m11 - m01 * m01;
    const float detM = fmaf(m02, a02, fmaf(m01, a01, m00 * a00));
    if (!(detM > 0.f) || !isfinite(detM)) return false;
    const float rdm = __frcp_rn(detM);
    const float w0 = rdm * fmaf(a02, kp2, fmaf(a01, kp1, a00 * kp0));
    const float w1 = rdm * fmaf(a12, kp2, fmaf(a11, kp1, a01 * kp0));
    const float w2 = rdm * fmaf(a22, kp2, fmaf(a12, kp1, a02 * kp0));
    const float wn = fmaf(w2, w2, fmaf(w1, w1, w0 * w0));
    if (!(wn <= (step == 0 ? 1e-8f : 1e-20f))) return false;
    // D = [w]x - S, and this lane's entry of X D
    const float d[9] = {-sm[0],      -w2 - sm[1], w1 - sm[2],  w2 - sm[3], -sm[4],
                        -w0 - sm[5], -w1 - sm[6], w0 - sm[7], -sm[8]};
    float p = 0.f;
#pragma unroll
    for (int k = 0; k < 9; ++k) {
      const float xd = fmaf(x[(k / 3) * 3 + 2], d[6 + k % 3], fmaf(x[(k / 3) * 3 + 1], d[3 + k % 3], x[(k / 3) * 3] * d[k % 3]));
      p = (e == k) ? xd : p;
    }
    Qd += (double)p;
  }
  Qd = wget(Qd, q);
  Q = Qd;
  return true;
}

// The pose's rotation is a product of increments that are orthogonal to
// float64 rounding; one Newton-Schulz step on it before the next product
// keeps R^T R - I at rounding (a second changes nothing above it).  False (the
// caller takes the SVD route) when R^T R is further than 1e-6 from I.
__device__ inline bool reorth_warp(double R, Lane3 L, double& out) {
  const double I = (L.r == L.c) ? 1.0 : 0.0;
  const double e = wmul_ta(R, R, L) - I;
  if (!(wmax9(fabsf((float)e)) <= 1e-6f)) return false;
  out = wmul(R, fma(-0.5, e, I), L);
  return true;
}

// The update in two halves.  What does not depend on this iteration's totals
// (the schedule of Eq. 12, the scale factor, s^2 R^T S0 R, the template mean, the
// re-orthonormalised R) is formed by four warps, on the SM's four schedulers,
// while other warps still add the totals; warp 0 then forms the rest.  All of
// it is float64 latency (see warp-parallel 3x3 algebra), so the split takes
// two thirds of the instructions off the critical path.
struct PosePre {
  double R[9];      // the pose's rotation, re-orthonormalised
  double SRR[9];    // s^2 R^T S0 R
  double yb[3];     // template mean at the pose
  double tmy[3];    // t - yb
  double scr[64];   // scratch of the SVD routes
};
struct PoseRate {
  double sched;     // step_mode 0: eta0 G / G1; 1: G time^2
  double sn, cs;    // next scale, and its ratio to the present one
};
constexpr int POSE_PRE_WARPS = 4;

// Eq. 12 at 0-based iteration it (one warp).
__device__ inline void pose_schedule(int it, int E, const StepParams& sp, PoseRate& o) {
  // G / G1 = 0.1 + 0.9 / (1 + e), written over one division (each float64
  // division is a chain of about ten float64 instructions, about 65 cycles
  // each on GB300)
  const double e1 = 1.0 + exp(-((double)it - (double)E / 2.0));
  const double g = fma(0.1, e1, 0.9) / e1;
  if ((threadIdx.x & 31) == 0) o.sched = sp.step_mode == 0 ? sp.eta0 * g : sp.G1 * g * sp.time * sp.time;
}

// Scale model (Sec. III-B) at scale s: c from the largest covariance
// eigenvalues (one warp).
__device__ inline void pose_scale(double s, const DevStats* __restrict__ st, const StepParams& sp, PoseRate& o) {
  const double eY = s * s * st->eY0;
  double cs = 1.0;
  if (sp.scale_mode == 0) cs = sqrt(st->eX / eY);
  else if (sp.scale_mode == 1) cs = st->eX / eY;
  if ((threadIdx.x & 31) == 0) {
    o.cs = cs;
    o.sn = cs * s;
  }
}

// Part `role` of the first half (one warp each; all 32 lanes).
__device__ inline void pose_pre(int role, const DevPose* ps, const DevStats* __restrict__ st, const StepParams& sp,
                                PosePre& o, PoseRate& rate) {
  const Lane3 L = lane3();
  const int lane = threadIdx.x & 31;
  if (role == 0) {
    pose_schedule(ps->it, ps->E, sp, rate);
  } else if (role == 1) {
    pose_scale(ps->s, st, sp, rate);
  } else if (role == 2) {
    const double s = ps->s, R = ps->R[L.q];
    const double SR = wmul(st->S0[L.q], R, L);
    const double v = s * s * wmul_ta(R, SR, L);
    if (lane < 9) o.SRR[lane] = v;
  } else {
    const double s = ps->s, R = ps->R[L.q], tc = ps->t[L.c];
    const double yb =
        fma(s, fma(st->ybar0[2], ps->R[6 + L.c], fma(st->ybar0[1], ps->R[3 + L.c], st->ybar0[0] * ps->R[L.c])), tc);
    const double tmy = tc - yb;
    if (lane < 3) {
      o.yb[lane] = yb;
      o.tmy[lane] = tmy;
    }
    double Rn;
    if (!reorth_warp(R, L, Rn)) {
      if (lane < 9) o.scr[32 + lane] = R;
      __syncwarp();
      if (lane == 0) polar3(o.scr + 32, o.scr + 48);
      __syncwarp();
      Rn = o.scr[48 + L.q];
    }
    if (lane < 9) o.R[lane] = Rn;
  }
}

// Eq. 5.5's d_c = dq F_c and kappa = dq M from the totals (every lane).
__device__ __forceinline__ bool pose_step(const double* tot, const StepParams& sp, const PoseRate& o, double& dq,
                                          double& kappa) {
  if (sp.step_mode == 0) {
    // kappa = eta0 (G / G1) M / W, and Eq. 5.5's d = kappa F / M needs no M
    const double W = tot[3];
    bool ok = true;
    if (moderate64(W)) {
      dq = o.sched * wrcp(W);
    } else {
      ok = W > 0.0 && isfinite(W);
      dq = ok ? o.sched / W : 0.0;
    }
    kappa = dq * (double)sp.M;
    return ok;
  }
  kappa = o.sched;
  dq = kappa / (double)sp.M;
  return true;
}

// Second half, by one warp: the step from the 13 totals tot (F[3], W, T[3][3]),
// the Kabsch rotation and the composed pose, written to *ps.  Lane (r, c) owns
// entry (r, c) of each 3x3; lanes 9..11 carry the translation as a fourth row.
// False (every lane) where the step is not finite and the pose is kept.
// set_mean = false leaves ybs and its float pair to the caller.
__device__ inline bool pose_post(const double* tot, DevPose* ps, const DevStats* __restrict__ st, const StepParams& sp,
                                 PosePre& o, const PoseRate& rate, int* err, bool set_mean = true) {
  const Lane3 L = lane3();
  const int lane = threadIdx.x & 31;
  const int row = min(lane / 3, 3), col = lane < 12 ? lane % 3 : 2;
  double dq, kappa;
  bool bad = !pose_step(tot, sp, rate, dq, kappa);
  const double dc = dq * tot[col];
  // C^ = Y_D^T Y_c = s^2 R^T S0 R + kappa T   (Eq. 6 with the displaced cloud;
  // T[a][b] = sum_i f_i[a] (Y_i - ybar)[b])
  const double Ch = fma(kappa, tot[4 + L.q], o.SRR[L.q]);
  bad = bad || !finite64(Ch) || !finite64(dc);
  if (__any_sync(WFULL, bad)) {
    if (lane == 0) {
      atomicOr(err, ERR_NUMERIC);
      ps->it += 1;
    }
    return false;
  }
  // Eq. 6: C^ = U S V^T, dd = sign det(V U^T), R_inc = V diag(1, 1, dd) U^T.
  // For det C^ > 0 (dd = 1) that is Q^T, Q the orthogonal polar factor of C^
  // (C^ = (U V^T)(V S V^T)), taken by Newton's iteration (in float32 with
  // float64 corrections, else all in float64); the SVD handles det C^ <= 0,
  // near-singular C^ and the degenerate case.
  double Q;  // R_inc^T
  if (!polar_float_refined_warp(Ch, L, Q) && !polar_newton_warp(Ch, L, Q)) {
    double* scr = o.scr;
    if (lane < 9) scr[lane] = Ch;
    __syncwarp();
    if (lane == 0) {
      double U[9], Sg[3], V[9], Ri[9];
      svd3(scr, U, Sg, V);
      if (!(Sg[0] > 0.0) || Sg[1] <= 1e-12 * Sg[0]) {
        for (int q = 0; q < 9; ++q) Ri[q] = (q % 4 == 0) ? 1.0 : 0.0;
        ps->degenerate += 1;
      } else {
        const double dd = (det3(V) * det3(U)) >= 0.0 ? 1.0 : -1.0;
        const double D[3] = {1.0, 1.0, dd};
        for (int r = 0; r < 3; ++r)
          for (int c = 0; c < 3; ++c)
            Ri[r * 3 + c] = V[r * 3] * D[0] * U[c * 3] + V[r * 3 + 1] * D[1] * U[c * 3 + 1] +
                            V[r * 3 + 2] * D[2] * U[c * 3 + 2];
      }
      for (int q = 0; q < 9; ++q) scr[16 + q] = Ri[q];
    }
    __syncwarp();
    Q = scr[16 + L.c * 3 + L.r];
  }
  // Eq. 8, Eq. 9: Y(t+1) = c (Y - ybar) R_inc + ybar + d, composed into the pose:
  // rows 0..2 of [R; t - ybar] R_inc are the next rotation, row 3 its translation
  const double x = lane < 9 ? o.R[lane] : o.tmy[col];
  double y = wget(x, row * 3) * wget(Q, col * 3);
  y = fma(wget(x, row * 3 + 1), wget(Q, col * 3 + 1), y);
  y = fma(wget(x, row * 3 + 2), wget(Q, col * 3 + 2), y);
  if (row == 3) y = fma(rate.cs, y, o.yb[col] + dc);
  if (!__all_sync(WFULL, finite64(rate.cs) && finite64(y))) {
    if (lane == 0) {
      atomicOr(err, ERR_NUMERIC);
      ps->it += 1;
    }
    return false;
  }
  // the new pose and its float32 map: A = s R, b = t - xbar
  const float f = (float)fma(lane < 9 ? rate.sn : 1.0, y, lane < 9 ? 0.0 : -st->xbar[col]);
  if (lane < 9) {
    ps->R[lane] = y;
    ps->A[lane] = f;
  } else if (lane < 12) {
    ps->t[col] = y;
    ps->b[col] = f;
  }
  if (lane == 12) {
    ps->s = rate.sn;
    ps->it += 1;
  }
  if (!set_mean) return true;
  // the template mean at the new pose, as refresh_pose forms it
  const double mean = fma(rate.sn, fma(st->ybar0[2], wget(y, 6 + col), fma(st->ybar0[1], wget(y, 3 + col), st->ybar0[0] * wget(y, col))),
                          wget(y, 9 + col));
  if (lane < 3) set_ybs(ps, lane, mean - st->xbar[col]);
  return true;
}

}  // namespace scgr
