// C ABI, differentiation form: the shape-weighted potential, its adjoint
// (recomputed tiles or stored pair terms) and the force-field VJP.
#include <cuda_runtime.h>

#include <algorithm>
#include <cmath>
#include <cstring>
#include <string>
#include <vector>

#include "context.cuh"

using namespace scgr;
using namespace scgr::api;

namespace {

// exp([w]_x) = I + a K + b K^2 (Rodrigues), K = [w]_x
void axis_angle_terms(const double* w, double K[9], double K2[9], double& th2) {
  const double k[9] = {0.0, -w[2], w[1], w[2], 0.0, -w[0], -w[1], w[0], 0.0};
  th2 = w[0] * w[0] + w[1] * w[1] + w[2] * w[2];
  for (int r = 0; r < 3; ++r)
    for (int c = 0; c < 3; ++c) {
      K[r * 3 + c] = k[r * 3 + c];
      K2[r * 3 + c] = k[r * 3] * k[c] + k[r * 3 + 1] * k[3 + c] + k[r * 3 + 2] * k[6 + c];
    }
}

// Row-vector rotation R = exp([w]_x)^T and the rest of the pose.
HostPose pose_of(const double pose7[7]) {
  HostPose hp;
  double K[9], K2[9], th2, a, b;
  axis_angle_terms(pose7, K, K2, th2);
  if (th2 < 1e-16) {
    a = 1.0 - th2 / 6.0;
    b = 0.5 - th2 / 24.0;
  } else {
    const double th = std::sqrt(th2);
    a = std::sin(th) / th;
    b = (1.0 - std::cos(th)) / th2;
  }
  for (int r = 0; r < 3; ++r)
    for (int c = 0; c < 3; ++c) hp.R[c * 3 + r] = (r == c ? 1.0 : 0.0) + a * K[r * 3 + c] + b * K2[r * 3 + c];
  for (int c = 0; c < 3; ++c) hp.t[c] = pose7[3 + c];
  hp.s = pose7[6];
  return hp;
}

// (dU/domega, dU/dt, dU/ds) from the chain-rule sums tot (sum G, sum G.(Y0 R),
// sum Y0^T G).
void pose_gradient(const double* tot, const double pose7[7], const HostPose& hp, double grad7[7]) {
  double B[9];  // (dU/dR) R_col, R_col = R^T, dU/dR = s sum Y0^T G
  for (int a = 0; a < 3; ++a)
    for (int c = 0; c < 3; ++c) {
      double acc = 0.0;
      for (int q = 0; q < 3; ++q) acc += hp.s * tot[4 + a * 3 + q] * hp.R[c * 3 + q];
      B[a * 3 + c] = acc;
    }
  const double w[3] = {B[5] - B[7], B[6] - B[2], B[1] - B[3]};
  double K[9], K2[9], th2, c1, c2;  // J_r = I - c1 K + c2 K^2
  axis_angle_terms(pose7, K, K2, th2);
  if (th2 < 1e-12) {
    c1 = 0.5 - th2 / 24.0;
    c2 = 1.0 / 6.0 - th2 / 120.0;
  } else {
    const double th = std::sqrt(th2);
    c1 = (1.0 - std::cos(th)) / th2;
    c2 = (th - std::sin(th)) / (th2 * th);
  }
  for (int k = 0; k < 3; ++k) {
    double g = 0.0;
    for (int r = 0; r < 3; ++r) g += ((r == k ? 1.0 : 0.0) - c1 * K[r * 3 + k] + c2 * K2[r * 3 + k]) * w[r];
    grad7[k] = g;
  }
  for (int c = 0; c < 3; ++c) grad7[3 + c] = tot[c];
  grad7[6] = tot[3];
}

scgr_status check_potential(scgr_ctx* c, const double pose7[7], double* U_out) {
  if (!c || !pose7 || !U_out) return fail(c, SCGR_ERR_INVALID_ARG, "NULL argument");
  c->err.clear();
  if (!c->have_desc) return fail(c, SCGR_ERR_STATE, "compute descriptors first");
  for (int q = 0; q < 7; ++q)
    if (!std::isfinite(pose7[q])) return fail(c, SCGR_ERR_INVALID_ARG, "non-finite pose");
  if (!(pose7[6] > 0.0)) return fail(c, SCGR_ERR_INVALID_ARG, "scale must be > 0");
  if (c->rows >= 0) return fail(c, SCGR_ERR_STATE, "the potential needs the whole template (a row range is set)");
  return SCGR_OK;
}

// Sums of the pass to the host: U, the pose gradient, the device error word.
scgr_status finish_potential(scgr_ctx* c, const double* upart, int64_t nu, bool grad, const double pose7[7],
                             const HostPose& hp, double* U_out, double* grad_pose7) {
  SCGR_CK(c, launch_potential_finish(c->L(), upart, nu, (const double*)c->blockpart.p,
                                     grad ? combine_blocks(c->mpad) : 0, c->errword, c->aux));
  double h[15];
  SCGR_CK(c, cudaMemcpyAsync(h, c->aux, sizeof(h), cudaMemcpyDeviceToHost, c->stream));
  SCGR_CK(c, cudaStreamSynchronize(c->stream));
  *U_out = h[0] / (c->prm.p + 1.0);
  if (grad_pose7) pose_gradient(h + 1, pose7, hp, grad_pose7);
  return h[14] == 0.0 ? SCGR_OK : read_error_word(c);
}

}  // namespace

extern "C" {

scgr_status scgr_potential(scgr_ctx* c, const double pose7[7], double* U_out, double* grad_pose7,
                           float* grad_xyz_dev) {
  NvtxRange nvtx_range("scgr_potential");
  const scgr_status ck = check_potential(c, pose7, U_out);
  if (ck != SCGR_OK) return ck;
  Launch L = c->L();
  const HostPose hp = pose_of(pose7);
  const bool grad = grad_pose7 || grad_xyz_dev;
  SCGR_CK(c, launch_pose_from_host(L, hp, c->pose_eval, c->stats));
  const ForcePlan& fu = c->fpot;
  // the split partials: the force pass's (nothing reads them between calls) where they suffice
  const size_t need = (size_t)fu.splits * c->mpad * sizeof(float4);
  if (grad && need > c->partial.cap) SCGR_CK(c, ensure(c->ppart, need));
  float4* const part = (float4*)(need > c->partial.cap ? c->ppart.p : c->partial.p);
  SCGR_CK(c, launch_potential(L, fu, grad, (const float4*)c->Xr.p, (const float2*)c->XA.p,
                              (int)(c->npad / c->fp.tile_j), (const float4*)c->Y0r.p, (int)c->mpad, (int)c->m,
                              (const float*)c->aY32.p, c->prm.g_mode, c->pose_eval, c->qexp, part, (double*)c->upart.p));
  if (grad)
    SCGR_CK(c, launch_adjoint_combine(L, part, fu.splits, (int)c->mpad, (int)c->m,
                                      (const float4*)c->Y0r.p, (const double*)c->aY64.p, c->prm.g_mode,
                                      c->pose_eval, grad_xyz_dev, (double*)c->blockpart.p));
  return finish_potential(c, (const double*)c->upart.p, (int64_t)fu.splits * fu.iblocks, grad, pose7, hp, U_out,
                          grad_pose7);
}

scgr_status scgr_potential_stored(scgr_ctx* c, const double pose7[7], double* U_out, double* grad_pose7,
                                  float* grad_xyz_dev) {
  NvtxRange nvtx_range("scgr_potential_stored");
  const scgr_status ck = check_potential(c, pose7, U_out);
  if (ck != SCGR_OK) return ck;
  const int npad = (int)c->npad, m = (int)c->m;
  const int64_t nu = (int64_t)store_pairs_columns(npad) * store_pairs_row_blocks(m);
  SCGR_CK(c, ensure(c->wstore, (size_t)npad * m * sizeof(float)));
  SCGR_CK(c, ensure(c->wupart, (size_t)nu * sizeof(double)));
  SCGR_CK(c, ensure(c->wpartial, (size_t)c->mpad * sizeof(float4)));
  Launch L = c->L();
  const HostPose hp = pose_of(pose7);
  const bool grad = grad_pose7 || grad_xyz_dev;
  SCGR_CK(c, launch_pose_from_host(L, hp, c->pose_eval, c->stats));
  // forward: store w_ij and sum U
  SCGR_CK(c, launch_store_pairs(L, (const float2*)c->XA.p, (const float4*)c->Xr.p, npad, (const float4*)c->Y0r.p,
                                (const double*)c->aY64.p, c->prm.g_mode, m, c->pose_eval, c->qexp,
                                (float*)c->wstore.p, (double*)c->wupart.p));
  if (grad) {
    // backward from the stored terms
    SCGR_CK(c, launch_stored_rows(L, (const float*)c->wstore.p, npad, m, (const float4*)c->Xr.p,
                                  (float4*)c->wpartial.p));
    SCGR_CK(c, launch_adjoint_combine(L, (const float4*)c->wpartial.p, 1, (int)c->mpad, m, (const float4*)c->Y0r.p,
                                      (const double*)c->aY64.p, c->prm.g_mode, c->pose_eval, grad_xyz_dev,
                                      (double*)c->blockpart.p));
  }
  return finish_potential(c, (const double*)c->wupart.p, nu, grad, pose7, hp, U_out, grad_pose7);
}

scgr_status scgr_force_vjp(scgr_ctx* c, const float* v_dev, float* grad_dev) {
  NvtxRange nvtx_range("scgr_force_vjp");
  if (!c || !v_dev || !grad_dev) return fail(c, SCGR_ERR_INVALID_ARG, "NULL argument");
  c->err.clear();
  if (!c->have_desc) return fail(c, SCGR_ERR_STATE, "compute descriptors first");
  if (c->rows >= 0) return fail(c, SCGR_ERR_STATE, "the VJP needs the whole template (a row range is set)");
  SCGR_CK(c, launch_force_vjp(c->L(), c->vjp, (const float4*)c->Xr.p, (const float2*)c->XA.p,
                              (int)(c->npad / FORCE_TJ), (const float4*)c->Y0r.p, (int)c->mpad,
                              (const double*)c->aY64.p, c->prm.g_mode, (int)c->m, c->pose, c->prm.p, v_dev, grad_dev,
                              (float*)(vjp_part_bytes(c->vjp, c->mpad) > c->partial.cap ? c->vjppart.p : c->partial.p)));
  return SCGR_OK;
}

}  // extern "C"
