// Internal helpers of the C ABI: argument checks, buffers, error words, the
// descriptor pass and the iteration launch sequence.
#include <cuda_runtime.h>

#include <atomic>
#include <cmath>
#include <cstring>
#include <string>
#include <vector>

#include "context.cuh"

using namespace scgr;

namespace scgr {
namespace api {

scgr_status fail(scgr_ctx* c, scgr_status st, const std::string& msg) {
  if (c) c->err = msg;
  return st;
}

scgr_status cuda_fail(scgr_ctx* c, cudaError_t e, const char* where) {
  cudaGetLastError();  // clear a sticky launch error where possible
  std::string msg = std::string(where) + ": " + cudaGetErrorString(e);
  if (e == cudaErrorMemoryAllocation) return fail(c, SCGR_ERR_OOM, msg);
  return fail(c, SCGR_ERR_CUDA, msg);
}

// Test hook: while > 0, the next allocations fail (host-side fault
// injection; nothing is asked of the device).
std::atomic<int> g_fail_allocs{0};

cudaError_t ensure(DevBuf& b, size_t bytes) {
  if (bytes == 0) bytes = 16;
  if (b.cap >= bytes) return cudaSuccess;
  if (g_fail_allocs.load() > 0) {
    g_fail_allocs.fetch_sub(1);
    return cudaErrorMemoryAllocation;
  }
  if (b.p) cudaFree(b.p);
  b.p = nullptr;
  b.cap = 0;
  cudaError_t e = cudaMalloc(&b.p, bytes);
  if (e == cudaSuccess) b.cap = bytes;
  return e;
}

void release(DevBuf& b) {
  if (b.p) cudaFree(b.p);
  b.p = nullptr;
  b.cap = 0;
}

scgr_status check_params(const scgr_params* p, std::string& why) {
  if (!p) { why = "params is NULL"; return SCGR_ERR_INVALID_ARG; }
  if (p->k < 3 || p->k > 32) { why = "k must be in [3, 32]"; return SCGR_ERR_INVALID_ARG; }
  if (!(p->p >= 1.0) || !std::isfinite(p->p)) { why = "p must be finite and >= 1 (Eq. 11)"; return SCGR_ERR_INVALID_ARG; }
  if (!std::isfinite(p->sigma)) { why = "sigma must be finite"; return SCGR_ERR_INVALID_ARG; }
  if (p->g_mode != 0 && p->g_mode != 1) { why = "g_mode must be 0 or 1"; return SCGR_ERR_INVALID_ARG; }
  if (!(p->G1 > 0.0) || !std::isfinite(p->G1)) { why = "G1 must be > 0"; return SCGR_ERR_INVALID_ARG; }
  if (p->step_mode != 0 && p->step_mode != 1) { why = "step_mode must be 0 or 1"; return SCGR_ERR_INVALID_ARG; }
  if (!(p->eta0 > 0.0) || !std::isfinite(p->eta0)) { why = "eta0 must be > 0"; return SCGR_ERR_INVALID_ARG; }
  if (!std::isfinite(p->time)) { why = "time must be finite"; return SCGR_ERR_INVALID_ARG; }
  if (p->scale_mode < 0 || p->scale_mode > 2) { why = "scale_mode must be 0, 1 or 2"; return SCGR_ERR_INVALID_ARG; }
  if (p->neigh_mode != 0 && p->neigh_mode != 1) { why = "neigh_mode must be 0 or 1"; return SCGR_ERR_INVALID_ARG; }
  if (p->neigh_mode == 1 && !(p->radius_scale > 0.0 && std::isfinite(p->radius_scale))) { why = "radius_scale must be > 0"; return SCGR_ERR_INVALID_ARG; }
  return SCGR_OK;
}

StepParams step_params(const scgr_ctx* c) {
  StepParams sp;
  sp.G1 = c->prm.G1;
  sp.eta0 = c->prm.eta0;
  sp.time = c->prm.time;
  sp.step_mode = c->prm.step_mode;
  sp.scale_mode = c->prm.scale_mode;
  sp.M = (int)c->m;
  return sp;
}

scgr_status read_error_word(scgr_ctx* c) {
  int h = 0;
  SCGR_CK(c, cudaMemcpyAsync(&h, c->errword, sizeof(int), cudaMemcpyDeviceToHost, c->stream));
  SCGR_CK(c, cudaStreamSynchronize(c->stream));
  if (h == 0) return SCGR_OK;
  SCGR_CK(c, cudaMemsetAsync(c->errword, 0, sizeof(int), c->stream));
  SCGR_CK(c, cudaStreamSynchronize(c->stream));
  if (h & ERR_NONFINITE)
    return fail(c, SCGR_ERR_NONFINITE, "an input coordinate is NaN/Inf or larger than 1e18 in magnitude");
  if (h & ERR_TIMEOUT) return fail(c, SCGR_ERR_TIMEOUT, "a bounded device-side wait gave up");
  return fail(c, SCGR_ERR_NUMERIC, "the iteration step became non-finite (zero or non-finite total weight)");
}

// Whether a caller is capturing the stream (a stream that cannot be asked is not being captured).
static bool stream_capturing(cudaStream_t st) {
  cudaStreamCaptureStatus cap = cudaStreamCaptureStatusNone;
  if (cudaStreamIsCapturing(st, &cap) == cudaSuccess) return cap != cudaStreamCaptureStatusNone;
  cudaGetLastError();
  return false;
}

scgr_status set_cloud(scgr_ctx* c, const float* xyz, int64_t n, bool host, bool ref) {
  if (!c) return SCGR_ERR_INVALID_ARG;
  c->err.clear();
  if (!xyz) return fail(c, SCGR_ERR_INVALID_ARG, "xyz is NULL");
  const int64_t minpts = ref ? c->prm.k : (c->prm.k > 3 ? c->prm.k : 3);
  if (n < minpts) return fail(c, SCGR_ERR_INVALID_ARG, ref ? "reference has fewer than k points" : "template has fewer than max(k, 3) points");
  if (n > (int64_t(1) << 30)) return fail(c, SCGR_ERR_INVALID_ARG, "more than 2^30 points");
  DevBuf& dst = ref ? c->X4 : c->Y4;
  SCGR_CK(c, ensure(dst, (size_t)n * sizeof(float4)));
  const float* src = xyz;
  if (host) {
    SCGR_CK(c, ensure(c->stage, (size_t)n * 3 * sizeof(float)));
    SCGR_CK(c, cudaMemcpyAsync(c->stage.p, xyz, (size_t)n * 3 * sizeof(float), cudaMemcpyHostToDevice, c->stream));
    src = (const float*)c->stage.p;
  }
  SCGR_CK(c, launch_pack(c->L(), src, n, (float4*)dst.p, c->errword));
  if (ref) {
    c->n = n;
    c->have_X = true;
    c->grid_ok[0] = c->coarse_ok = false;
    // a replay of the capture will change the reference without a call
    if (stream_capturing(c->stream)) c->replayed_X = true;
  }
  else { c->m = n; c->have_Y = true; c->grid_ok[1] = false; }
  c->have_desc = false;
  return SCGR_OK;
}

// Launch the force kernel, bracketed by timing events when enabled.
scgr_status force_launch(scgr_ctx* c) {
  const int ntiles = (int)(c->npad / c->fp.tile_j);
  const bool timed = c->timing && !c->capturing;
  if (timed) {
    if (c->ev_used + 2 > c->ev.size()) {
      for (int q = 0; q < 2; ++q) {
        cudaEvent_t e;
        SCGR_CK(c, cudaEventCreate(&e));
        c->ev.push_back(e);
      }
    }
    SCGR_CK(c, cudaEventRecord(c->ev[c->ev_used], c->stream));
  }
  SCGR_CK(c, launch_force(c->L(), c->fp, (const float4*)c->Xr.p, (const float2*)c->XA.p, ntiles,
                          (const float4*)c->Y0r.p, (int)c->mpad, c->pose, c->qexp, (float4*)c->partial.p));
  if (timed) {
    SCGR_CK(c, cudaEventRecord(c->ev[c->ev_used + 1], c->stream));
    c->ev_used += 2;
  }
  return SCGR_OK;
}

// Fold finished event pairs into the tally (the stream must be idle).
scgr_status collect_timing(scgr_ctx* c) {
  for (size_t q = 0; q + 1 < c->ev_used; q += 2) {
    float ms = 0.f;
    SCGR_CK(c, cudaEventElapsedTime(&ms, c->ev[q], c->ev[q + 1]));
    c->timed_ms += ms;
    c->timed_launches += 1;
  }
  c->ev_used = 0;
  return SCGR_OK;
}

// The clouds' descriptions for the grid kernels: which = 0 the reference, 1
// the template; first = 1 puts the template alone at index 0.
static GridCloud grid_cloud(scgr_ctx* c, int which, bool grid, bool stats) {
  GridCloud g{};
  g.P = (const float4*)(which == 0 ? c->X4.p : c->Y4.p);
  g.n = (int)(which == 0 ? c->n : c->m);
  g.spec = (GridSpec*)c->gspec.p + which;
  if (grid) {
    g.cell = (int2*)c->gcell[which].p;
    g.start = (int*)c->gstart[which].p;
    g.tot = (int*)c->gtot[which].p;
    g.sorted = (float4*)c->gsorted[which].p;
  }
  g.knn = (int32_t*)(which == 0 ? c->knnX.p : c->knnY.p);
  DevStats* st = c->stats;
  g.mean = which == 0 ? st->xbar : st->ybar0;
  if (stats) {
    g.scatter = which == 0 ? st->CX : st->S0;
    g.lmax = which == 0 ? &st->eX : &st->eY0;
  } else {
    g.mean = nullptr;
  }
  return g;
}

static scgr_status grid_buffers(scgr_ctx* c, int which) {
  const int64_t n = which == 0 ? c->n : c->m;
  SCGR_CK(c, ensure(c->gcell[which], (size_t)n * sizeof(int2)));
  SCGR_CK(c, ensure(c->gstart[which], grid_start_entries(n) * sizeof(int)));
  SCGR_CK(c, ensure(c->gtot[which], grid_tot_entries(n) * sizeof(int)));
  SCGR_CK(c, ensure(c->gsorted[which], (size_t)n * sizeof(float4)));
  return SCGR_OK;
}

// Whether cloud `which` takes the grid search for its neighbours: always,
// unless SCGR_TUNE_KNN_GRID_MIN has been set above its size.
static bool grid_knn(const scgr_ctx* c, int which) {
  return c->prm.neigh_mode == 0 && (which == 0 ? c->n : c->m) >= (c->knn_grid_min < 0 ? 0 : c->knn_grid_min);
}

// One cloud's grid alone, without statistics.
static scgr_status build_grid(scgr_ctx* c, int which) {
  SCGR_CK(c, ensure(c->gspec, 2 * sizeof(GridSpec)));
  const scgr_status st = grid_buffers(c, which);
  if (st != SCGR_OK) return st;
  CloudSet cs{};
  cs.one[0] = grid_cloud(c, which, true, false);
  SCGR_CK(c, launch_clouds(c->L(), cs, 1, cs.one[0].n, false, false, c->red, (float*)(c->red + 2 * CLOUD_PARTS * 6)));
  SCGR_CK(c, launch_grid_sort(c->L(), cs, 1, cs.one[0].n, c->red));
  c->grid_ok[which] = true;
  if (which == 0) c->coarse_ok = false;
  return SCGR_OK;
}

// The descriptor pass's first part: means, scatter matrices and largest
// eigenvalues of both clouds, their boxes, and the points sorted into grid
// cells where the neighbour search wants that.  Both clouds share each
// launch; nothing waits for the host.
scgr_status prepare_clouds(scgr_ctx* c) {
  c->grid_ok[0] = c->grid_ok[1] = false;
  if (stream_capturing(c->stream)) c->replayed_X = true;  // the grid is there once it is replayed
  SCGR_CK(c, ensure(c->gspec, 2 * sizeof(GridSpec)));
  CloudSet cs{};
  for (int w = 0; w < 2; ++w) {
    if (grid_knn(c, w)) {
      const scgr_status st = grid_buffers(c, w);
      if (st != SCGR_OK) return st;
    }
    cs.one[w] = grid_cloud(c, w, grid_knn(c, w), true);
  }
  const int most = (int)(c->n > c->m ? c->n : c->m);
  double* part = c->red;  // CLOUD_SCRATCH_DOUBLES
  SCGR_CK(c, launch_clouds(c->L(), cs, 2, most, true, grid_knn(c, 0) && grid_knn(c, 1), part,
                           (float*)(part + 2 * CLOUD_PARTS * 6)));
  if (grid_knn(c, 0) && grid_knn(c, 1)) {
    SCGR_CK(c, launch_grid_sort(c->L(), cs, 2, most, part));
  } else if (grid_knn(c, 0) || grid_knn(c, 1)) {
    const int w = grid_knn(c, 0) ? 0 : 1;
    cs.one[0] = cs.one[w];
    cs.one[0].scatter = nullptr;  // finished above
    SCGR_CK(c, launch_grid_sort(c->L(), cs, 1, cs.one[0].n, part));
  }
  for (int w = 0; w < 2; ++w) c->grid_ok[w] = grid_knn(c, w);
  c->coarse_ok = false;
  return SCGR_OK;
}

// k nearest neighbours of both clouds: the grid search or brute force by the
// size and the knob alone, whatever grids earlier calls have left.  Clouds of
// fewer than KNN_FUSED_KEY points keep the key rounding of the brute-force
// search, which served them before (grid_key).
static scgr_status knn_clouds(scgr_ctx* c) {
  const int k = c->prm.k;
  bool grid[2], fused[2];
  CloudSet cs{};
  for (int w = 0; w < 2; ++w) {
    grid[w] = grid_knn(c, w);
    fused[w] = c->knn_grid_min < 0 && (w == 0 ? c->n : c->m) < KNN_FUSED_KEY;
    if (grid[w] && !c->grid_ok[w]) {  // the knob has changed since the descriptor pass
      const scgr_status st = build_grid(c, w);
      if (st != SCGR_OK) return st;
    }
    cs.one[w] = grid_cloud(c, w, grid[w], false);
  }
  if (grid[0] && grid[1] && fused[0] == fused[1]) {
    SCGR_CK(c, launch_knn_grid(c->L(), cs, 2, (int)(c->n > c->m ? c->n : c->m), k, fused[0]));
    return SCGR_OK;
  }
  for (int w = 0; w < 2; ++w) {
    CloudSet one{};
    one.one[0] = cs.one[w];
    if (grid[w]) {
      SCGR_CK(c, launch_knn_grid(c->L(), one, 1, one.one[0].n, k, fused[w]));
    } else {
      SCGR_CK(c, launch_knn(c->L(), one.one[0].P, one.one[0].n, k, one.one[0].knn));
    }
  }
  return SCGR_OK;
}

// Nearest reference point of nq external queries (float32 [nq][3] on the
// device): brute force below nearest_grid_min reference points, else the exact
// two-level grid search over the reference (the same result): fine cells
// around the query, then coarse cells that skip empty space.  The reference's
// grid is the descriptor pass's, or built here on the first query, and kept
// until the reference changes.
//
// A search that a caller captures may be replayed after the reference has
// changed, and brute force reads the points as they then are; from
// CAPTURED_GRID_MIN points on a captured search keeps the grid it finds
// (without one it is brute force: nothing can be allocated).  Where the
// reference itself was set inside a capture, a replay changes it without a
// call, and where the descriptor pass was captured its grid is there only after
// a replay: from then on the grid is built again for every search.
constexpr int64_t CAPTURED_GRID_MIN = 65536;
scgr_status nearest_reference(scgr_ctx* c, const float* q3, int nq, int32_t* idx_out, float* key_out) {
  const float4* X4 = (const float4*)c->X4.p;
  const int n = (int)c->n;
  bool grid = (int64_t)n >= c->nearest_grid_min;
  if (grid && stream_capturing(c->stream))
    grid = (int64_t)n >= CAPTURED_GRID_MIN && c->grid_ok[0] && c->coarse_ok && !c->replayed_X;
  else if (c->replayed_X)
    c->grid_ok[0] = c->coarse_ok = false;
  if (!grid) {
    SCGR_CK(c, launch_nearest(c->L(), X4, n, q3, nq, idx_out, key_out));
    return SCGR_OK;
  }
  if (!c->grid_ok[0]) {
    const scgr_status st = build_grid(c, 0);
    if (st != SCGR_OK) return st;
  }
  CloudSet cs{};
  cs.one[0] = grid_cloud(c, 0, true, false);
  if (!c->coarse_ok) {
    SCGR_CK(c, ensure(c->gccount, grid_start_entries(n) * sizeof(int)));
    SCGR_CK(c, launch_coarse_count(c->L(), cs, n, (int*)c->gccount.p));
    c->coarse_ok = true;
  }
  SCGR_CK(c, launch_nearest_grid(c->L(), cs, c->nearest_levels, (const int*)c->gccount.p, q3, nq, idx_out, key_out));
  return SCGR_OK;
}

// Radius neighbourhoods in Morton order from this size of the larger cloud on:
// the order costs seven launches and saves the pairs beyond the radius (scale 1
// and 0.5, the descriptor pass of n + 0.9 n points, in index order 4,000: 190 and
// 209 us, 6,000: 276 and 274, 8,000: 404 and 399, 40,000: 7222 and 7089; in Morton
// order 209 and 197, 247 and 214, 284 and 242, 1860 and 984).
constexpr int RADIUS_ORDER_MIN = 5120;

// Curvature of both clouds for the current neighbourhood mode (k nearest or
// radius), then sigma (scaled by sigma_scale).
scgr_status curvatures(scgr_ctx* c, int k, double radius_scale, double sigma_scale) {
  const int n = (int)c->n, m = (int)c->m;
  Launch L = c->L();
  const float4* X4 = (const float4*)c->X4.p;
  const float4* Y4 = (const float4*)c->Y4.p;
  DevStats* st = c->stats;
  SCGR_CK(c, ensure(c->sigpart, sigma_part_bytes(n)));
  if (c->prm.neigh_mode == 0) {
    SCGR_CK(c, ensure(c->knnX, (size_t)n * k * sizeof(int32_t)));
    SCGR_CK(c, ensure(c->knnY, (size_t)m * k * sizeof(int32_t)));
    const int k_prev = c->prm.k;
    c->prm.k = k;
    const scgr_status ks = knn_clouds(c);
    if (ks != SCGR_OK) {
      c->prm.k = k_prev;
      return ks;
    }
    SCGR_CK(c, launch_curvature2(L, X4, (const int32_t*)c->knnX.p, n, (double*)c->aX64.p, (float*)c->aX32.p,
                                 (double*)c->sigpart.p, Y4, (const int32_t*)c->knnY.p, m, (double*)c->aY64.p, (float*)c->aY32.p, k));
  } else {
    c->prm.radius_scale = radius_scale;
    const double s2 = radius_scale * radius_scale;
    const bool ordered = (n > m ? n : m) >= RADIUS_ORDER_MIN;
    const size_t bx = radius_scratch_bytes(n, c->num_sms, ordered), by = radius_scratch_bytes(m, c->num_sms, ordered);
    SCGR_CK(c, ensure(c->radpart, bx > by ? bx : by));
    const GridSpec* spec = (const GridSpec*)c->gspec.p;
    const float *bX = nullptr, *bY = nullptr;
    if (ordered) {
      SCGR_CK(c, ensure(c->ord[0], order_bytes(n)));
      SCGR_CK(c, ensure(c->ord[1], order_bytes(m)));
      OrderClouds oc;
      oc.c[0] = order_cloud(c->ord[0].p, X4, spec, n);
      oc.c[1] = order_cloud(c->ord[1].p, Y4, spec + 1, m);
      SCGR_CK(c, launch_order(L, oc));
      X4 = oc.c[0].sorted;
      Y4 = oc.c[1].sorted;
      bX = oc.c[0].box;
      bY = oc.c[1].box;
    }
    SCGR_CK(c, launch_radius_curvature(L, X4, n, bX, &st->eX, s2, spec, c->num_sms, (double*)c->radpart.p,
                                       (double*)c->aX64.p, (float*)c->aX32.p, (double*)c->sigpart.p));
    SCGR_CK(c, launch_radius_curvature(L, Y4, m, bY, &st->eY0, s2, spec + 1, c->num_sms, (double*)c->radpart.p,
                                       (double*)c->aY64.p, (float*)c->aY32.p, nullptr));
  }
  const double user = c->prm.sigma > 0.0 ? c->prm.sigma * sigma_scale : 0.0;
  SCGR_CK(c, launch_sigma_finish(L, (const double*)c->sigpart.p, n, user, sigma_scale, st));
  return SCGR_OK;
}

// The force plan of the context's template rows, the plans of the potential
// and the force VJP beside it, and the buffers whose size they set.  The
// potential runs 1 or 2 points x 128 threads (the shapes its kernel has) in
// whole tiles; the force kernel's knobs do not shape it.
static scgr_status plan_and_size(scgr_ctx* c) {
  const int64_t mloc = c->rows >= 0 ? c->rows : c->m;
  c->fp = plan_force(mloc, c->npad, c->prm.p, c->num_sms, c->ftune);
  c->mpad = force_mpad(mloc, c->fp);
  ForceTuning t;
  t.P = mloc >= 4096 ? 2 : 1;
  t.tpb = 128;
  t.occ = 0;
  ForcePlan& fu = c->fpot;
  fu = plan_force(mloc, c->npad, c->prm.p, c->num_sms, t);
  const int force_splits = fu.splits;
  if (fu.half) {
    fu.half = 0;
    fu.splits = (int)(c->npad / FORCE_TJ);  // of one tile
  }
  SCGR_CK(c, ensure(c->Y0r, (size_t)c->mpad * sizeof(float4)));
  SCGR_CK(c, ensure(c->partial, (size_t)c->fp.splits * c->mpad * sizeof(float4)));
  SCGR_CK(c, ensure(c->blockpart, (size_t)combine_blocks(c->mpad) * 13 * sizeof(double)));
  SCGR_CK(c, ensure(c->fixpart, fixed_part_bytes(c->num_sms)));
  SCGR_CK(c, ensure(c->upart, (size_t)fu.splits * fu.iblocks * sizeof(double)));
  c->vjp = plan_vjp(mloc, c->npad, c->prm.p, c->num_sms, force_splits);
  // its scratch is the force pass's partials (nothing reads them between calls) where they suffice, as they do
  // unless a knob has made them small
  const size_t vjp_bytes = vjp_part_bytes(c->vjp, c->mpad);
  if (vjp_bytes > c->partial.cap) SCGR_CK(c, ensure(c->vjppart, vjp_bytes));
  return SCGR_OK;
}

// A failed allocation leaves the plans without their buffers: no pass may run
// on them, so the descriptors are wanted again.
scgr_status plan_buffers(scgr_ctx* c) {
  const scgr_status st = plan_and_size(c);
  if (st != SCGR_OK) c->have_desc = false;
  return st;
}

// Recompute the force plan (after a tuning change) and the buffers and
// template records that depend on it; descriptors and pose are kept.
scgr_status replan(scgr_ctx* c) {
  const int64_t mloc = c->rows >= 0 ? c->rows : c->m;
  const scgr_status ps = plan_buffers(c);
  if (ps != SCGR_OK) return ps;
  SCGR_CK(c, launch_records(c->L(), (const float4*)c->X4.p, (const double*)c->aX64.p, (int)c->n, (int)c->npad,
                            (const float4*)c->Y4.p + c->row0, (const double*)c->aY64.p + c->row0, (int)mloc,
                            (int)c->mpad, c->prm.g_mode, c->stats, (float4*)c->Xr.p, (float2*)c->XA.p,
                            (float4*)c->Y0r.p));
  drop_graph(c);
  return SCGR_OK;
}

// Odd integer p needs no all-pairs pass per iteration.  For p = 1 the pair
// weight aX s_ij d^0 does not depend on the pose, so the force kernel's
// per-split sums (sum w, sum w X') are the same in every iteration: they are
// computed once.  Templates of the fused tail's size then combine them in
// every iteration (bit-identical to recomputing them); for larger ones the
// iteration's totals come from 22 moments of the sums, and one launch runs all
// iterations (launch_fixed_run; equal up to rounding): 35,000 x 30,800, 200
// iterations 4.6 -> 1.3 ms.
// For p = 3 the sums are a quadratic form in the template point over 14
// pose-free moments of g (computed once per run; an exact re-association, so
// equal to the direct pass up to rounding).
// Small problems of the other exponents run all iterations in one launch of
// a thread-block cluster (launch_small_run) unless the force launches are to be
// timed.  The cluster's 16 SMs bound its pair rate, so from SMALL_MAX_PAIRS on
// the whole GPU is faster, launches and all (an iteration, cluster against
// launches: 500 x 500 7.6 and 20.9 us, 1,000 x 1,000 11.0 and 22.7, 2,000 x
// 2,000 26.4 and 28.4, 3,000 x 1,600 35.8 and 31.7).
constexpr int64_t SMALL_MAX_PAIRS = 4200000;
scgr_status enqueue_iterations(scgr_ctx* c, int iters) {
  const int nb = combine_blocks(c->mpad);
  const StepParams sp = step_params(c);
  const bool pose_free = c->fp.pmode == 1 && c->reuse_pose_free;
  const bool moments = c->fp.pmode == 3 && c->reuse_pose_free;
  const int mloc = (int)(c->rows >= 0 ? c->rows : c->m);
  if (moments && iters > 0) {
    const int ntiles = (int)(c->npad / c->fp.tile_j);
    const int S = moments_splits(ntiles, c->num_sms, c->mpad);
    SCGR_CK(c, ensure(c->mpart, (size_t)S * c->mpad * 14 * sizeof(double)));
    SCGR_CK(c, ensure(c->mom, (size_t)c->mpad * 14 * sizeof(double)));
    SCGR_CK(c, launch_moments(c->L(), (const float4*)c->Xr.p, (const float2*)c->XA.p, ntiles, (const float4*)c->Y0r.p,
                              (int)c->mpad, mloc, S, (double*)c->mpart.p, (double*)c->mom.p));
  }
  const bool fused = c->fused_tail && c->mpad <= FUSED_MAX_SLOTS;
  if (pose_free && !fused && iters > 0) {
    const scgr_status fs = force_launch(c);
    if (fs != SCGR_OK) return fs;
    SCGR_CK(c, launch_fixed_moments(c->L(), (const float4*)c->partial.p, c->fp.splits, (int)c->mpad, mloc,
                                    (const float4*)c->Y0r.p, (const double*)c->aY64.p, c->prm.g_mode, c->stats,
                                    c->num_sms, (double*)c->fixpart.p));
    SCGR_CK(c, launch_fixed_run(c->L(), (const double*)c->fixpart.p, mloc, c->num_sms, c->pose, c->stats, sp, iters,
                                c->errword));
    return SCGR_OK;
  }
  if (fused && c->small_ok && !c->timing && !moments && c->fp.pmode != 1 && c->npad <= SMALL_MAX_POINTS &&
      c->n * c->m <= SMALL_MAX_PAIRS && iters > 0) {
    SCGR_CK(c, launch_small_run(c->L(), c->fp.pmode, (const float4*)c->Xr.p, (const float2*)c->XA.p, (int)c->npad,
                                (const float4*)c->Y0r.p, (const float*)c->aY32.p, c->prm.g_mode, (int)c->m, c->pose,
                                c->stats, sp, c->qexp, iters, c->errword));
    return SCGR_OK;
  }
  for (int t = 0; t < iters; ++t) {
    if (moments) {
      SCGR_CK(c, launch_combine_moments(c->L(), (const double*)c->mom.p, mloc, (int)c->mpad, (const float4*)c->Y0r.p,
                                        (const double*)c->aY64.p, c->prm.g_mode, c->pose, nullptr,
                                        (double*)c->blockpart.p));
      SCGR_CK(c, launch_finalize(c->L(), (const double*)c->blockpart.p, nb, c->pose, c->stats, sp, c->errword));
      continue;
    }
    if (!(pose_free && t > 0)) {
      scgr_status fs = force_launch(c);
      if (fs != SCGR_OK) return fs;
    }
    if (fused) {
      // small templates: combine and finalize in one block (one launch less per iteration)
      SCGR_CK(c, launch_combine_finalize(c->L(), (const float4*)c->partial.p, c->fp.splits, (int)c->mpad, (int)c->m,
                                         (const float4*)c->Y0r.p, (const float*)c->aY32.p, c->prm.g_mode, c->pose,
                                         c->stats, sp, c->errword));
      continue;
    }
    SCGR_CK(c, launch_combine(c->L(), (const float4*)c->partial.p, c->fp.splits, (int)c->mpad, (int)c->m,
                              (const float4*)c->Y0r.p, (const float*)c->aY32.p, c->prm.g_mode, c->pose,
                              nullptr, (double*)c->blockpart.p));
    SCGR_CK(c, launch_finalize(c->L(), (const double*)c->blockpart.p, nb, c->pose, c->stats, sp, c->errword));
  }
  return SCGR_OK;
}

void drop_graph(scgr_ctx* c) {
  if (c->gexec) cudaGraphExecDestroy(c->gexec);
  if (c->graph) cudaGraphDestroy(c->graph);
  c->gexec = nullptr;
  c->graph = nullptr;
  c->graph_iters = -1;
}

}  // namespace api
}  // namespace scgr
