// batch.cu -- batched stepping of many independent simulations (lbm_batch_*).
//
// Every step takes one launch per physics class (body force on or off, BGK or TRT; a
// batch of like simulations has one class) for the bulk tiles of all simulations that
// step in bulk (lbm_sim::fused), with one launch for their boundary tiles beside it on
// a second stream of the batch, and one launch per class for the tiles of the others.
// The steps replay from captured CUDA graphs.
#include <cuda_runtime.h>

#include <algorithm>
#include <string>
#include <vector>

#include "kernels.cuh"
#include "lbm.h"
#include "sim.hpp"

using namespace lbm;

struct lbm_batch_s {
  std::vector<lbm_sim *> sims;
  std::vector<int> base_cur;  // each simulation's buffer index when the entries were built
  std::vector<int> base_ver;  // each simulation's version when the entries were built
  int lattice = 0, dtype = 1;
  cudaStream_t stream = nullptr;
  BatchEntry *entries = nullptr;
  int4 *tiles = nullptr;
  long long ntiles = 0;
  struct Range {
    long long first = 0, count = 0;
    int smem = 0;  // dynamic shared memory of a block
  };
  Range bulk[4], rest[4], boundary;  // tiles by physics class: bulk tiles, the other simulations'; boundary tiles
  cudaStream_t aux = nullptr;        // the boundary tiles' stream, forked and joined around every step
  cudaEvent_t ev_fork = nullptr, ev_join = nullptr;
  cudaStream_t cap = nullptr;        // the stream that steps are captured on
  int bx = 32, by = 4, variant = 3, T = 1;
  bool tiles_ok = false;
  int parity = 0;  // batch steps taken since the entries were built, mod 2
  cudaGraphExec_t graph[2] = {nullptr, nullptr};
  std::string err;
};

static constexpr int kBatchGraphSteps = 32;

static int bfail(lbm_batch b, int code, const std::string &msg) {
  if (b) b->err = msg;
  return code;
}

#define B_CUDA(b, call)                                                                          \
  do {                                                                                           \
    cudaError_t e_ = (call);                                                                     \
    if (e_ != cudaSuccess)                                                                       \
      return bfail((b), e_ == cudaErrorMemoryAllocation ? LBM_ERR_OOM : LBM_ERR_CUDA,           \
                   std::string(#call) + ": " + cudaGetErrorString(e_));                          \
  } while (0)

// One step of the whole batch. The kernels of a step only read the buffers of one
// parity and write disjoint slots of the other, so that they need no order.
static cudaError_t batch_launch(const lbm_batch_s *b, int parity) {
  Launch l;
  l.block = dim3(b->bx, b->by, 1);
  const auto run = [&](int kind, int phys, const lbm_batch_s::Range &r, int T, cudaStream_t st) {
    if (r.count == 0) return cudaSuccess;
    l.stream = st;
    l.smem = r.smem;
    l.grid = dim3((unsigned)((r.count + T - 1) / T));
    return launch_step_batch(b->lattice, b->dtype, b->variant, kind, phys, b->entries, b->tiles + r.first,
                             (int)r.count, T, parity, l);
  };
  cudaError_t e = cudaSuccess;
  const bool fork = b->boundary.count > 0;
  if (fork) {
    e = cudaEventRecord(b->ev_fork, b->stream);
    if (e == cudaSuccess) e = cudaStreamWaitEvent(b->aux, b->ev_fork, 0);
    if (e == cudaSuccess) e = run(kBatchBoundary, 0, b->boundary, 1, b->aux);
  }
  for (int c = 0; c < 4 && e == cudaSuccess; ++c) e = run(kBatchBulk, c, b->bulk[c], b->T, b->stream);
  for (int c = 0; c < 4 && e == cudaSuccess; ++c) e = run(kBatchStep, c, b->rest[c], b->T, b->stream);
  if (fork && e == cudaSuccess) {
    e = cudaEventRecord(b->ev_join, b->aux);
    if (e == cudaSuccess) e = cudaStreamWaitEvent(b->stream, b->ev_join, 0);
  }
  return e;
}

static void drop_batch_graphs(lbm_batch b) {
  for (int k = 0; k < 2; ++k)
    if (b->graph[k]) { cudaGraphExecDestroy(b->graph[k]); b->graph[k] = nullptr; }
}

// Entries (views and buffers at the current buffer index of each simulation) and
// the tile table for the batch's launch shape.
static int build_batch(lbm_batch b) {
  const int n = (int)b->sims.size();
  std::vector<BatchEntry> e(n);
  std::vector<int4> t;
  b->base_cur.resize(n);
  b->base_ver.resize(n);
  const int tpb = b->bx * b->by;
  // The tables one after another: per physics class the bulk tiles and the other
  // simulations' tiles, in batch order, then the boundary tiles of the former.
  std::vector<int4> bulk[4], rest[4], bnd;
  lbm_batch_s::Range rb[4], rr[4], rbnd;
  for (int k = 0; k < n; ++k) {
    lbm_sim *s = b->sims[k];
    const int c = (s->has_force ? PH_FORCE : 0) | (s->collision == LBM_COLL_TRT ? PH_TRT : 0);
    const int save_bx = s->step_bx, save_var = s->variant;
    s->step_bx = b->bx;        // the view's tile-row count follows the batch's block width
    s->variant = b->variant;   // and its one-node lattice tiles (a simulation may be set to node pairs)
    e[k].v = s->view();
    const bool fused = s->fused();
    s->step_bx = save_bx;
    s->variant = save_var;
    e[k].v.tiles = nullptr;
    e[k].f0 = s->f[s->cur];
    e[k].f1 = s->f[s->cur ^ 1];
    b->base_cur[k] = s->cur;
    b->base_ver[k] = s->version;
    const int gx = s->nxp / b->bx, gy = (s->ny + b->by - 1) / b->by;
    std::vector<int4> &lat = fused ? bulk[c] : rest[c], &bt = fused ? bnd : rest[c];
    lbm_batch_s::Range &rl = fused ? rb[c] : rr[c];
    if (fused) rl.smem = std::max(rl.smem, s->step_smem(tpb, false, s->nb > 0));
    else if (s->nb > 0) rl.smem = std::max(rl.smem, s->step_smem(tpb, true, false));
    std::vector<uint32_t> hc(fused || s->nb == 0 ? 0 : s->np / 32 + 1, 0u);
    if (!hc.empty()) {
      B_CUDA(b, cudaMemcpyAsync(hc.data(), s->cbase, hc.size() * sizeof(uint32_t), cudaMemcpyDeviceToHost, b->stream));
      B_CUDA(b, cudaStreamSynchronize(b->stream));
    }
    const long long pchunks = (long long)s->nxp * s->ny / 32;
    for (int z = 0; z < s->nz; ++z) {
      for (int i = 0; i < gx * gy; ++i)
        lat.push_back(fused ? make_int4(k, z, i % gx, i / gx) : make_int4(k, z, i, 0));
      if (s->nb == 0) continue;
      const long long r0 = fused ? s->rplane[z] : hc[z * pchunks], r1 = fused ? s->rplane[z + 1] : hc[(z + 1) * pchunks];
      for (long long r = r0; r < r1; r += tpb)
        bt.push_back(make_int4(k, -1, (int)r, (int)std::min<long long>(tpb, r1 - r)));
    }
    if (fused && !bnd.empty()) rbnd.smem = std::max(rbnd.smem, s->step_smem(tpb, true, false));
  }
  const auto place = [&](const std::vector<int4> &src, lbm_batch_s::Range &r) {
    r.first = (long long)t.size();
    r.count = (long long)src.size();
    t.insert(t.end(), src.begin(), src.end());
  };
  for (int c = 0; c < 4; ++c) {
    place(bulk[c], rb[c]);
    place(rest[c], rr[c]);
    b->bulk[c] = rb[c];
    b->rest[c] = rr[c];
  }
  place(bnd, rbnd);
  b->boundary = rbnd;
  if (rbnd.count > 0 && !b->aux) {  // highest priority: the boundary blocks start as soon as the step does
    int lo = 0, hi = 0;
    B_CUDA(b, cudaDeviceGetStreamPriorityRange(&lo, &hi));
    B_CUDA(b, cudaStreamCreateWithPriority(&b->aux, cudaStreamNonBlocking, hi));
    B_CUDA(b, cudaEventCreateWithFlags(&b->ev_fork, cudaEventDisableTiming));
    B_CUDA(b, cudaEventCreateWithFlags(&b->ev_join, cudaEventDisableTiming));
  }
  drop_batch_graphs(b);
  cudaFree(b->entries);
  cudaFree(b->tiles);
  b->entries = nullptr;
  b->tiles = nullptr;
  b->ntiles = (long long)t.size();
  if (b->ntiles >= (1LL << 31)) return bfail(b, LBM_ERR_ARG, "batch too large: more than 2^31 tiles");
  B_CUDA(b, cudaMalloc(&b->entries, n * sizeof(BatchEntry)));
  B_CUDA(b, cudaMalloc(&b->tiles, std::max<long long>(1, b->ntiles) * sizeof(int4)));
  B_CUDA(b, cudaMemcpyAsync(b->entries, e.data(), n * sizeof(BatchEntry), cudaMemcpyHostToDevice, b->stream));
  if (b->ntiles)
    B_CUDA(b, cudaMemcpyAsync(b->tiles, t.data(), b->ntiles * sizeof(int4), cudaMemcpyHostToDevice, b->stream));
  B_CUDA(b, cudaStreamSynchronize(b->stream));
  b->parity = 0;
  b->tiles_ok = true;
  return LBM_OK;
}

// The entries are valid while every simulation is still at its recorded buffer
// index shifted by the batch's own steps, with unchanged options and geometry.
static bool entries_current(const lbm_batch_s *b) {
  if (!b->tiles_ok || b->base_cur.size() != b->sims.size()) return false;
  for (size_t k = 0; k < b->sims.size(); ++k)
    if (b->sims[k]->cur != (b->base_cur[k] ^ b->parity) || b->sims[k]->version != b->base_ver[k] ||
        !b->sims[k]->geom_ok)
      return false;
  return b->tiles_ok;
}

static int batch_direct(lbm_batch b, int n) {
  for (int k = 0; k < n; ++k) {
    cudaError_t e = batch_launch(b, b->parity);
    if (e != cudaSuccess) return bfail(b, LBM_ERR_CUDA, cudaGetErrorString(e));
    b->parity ^= 1;
    for (lbm_sim *s : b->sims) s->cur ^= 1;
  }
  return LBM_OK;
}

// A graph of n steps from parity p, captured on a stream of the batch's own (see lbm_sim::capture).
static int batch_capture(lbm_batch b, int n, int p, cudaGraphExec_t *out) {
  if (!b->cap) B_CUDA(b, cudaStreamCreateWithFlags(&b->cap, cudaStreamNonBlocking));
  const cudaStream_t user = b->stream;
  b->stream = b->cap;
  cudaGraph_t g = nullptr;
  cudaError_t e = cudaStreamBeginCapture(b->stream, cudaStreamCaptureModeThreadLocal);
  if (e == cudaSuccess) {
    cudaError_t l = cudaSuccess;
    for (int k = 0; k < n && l == cudaSuccess; ++k) l = batch_launch(b, (p + k) & 1);
    e = cudaStreamEndCapture(b->stream, &g);
    if (l != cudaSuccess) e = l;
  }
  b->stream = user;
  if (e != cudaSuccess) {
    if (g) cudaGraphDestroy(g);
    return bfail(b, LBM_ERR_CUDA, std::string("capture: ") + cudaGetErrorString(e));
  }
  e = cudaGraphInstantiate(out, g, 0);
  cudaGraphDestroy(g);
  if (e != cudaSuccess) { *out = nullptr; return bfail(b, LBM_ERR_CUDA, cudaGetErrorString(e)); }
  return LBM_OK;
}

extern "C" int lbm_batch_create(const lbm_handle *sims, int n, lbm_batch *out) {
  if (!out || !sims || n < 1) return LBM_ERR_ARG;
  *out = nullptr;
  lbm_batch b = new lbm_batch_s();
  for (int k = 0; k < n; ++k) {
    lbm_sim *s = sims[k];
    if (!s) { delete b; return LBM_ERR_ARG; }
    if (!s->geom_ok || !s->state_ok) { delete b; return LBM_ERR_STATE; }
    if (s->mb.on) { delete b; return LBM_ERR_ARG; }  // moving bodies step alone
    if (k == 0) {
      b->lattice = s->lattice;
      b->dtype = s->dtype;
      b->stream = s->stream;
    } else if (s->lattice != b->lattice || s->dtype != b->dtype || s->stream != b->stream) {
      delete b;
      return LBM_ERR_ARG;  // one lattice, one storage type and one stream per batch
    }
    for (int j = 0; j < k; ++j)
      if (sims[j] == s) { delete b; return LBM_ERR_ARG; }
    b->sims.push_back(s);
  }
  if (b->dtype == LBM_F64) b->variant = 0;
  *out = b;
  return LBM_OK;
}

extern "C" int lbm_batch_destroy(lbm_batch b) {
  if (!b) return LBM_OK;
  if (b->stream) cudaStreamSynchronize(b->stream);
  drop_batch_graphs(b);
  cudaFree(b->entries);
  cudaFree(b->tiles);
  if (b->aux) { cudaStreamSynchronize(b->aux); cudaStreamDestroy(b->aux); }
  if (b->cap) cudaStreamDestroy(b->cap);
  if (b->ev_fork) cudaEventDestroy(b->ev_fork);
  if (b->ev_join) cudaEventDestroy(b->ev_join);
  delete b;
  return LBM_OK;
}

extern "C" const char *lbm_batch_last_error(lbm_batch b) { return b ? b->err.c_str() : ""; }

extern "C" int lbm_batch_set_launch(lbm_batch b, int bx, int by, int variant, int tiles) {
  if (!b) return LBM_ERR_ARG;
  if (bx < 32 || bx % 32 || by < 1 || bx * by > 256 || variant < 0 || variant > 3 || tiles < 1 || tiles > 4)
    return bfail(b, LBM_ERR_ARG, "invalid launch configuration");
  if (b->dtype == LBM_F64 && variant != 0) return bfail(b, LBM_ERR_ARG, "FP64 takes variant 0 only");
  if (b->dtype == LBM_F64 && b->lattice == LBM_D3Q27 && bx * by > 128)
    return bfail(b, LBM_ERR_ARG, "FP64 on D3Q27 takes at most 128 threads per block (shared staging)");
  for (lbm_sim *s : b->sims)
    if (s->nxp % bx) return bfail(b, LBM_ERR_ARG, "bx must divide the padded row length of every simulation");
  b->bx = bx; b->by = by; b->variant = variant; b->T = tiles;
  b->tiles_ok = false;
  drop_batch_graphs(b);
  return LBM_OK;
}

extern "C" int lbm_batch_step(lbm_batch b, int n) {
  if (!b) return LBM_ERR_ARG;
  if (n < 0) return bfail(b, LBM_ERR_ARG, "negative step count");
  if (n == 0) return LBM_OK;
  for (lbm_sim *s : b->sims) {
    if (!s->geom_ok || !s->state_ok) return bfail(b, LBM_ERR_STATE, "a simulation lost its geometry or state");
    if (s->mb.on) return bfail(b, LBM_ERR_ARG, "a simulation with a moving body cannot be batched");
  }
  if (!entries_current(b)) {
    int rc = build_batch(b);
    if (rc) return rc;
  }
  cudaStreamCaptureStatus capturing = cudaStreamCaptureStatusNone;  // by the caller, into whose graph no other launches
  B_CUDA(b, cudaStreamIsCapturing(b->stream, &capturing));
  if (capturing != cudaStreamCaptureStatusNone) return batch_direct(b, n);
  int reps = n / kBatchGraphSteps, rest = n % kBatchGraphSteps;
  if (reps > 0) {
    const int p = b->parity;
    if (!b->graph[p]) {
      int rc = batch_capture(b, kBatchGraphSteps, p, &b->graph[p]);
      if (rc) return rc;
    }
    for (int k = 0; k < reps; ++k) B_CUDA(b, cudaGraphLaunch(b->graph[p], b->stream));
    // kBatchGraphSteps is even: parities and buffer indices are unchanged
  }
  return batch_direct(b, rest);
}

// Time of `steps` steps at the launch in use, as lbm_batch_step runs them: replayed from a
// graph (at most kBatchGraphSteps long).
static int time_batch(lbm_batch b, int steps, cudaEvent_t e0, cudaEvent_t e1, float *ms) {
  const int len = std::min(steps, kBatchGraphSteps);
  cudaGraphExec_t g = nullptr;
  int rc = build_batch(b);
  if (rc == LBM_OK) rc = batch_direct(b, 2);
  if (rc == LBM_OK) rc = batch_capture(b, len, b->parity, &g);
  if (rc) return rc;
  cudaError_t e = cudaGraphUpload(g, b->stream);
  if (e == cudaSuccess) e = cudaEventRecord(e0, b->stream);
  for (int n = steps; n >= len && e == cudaSuccess; n -= len) e = cudaGraphLaunch(g, b->stream);
  if (e == cudaSuccess && (len & 1)) {  // an odd graph runs once and ends at the other buffers
    b->parity ^= 1;
    for (lbm_sim *s : b->sims) s->cur ^= 1;
  }
  if (e == cudaSuccess) rc = batch_direct(b, steps % len);
  if (e == cudaSuccess) e = cudaEventRecord(e1, b->stream);
  if (e == cudaSuccess) e = cudaEventSynchronize(e1);
  if (e == cudaSuccess) e = cudaEventElapsedTime(ms, e0, e1);
  cudaGraphExecDestroy(g);
  if (e != cudaSuccess) return bfail(b, LBM_ERR_CUDA, cudaGetErrorString(e));
  return rc;
}

extern "C" int lbm_batch_autotune(lbm_batch b, int steps, int *bx, int *by, int *variant, int *tiles,
                                  double *ms_per_step) {
  if (!b || steps < 1) return LBM_ERR_ARG;
  cudaEvent_t e0, e1;
  B_CUDA(b, cudaEventCreate(&e0));
  B_CUDA(b, cudaEventCreate(&e1));
  int best[4] = {b->bx, b->by, b->variant, b->T};
  float best_ms = 1e30f;
  int rc = time_batch(b, steps, e0, e1, &best_ms);  // the launch in use is the one to beat
  const int topts[3] = {1, 2, 4};
  const int max_threads = (b->dtype == LBM_F64 && b->lattice == LBM_D3Q27) ? 128 : 256;  // shared staging
  for (int threads = 128; threads <= max_threads && rc == LBM_OK; threads *= 2)
    for (int bxx = 32; bxx <= threads && rc == LBM_OK; bxx *= 2) {
      bool ok = true;
      for (lbm_sim *s : b->sims) ok = ok && (s->nxp % bxx == 0);
      if (!ok) continue;
      for (int var = 0; var <= (b->dtype == LBM_F64 ? 0 : 3) && rc == LBM_OK; var += 3)  // 1 and 2: the kernels of 0
        for (int k = 0; k < 3 && rc == LBM_OK; ++k) {
          rc = lbm_batch_set_launch(b, bxx, threads / bxx, var, topts[k]);
          if (rc) break;
          float ms = 1e30f;
          rc = time_batch(b, steps, e0, e1, &ms);
          if (rc == LBM_OK && ms < best_ms) { best_ms = ms; best[0] = bxx; best[1] = threads / bxx; best[2] = var; best[3] = topts[k]; }
        }
    }
  cudaEventDestroy(e0);
  cudaEventDestroy(e1);
  if (rc) return rc;
  rc = lbm_batch_set_launch(b, best[0], best[1], best[2], best[3]);
  if (rc) return rc;
  if (bx) *bx = best[0];
  if (by) *by = best[1];
  if (variant) *variant = best[2];
  if (tiles) *tiles = best[3];
  if (ms_per_step) *ms_per_step = best_ms / steps;
  return LBM_OK;
}
