// The tile autotuner (ddfd_autotune, ddfd_batch_autotune): times a few
// forward and adjoint steps per candidate z depth of the thread-block tiles
// with CUDA events: first the full items' depth (the lean ones' fixed), then, in
// FP32, the lean items' depth.  The depth that the handle has is timed first and
// stays unless a candidate is faster.  A GPU tuning aid; the paper has no
// counterpart.
#include "ddfd_host.h"

using namespace ddfd;
using namespace ddfd::host;

namespace {

const int kTileKz[] = {4, 6, 8, 12, 16, 24, 32};

// A candidate replaces the handle's depth if it is faster by more than two timings of
// one depth differ (up to 0.5 %, 13^3 to 301^3).
constexpr float kGain = 0.99f;

// Runs trial(kz, kz_lean, &ms) for the handle's z depth of one kind of item and for
// every candidate, the other kind's held; *kz (lean = false) or *kz_lean (lean =
// true) becomes the depth to run with, *fastest the fastest candidate.
template <typename Trial>
int autotune_one(int n, bool lean, Trial trial, int *kz, int *kz_lean, int *fastest) {
  int st;
  float kept_ms = 0.0f, best_ms = 3.4e38f;
  int &depth = lean ? *kz_lean : *kz;
  const int kept = depth;
  auto run = [&](int c, float *ms) { return lean ? trial(*kz, c, ms) : trial(c, *kz_lean, ms); };
  if ((st = run(kept, &kept_ms))) return st;
  bool listed = false;  // the kept depth is itself a candidate
  for (int c : kTileKz) {
    if (c > n) break;
    if (c == kept) {
      listed = true;
      continue;
    }
    float ms = 0.0f;
    if ((st = run(c, &ms))) return st;
    if (ms < best_ms) {
      best_ms = ms;
      *fastest = c;
    }
  }
  if (best_ms < kGain * kept_ms)
    depth = *fastest;
  else if (listed)
    *fastest = kept;
  return DDFD_OK;
}

template <typename Trial>
int autotune_kz(int n, bool fp32, Trial trial, int *kz, int *kz_lean, int *fastest) {
  int fastest_lean = 0;
  int st = autotune_one(n, false, trial, kz, kz_lean, fastest);
  if (!st && fp32) st = autotune_one(n, true, trial, kz, kz_lean, &fastest_lean);
  return st;
}

// Times what enqueue(stream, &launches) puts into a graph, as the sequences run
// (launched eagerly, a small grid's steps would wait for the host): the faster of two
// runs after an untimed one, each after clear(stream).
template <typename Clear, typename Enqueue>
cudaError_t time_steps(cudaStream_t cap, cudaStream_t sm, const cudaEvent_t *ev, Clear clear, Enqueue enqueue, float *ms,
                       int64_t *launches) {
  int64_t nk = 0;
  cudaError_t e = cudaStreamBeginCapture(cap, cudaStreamCaptureModeRelaxed);
  if (e != cudaSuccess) return e;
  enqueue(cap, &nk);
  const cudaError_t el = cudaGetLastError();
  cudaGraph_t g = nullptr;
  cudaGraphExec_t ge = nullptr;
  e = cudaStreamEndCapture(cap, &g);
  if (e == cudaSuccess) e = el;
  if (e == cudaSuccess) e = cudaGraphInstantiate(&ge, g, 0);
  *ms = 3.4e38f;
  for (int r = 0; e == cudaSuccess && r < 3; ++r) {
    float t = 0.0f;
    if ((e = clear(sm)) || (e = cudaEventRecord(ev[0], sm)) || (e = cudaGraphLaunch(ge, sm)) ||
        (e = cudaEventRecord(ev[1], sm)) || (e = cudaEventSynchronize(ev[1])) ||
        (e = cudaEventElapsedTime(&t, ev[0], ev[1])))
      break;
    if (r > 0) *ms = std::min(*ms, t);
    *launches += nk;
  }
  if (ge) cudaGraphExecDestroy(ge);
  if (g) cudaGraphDestroy(g);
  return e;
}

// Fields of the new nodes of a refined mesh, cleared.
cudaError_t clear_new_nodes(ddfd_problem *p, cudaStream_t sm) {
  cudaError_t e = cudaSuccess;
  for (int q = 0; q < 2 && p->n_new && e == cudaSuccess; ++q) {
    e = cudaMemsetAsync(p->X[q], 0, 3 * (size_t)p->n_new * p->esz, sm);
    if (e == cudaSuccess && p->XMu[q]) e = cudaMemsetAsync(p->XMu[q], 0, 3 * (size_t)p->n_new * p->esz, sm);
  }
  return e;
}

// E^n on the free nodes for trial step st (any valid slot of the history).
long long trial_hist_index(const ddfd_problem *p, int st) {
  return p->nsnap ? (long long)(st % p->seg) + 1 : (long long)st + 1;
}

template <typename T>
int single_trial(ddfd_problem *p, int steps, int kz, int kz_lean, float *ms) {
  const size_t fbytes = 3 * (size_t)p->cs * sizeof(T);
  const size_t trn = (size_t)p->n_src * (p->Nt + 1) * p->n_det * 3;
  p->kz = kz;
  p->kz_lean = kz_lean;
  if (int bs = build_items(p)) return bs;  // the trial runs the dispatch order (and split) of these depths
  auto clear = [&](cudaStream_t sm) {
    cudaError_t e = clear_new_nodes(p, sm);
    for (int q = 0; q < 2 && e == cudaSuccess; ++q) {
      e = cudaMemsetAsync(p->E[q], 0, fbytes, sm);
      if (e == cudaSuccess && p->Mu[q]) e = cudaMemsetAsync(p->Mu[q], 0, fbytes, sm);
    }
    return e != cudaSuccess || !trn ? e : cudaMemsetAsync(p->res, 0, trn * sizeof(double), sm);
  };
  auto enqueue = [&](cudaStream_t sm, int64_t *nk) {
    StepParams<T> P = base_params<T>(p);
    set_source(P, p, 0);
    int ic = 1, io = 0;
    bool chained = false;  // as in the sequences: every kernel but the first follows a kernel
    for (int st = 0; st < steps; ++st) {
      set_forward_step(P, p, 0, st, p->E[ic], p->E[io],
                       p->fonly ? nullptr : (T *)p->hist + trial_hist_index(p, st) * 3 * p->hcs);
      enqueue_ebe<T>(p, p->E[ic], false, sm, nk, p->X[ic], nullptr, chained);
      chained = chained || p->ebe_rows > 0;
      *nk += launch_forward_step(single_launch(P, p->mE_halo[ic], p->mE_ctr[io], p, chained), sm);
      enqueue_new_step<T>(p, p->X[ic], p->X[io], false, P, sm, nk);
      chained = true;
      std::swap(ic, io);
    }
    ic = 1, io = 0;
    for (int k = p->fonly ? 0 : steps; k >= 1; --k) {  // forward_only handles time the forward alone
      set_adjoint_step(P, p, 0, k, p->Mu[ic], p->Mu[io],
                       (const T *)p->hist + trial_hist_index(p, k - 1) * 3 * p->hcs, steps);
      enqueue_ebe<T>(p, p->Mu[ic], true, sm, nk, p->XMu[ic], nullptr, true);
      *nk += launch_adjoint_step(single_launch(P, p->mM_halo[ic], p->mM_ctr[io], p, true), sm);
      enqueue_new_step<T>(p, p->XMu[ic], p->XMu[io], true, P, sm, nk);
      std::swap(ic, io);
    }
  };
  CK(time_steps(p->cap_stream, p->stream, p->ev, clear, enqueue, ms, &p->launches));
  return DDFD_OK;
}

template <typename T>
int batch_trial(ddfd_batch *b, int steps, int kz, int kz_lean, float *ms) {
  const size_t slab = 3 * (size_t)b->cs * sizeof(T) * b->m.size();
  b->kz = kz;
  b->kz_lean = kz_lean;
  if (int bs = build_batch_items(b)) return bs;  // the trial runs the dispatch orders of these depths
  auto clear = [&](cudaStream_t sm) {
    cudaError_t e = cudaSuccess;
    for (int q = 0; q < 2 && e == cudaSuccess; ++q) {
      e = cudaMemsetAsync(b->E[q], 0, slab, sm);
      if (e == cudaSuccess && b->Mu[q]) e = cudaMemsetAsync(b->Mu[q], 0, slab, sm);
    }
    for (ddfd_problem *p : b->m) {
      const size_t trn = (size_t)(p->Nt + 1) * p->n_det * 3;
      if (e == cudaSuccess) e = clear_new_nodes(p, sm);
      if (e == cudaSuccess && trn) e = cudaMemsetAsync(p->res, 0, trn * sizeof(double), sm);
    }
    return e;
  };
  const std::vector<int> all = all_members(b);
  bool any_fonly = false;
  for (ddfd_problem *p : b->m) any_fonly |= p->fonly;
  auto enqueue = [&](cudaStream_t sm, int64_t *nk) {
    bool chained = false;
    // one step of the batch: the members' gathers, the step, the new nodes
    auto step = [&](bool adj, int ic, int io, auto fill) {
      for (ddfd_problem *p : b->m) {
        enqueue_ebe<T>(p, adj ? p->Mu[ic] : p->E[ic], adj, sm, nk, adj ? p->XMu[ic] : p->X[ic], b->errflag, chained);
        chained = chained || p->ebe_rows > 0;
      }
      launch_groups<T>(b, adj, all, adj ? b->maps.M_halo[ic] : b->maps.E_halo[ic],
                       adj ? b->maps.M_ctr[io] : b->maps.E_ctr[io], fill, sm, nk, &b->items_all, chained);
      chained = true;
      for (ddfd_problem *p : b->m)
        if (p->n_new) {
          StepParams<T> P = base_params<T>(p);
          fill(P, p);
          enqueue_new_step<T>(p, adj ? p->XMu[ic] : p->X[ic], adj ? p->XMu[io] : p->X[io], adj, P, sm, nk);
        }
    };
    int ic = 1, io = 0;
    for (int st = 0; st < steps; ++st) {
      step(false, ic, io, [&](StepParams<T> &P, ddfd_problem *p) {
        set_forward_step(P, p, 0, st, p->E[ic], p->E[io],
                         p->fonly ? nullptr : (T *)p->hist + trial_hist_index(p, st) * 3 * p->hcs);
      });
      std::swap(ic, io);
    }
    ic = 1, io = 0;
    for (int k = any_fonly ? 0 : steps; k >= 1; --k) {  // forward_only members: forward trials only
      step(true, ic, io, [&](StepParams<T> &P, ddfd_problem *p) {
        set_adjoint_step(P, p, 0, k, p->Mu[ic], p->Mu[io],
                         (const T *)p->hist + trial_hist_index(p, k - 1) * 3 * p->hcs, steps);
      });
      std::swap(ic, io);
    }
  };
  BCK(time_steps(b->cap_stream, b->stream, b->ev, clear, enqueue, ms, &b->launches));
  return DDFD_OK;
}

}  // namespace

extern "C" {

int ddfd_autotune(ddfd_problem *p, int32_t steps, int32_t *tile_kz_out) {
  if (!p) return DDFD_E_ARG;
  p->err.clear();
  if (steps < 1 || steps > p->Nt) return fail(p, DDFD_E_ARG, "steps must be in [1, n_steps]");
  const int kz0 = p->kz, kzl0 = p->kz_lean;
  int kz = kz0, kzl = kzl0, fastest = 0;
  int st = autotune_kz(
      p->n, p->fp32 != 0,
      [&](int a, int l, float *ms) {
        return p->fp32 ? single_trial<float>(p, steps, a, l, ms) : single_trial<double>(p, steps, a, l, ms);
      },
      &kz, &kzl, &fastest);
  if (!st && (st = check_err(p))) kz = kz0, kzl = kzl0;
  p->kz = kz;
  p->kz_lean = kzl;
  p->state = ST_READY;
  drop_graphs(p);
  if (!st) st = build_items(p);
  const size_t fbytes = 3 * (size_t)p->cs * p->esz;
  for (int q = 0; q < 2; ++q) {
    CK(cudaMemsetAsync(p->E[q], 0, fbytes, p->stream));
    if (p->Mu[q]) CK(cudaMemsetAsync(p->Mu[q], 0, fbytes, p->stream));
  }
  if (st) return st;
  if (tile_kz_out) *tile_kz_out = fastest;
  return sync_check(p);
}

int ddfd_batch_autotune(ddfd_batch *b, int32_t steps, int32_t *tile_kz_out) {
  if (!b) return DDFD_E_ARG;
  b->err.clear();
  if (steps < 1 || steps > b->Nt) return bfail(b, DDFD_E_ARG, "steps must be in [1, n_steps]");
  const int kz0 = b->kz, kzl0 = b->kz_lean;
  int kz = kz0, kzl = kzl0, fastest = 0;
  int st = autotune_kz(
      b->n, b->fp32 != 0,
      [&](int a, int l, float *ms) {
        return b->fp32 ? batch_trial<float>(b, steps, a, l, ms) : batch_trial<double>(b, steps, a, l, ms);
      },
      &kz, &kzl, &fastest);
  if (!st && (st = batch_check_err(b))) kz = kz0, kzl = kzl0;
  b->kz = kz;
  b->kz_lean = kzl;
  drop_batch_graphs(b);
  for (ddfd_problem *p : b->m) {
    p->kz = b->kz;
    p->kz_lean = b->kz_lean;
    p->state = ST_READY;
    drop_graphs(p);
    if (!st && (st = build_items(p))) b->err = p->err;
  }
  if (!st) st = build_batch_items(b);
  const size_t slab = 3 * (size_t)b->cs * b->esz * b->m.size();
  for (int q = 0; q < 2; ++q) {
    BCK(cudaMemsetAsync(b->E[q], 0, slab, b->stream));
    if (b->Mu[q]) BCK(cudaMemsetAsync(b->Mu[q], 0, slab, b->stream));
  }
  if (st) return st;
  if (tile_kz_out) *tile_kz_out = fastest;
  BCK(cudaStreamSynchronize(b->stream));
  return DDFD_OK;
}

}  // extern "C"
