// Plan groups: several domains' extension + DFT pipelines (steps 5-7 of Section 3.5) in
// one call, every plan's work on its own stream forked from the caller's and joined back,
// so that the kernels of small domains run side by side.  Two forms: "branches", each
// plan's whole call on its stream; "persistent", the strip-point values of every
// mixed-form member (the fused blend + interpolation, steps 5-6) from one persistent
// kernel over all members' work items (plan, owner range, function), longest first, and
// then each plan's row and column DFTs on its stream (FP64 members: their whole call).
//
// The form, and the persistent kernel's CTA shape, are timed once for a set of function
// counts.  A call launches its kernels directly, whatever its buffers: capturing and
// instantiating a graph for new buffers costs more host time (and, timed on them, more
// device time) than the work itself: eight stars of 256^2 .. 2048^2 with 32 functions each
// took 34.8 ms per call when every call came with other buffers, the kernels 2.6 ms of it.
// A call with the arguments of the call before it is captured as a CUDA graph, which is
// replayed while the arguments (function counts and pointers) and every plan's workspace
// (base and size) stay the same.  The workspace is part of the key because the captured
// kernels hold its address: a later call on a member plan that needs more workspace frees
// the old one and allocates another, and a replay would then use freed memory.
#include <cuda_runtime.h>

#include <algorithm>
#include <cstring>
#include <numeric>
#include <vector>

#include "../../include/fc2d.h"
#include "fc2d_kernels.cuh"
#include "plan_internal.h"

namespace fc2d {
// capi.cu
fc2d_status ensure_plan_workspace(fc2d_plan_s* p, int n_f);
fc2d_status extend_coeffs_check(fc2d_plan_s* p, int n_f, const double* fg, const double* fb,
                                const void* fhat);
fc2d_status extend_coeffs_dft(fc2d_plan_s* p, int n_f, const double* fg, void* fhat,
                              cudaStream_t s);
bool group_fused(const fc2d_plan_s* p);
GiPlanArgs group_fused_args(fc2d_plan_s* p, int n_f, const double* fg, const double* fb,
                            std::vector<int32_t>* points);
}  // namespace fc2d

// A work item's cost for the ordering: its strip points plus a fixed part for the
// tables, the gather of 64 normals and the MMAs (about as long as interpolating this
// many points).
constexpr int64_t kItemFixed = 256;

struct fc2d_group_s {
  std::vector<fc2d_plan_t> plans;
  std::vector<cudaStream_t> branch;       // one stream per plan
  cudaStream_t cap = nullptr;             // tuning runs, and the capture origin
  cudaEvent_t fork = nullptr;
  std::vector<cudaEvent_t> join;
  cudaGraph_t graph = nullptr;
  cudaGraphExec_t exec = nullptr;
  std::vector<int> key_nf, graph_nf;      // arguments of the last call, of the graph
  std::vector<const void*> key_ptr, graph_ptr;
  std::vector<int> tuned_nf;              // function counts of the kept choice and items
  // the persistent blend + interpolation kernel: per-plan records, work items, counter
  cudaEvent_t fork_dft = nullptr;         // after the persistent kernel
  void* work = nullptr;
  size_t work_cap = 0;
  int4* items = nullptr;
  size_t items_cap = 0;
  int* counter = nullptr;
  int n_items = 0;
  // a caller's own capture holds the records' and items' addresses: the next set of function
  // counts takes other buffers, these stay until the group goes
  bool lent = false;
  std::vector<void*> retired;
  int nt = 0;                             // its threads per CTA (tuned)
  int persistent = 0;                     // the kept form (tuned)
  int forced_form = -1, forced_nt = 0;    // fc2d_group_tuning_set (-1: tune)
  // microseconds: queue kernel with 256 and 512 threads, a call with branches only, a
  // call with the queue kernel
  float tune_us[4] = {0.f, 0.f, 0.f, 0.f};
};

using namespace fc2d;

static void drop_graph(fc2d_group_s* g) {
  if (g->exec) cudaGraphExecDestroy(g->exec);
  if (g->graph) cudaGraphDestroy(g->graph);
  g->exec = nullptr;
  g->graph = nullptr;
  g->graph_nf.clear();
  g->graph_ptr.clear();
}

static void group_free(fc2d_group_s* g) {
  if (!g) return;
  drop_graph(g);
  for (cudaEvent_t e : g->join)
    if (e) cudaEventDestroy(e);
  if (g->fork) cudaEventDestroy(g->fork);
  if (g->fork_dft) cudaEventDestroy(g->fork_dft);
  if (g->work) cudaFree(g->work);
  if (g->items) cudaFree(g->items);
  for (void* q : g->retired) cudaFree(q);
  if (g->counter) cudaFree(g->counter);
  for (cudaStream_t s : g->branch)
    if (s) cudaStreamDestroy(s);
  if (g->cap) cudaStreamDestroy(g->cap);
  delete g;
}

extern "C" fc2d_status fc2d_group_create(const fc2d_plan_t* plans, int n, fc2d_group_t* out) {
  if (!plans || n < 1 || !out) return set_error(FC2D_ERR_ARG, "fc2d_group_create: bad argument");
  for (int i = 0; i < n; ++i) {
    if (!plans[i]) return set_error(FC2D_ERR_ARG, "fc2d_group_create: null plan");
    // the branches run concurrently on each plan's own workspace
    for (int j = 0; j < i; ++j)
      if (plans[j] == plans[i])
        return set_error(FC2D_ERR_ARG, "fc2d_group_create: a plan appears twice");
  }
  auto* g = new fc2d_group_s();
  g->plans.assign(plans, plans + n);
  bool ok = cudaStreamCreateWithFlags(&g->cap, cudaStreamNonBlocking) == cudaSuccess &&
            cudaEventCreateWithFlags(&g->fork, cudaEventDisableTiming) == cudaSuccess &&
            cudaEventCreateWithFlags(&g->fork_dft, cudaEventDisableTiming) == cudaSuccess &&
            cudaMalloc(&g->counter, sizeof(int)) == cudaSuccess;
  g->branch.assign(n, nullptr);
  g->join.assign(n, nullptr);
  for (int i = 0; ok && i < n; ++i)
    ok = cudaStreamCreateWithFlags(&g->branch[i], cudaStreamNonBlocking) == cudaSuccess &&
         cudaEventCreateWithFlags(&g->join[i], cudaEventDisableTiming) == cudaSuccess;
  if (!ok) {
    group_free(g);
    return set_error(FC2D_ERR_CUDA, "fc2d_group_create: stream or event creation failed");
  }
  *out = g;
  return FC2D_OK;
}

static fc2d_status grow(void** buf, size_t* cap, size_t bytes) {
  if (bytes <= *cap) return FC2D_OK;
  if (*buf) cudaFree(*buf);
  *buf = nullptr;
  *cap = 0;
  if (cudaMalloc(buf, bytes) != cudaSuccess) {
    *buf = nullptr;
    return set_error(FC2D_ERR_CUDA, "fc2d_group: device allocation failed");
  }
  *cap = bytes;
  return FC2D_OK;
}

// One call's arguments and what follows from them: the mixed-form members' records.
struct Call {
  const int* n_f;
  const double* const* fg;
  const double* const* fb;
  void* const* fhat;
  std::vector<char> fused;
  std::vector<unsigned char> work;
  std::vector<std::vector<int32_t>> points;  // strip points of each range, per record
  int n_fused = 0, max_ldS = 0, n_sm = 1;
  const double* bdry(int i) const { return fb ? fb[i] : nullptr; }
};

static fc2d_status describe(fc2d_group_s* g, Call& c) {
  const int n = (int)g->plans.size();
  const size_t rec = gi_work_bytes();
  c.fused.assign(n, 0);
  for (int i = 0; i < n; ++i) {
    fc2d_plan_s* p = g->plans[i];
    fc2d_status st = extend_coeffs_check(p, c.n_f[i], c.fg[i], c.bdry(i), c.fhat[i]);
    if (st) return st;
    if (!group_fused(p)) continue;
    c.points.emplace_back();
    const GiPlanArgs a = group_fused_args(p, c.n_f[i], c.fg[i], c.bdry(i), &c.points.back());
    c.work.resize((size_t)(c.n_fused + 1) * rec);
    int ld = 0;
    if ((st = gi_work_fill(a, c.work.data() + (size_t)c.n_fused * rec, &ld))) return st;
    c.max_ldS = std::max(c.max_ldS, ld);
    c.n_sm = std::max(c.n_sm, p->n_sm);
    c.fused[i] = 1;
    ++c.n_fused;
  }
  return FC2D_OK;
}

static fc2d_status queue(fc2d_group_s* g, const Call& c, int nt, cudaStream_t s) {
  fc2d_status st = launch_write_work(c.work.data(), c.n_fused, g->work, g->counter, s);
  if (st) return st;
  return launch_gather_interp_queue(g->work, g->items, g->n_items, g->counter, nt, c.max_ldS,
                                    std::min(g->n_items, c.n_sm * (512 / nt)), s);
}

// The whole call in one form on stream s.  Every branch that was forked is joined, also
// after an error.
static fc2d_status launch(fc2d_group_s* g, const Call& c, bool persistent, cudaStream_t s) {
  const int n = (int)g->plans.size();
  fc2d_status st = cuda_check(cudaEventRecord(g->fork, s), "fc2d_group: fork");
  if (!st && persistent) {
    st = queue(g, c, g->nt, s);
    if (!st) st = cuda_check(cudaEventRecord(g->fork_dft, s), "fc2d_group: fork");
  }
  for (int i = 0; i < n && !st; ++i) {
    const bool q = persistent && c.fused[i];
    st = cuda_check(cudaStreamWaitEvent(g->branch[i], q ? g->fork_dft : g->fork, 0), "fc2d_group: fork");
    if (st) break;
    st = q ? extend_coeffs_dft(g->plans[i], c.n_f[i], c.fg[i], c.fhat[i], g->branch[i])
           : fc2d_extend_coeffs(g->plans[i], c.n_f[i], c.fg[i], c.bdry(i), c.fhat[i], g->branch[i]);
    const cudaError_t e0 = cudaEventRecord(g->join[i], g->branch[i]);
    const cudaError_t e1 = cudaStreamWaitEvent(s, g->join[i], 0);
    if (!st && (e0 != cudaSuccess || e1 != cudaSuccess))
      st = set_error(FC2D_ERR_CUDA, "fc2d_group: join failed");
  }
  return st;
}

// Mean microseconds of `reps` runs of `run` on stream s after one warm-up.
template <typename F>
static fc2d_status time_runs(cudaStream_t s, int reps, float* us, F run) {
  cudaEvent_t e0 = nullptr, e1 = nullptr;
  float ms = -1.f;
  fc2d_status st = FC2D_OK;
  if (cudaEventCreate(&e0) == cudaSuccess && cudaEventCreate(&e1) == cudaSuccess) {
    for (int r = 0; r <= reps && !st; ++r) {
      if (r == 1) cudaEventRecord(e0, s);
      st = run();
    }
    cudaEventRecord(e1, s);
    if (cudaEventSynchronize(e1) == cudaSuccess) cudaEventElapsedTime(&ms, e0, e1);
  }
  if (e0) cudaEventDestroy(e0);
  if (e1) cudaEventDestroy(e1);
  *us = ms < 0.f ? 0.f : 1e3f * ms / reps;
  return st || ms >= 0.f ? st : set_error(FC2D_ERR_CUDA, "fc2d_group: tuning launch failed");
}

// For a new set of function counts: the work items of the mixed-form members, longest
// first, and the choice of the form (with mixed-form members the persistent kernel's CTA
// shape, 256 threads two per SM or 512 one per SM, then both forms, timed on the call's
// inputs).
static fc2d_status tune(fc2d_group_s* g, const Call& c) {
  const int n = (int)g->plans.size();
  g->tuned_nf.clear();
  std::vector<int4> items;
  std::vector<int64_t> cost;
  for (int i = 0, k = 0; i < n; ++i) {
    if (!c.fused[i]) continue;
    for (int r = 0; r < (int)c.points[k].size(); ++r)
      for (int f = 0; f < c.n_f[i]; ++f) {
        items.push_back(make_int4(k, r, f, 0));
        cost.push_back(c.points[k][r] + kItemFixed);
      }
    ++k;
  }
  // the previous call may still be reading the old items, and the tuning launches below
  // write the plans' workspaces and outputs: let earlier work finish
  fc2d_status st = cuda_check(cudaDeviceSynchronize(), "fc2d_group: synchronise");
  if (st) return st;
  // the captured graph holds the addresses of the items and records, and the number of items,
  // that are replaced here
  drop_graph(g);
  if (g->lent) {
    for (void* q : {g->work, (void*)g->items})
      if (q) g->retired.push_back(q);
    g->work = nullptr;
    g->items = nullptr;
    g->work_cap = g->items_cap = 0;
    g->lent = false;
  }
  g->n_items = (int)items.size();
  g->nt = 0;
  g->persistent = 0;
  for (float& u : g->tune_us) u = 0.f;
  if (g->n_items) {
    std::vector<int> order(items.size());
    std::iota(order.begin(), order.end(), 0);
    std::stable_sort(order.begin(), order.end(), [&](int x, int y) { return cost[x] > cost[y]; });
    std::vector<int4> sorted(items.size());
    for (size_t k = 0; k < items.size(); ++k) sorted[k] = items[order[k]];
    if ((st = grow(&g->work, &g->work_cap, c.work.size())) ||
        (st = grow(reinterpret_cast<void**>(&g->items), &g->items_cap, sorted.size() * sizeof(int4))))
      return st;
    if (cudaMemcpy(g->items, sorted.data(), sorted.size() * sizeof(int4), cudaMemcpyHostToDevice) !=
        cudaSuccess)
      return set_error(FC2D_ERR_CUDA, "fc2d_group: work upload failed");
    if (g->forced_form >= 0) {
      g->nt = g->forced_nt;
      g->persistent = g->forced_form;
    } else {
      for (int k = 0; k < 2 && !st; ++k)
        st = time_runs(g->cap, 3, &g->tune_us[k], [&] { return queue(g, c, k ? 512 : 256, g->cap); });
      g->nt = g->tune_us[0] <= g->tune_us[1] ? 256 : 512;
      for (int k = 0; k < 2 && !st; ++k)
        st = time_runs(g->cap, 3, &g->tune_us[2 + k], [&] { return launch(g, c, k == 1, g->cap); });
      g->persistent = g->tune_us[3] < g->tune_us[2] ? 1 : 0;
      if (st) return st;
    }
  }
  g->tuned_nf.assign(c.n_f, c.n_f + n);
  return FC2D_OK;
}

// Capture the call into g->graph / g->exec.
static fc2d_status capture(fc2d_group_s* g, const Call& c) {
  // a replay of the previous graph may still be running
  fc2d_status st = cuda_check(cudaDeviceSynchronize(), "fc2d_group: synchronise");
  if (st) return st;
  drop_graph(g);
  if (cudaStreamBeginCapture(g->cap, cudaStreamCaptureModeThreadLocal) != cudaSuccess)
    return set_error(FC2D_ERR_CUDA, "fc2d_group: stream capture failed to start");
  st = launch(g, c, g->persistent != 0, g->cap);
  const cudaError_t e = cudaStreamEndCapture(g->cap, &g->graph);
  if (!st && (e != cudaSuccess || !g->graph))
    st = set_error(FC2D_ERR_CUDA, "fc2d_group: stream capture failed");
  if (!st && cudaGraphInstantiate(&g->exec, g->graph, 0) != cudaSuccess) {
    g->exec = nullptr;
    st = set_error(FC2D_ERR_CUDA, "fc2d_group: graph instantiation failed");
  }
  if (st) drop_graph(g);
  return st;
}

extern "C" fc2d_status fc2d_group_extend_coeffs(fc2d_group_t g, const int* n_f,
                                                const double* const* f_grid_dev,
                                                const double* const* f_bdry_dev,
                                                void* const* fhat_dev, void* stream) {
  if (!g || !n_f || !f_grid_dev || !fhat_dev)
    return set_error(FC2D_ERR_ARG, "fc2d_group_extend_coeffs: null argument");
  const int n = (int)g->plans.size();
  std::vector<int> knf(n_f, n_f + n);
  std::vector<const void*> kptr;
  // inside a caller's capture its graph takes the kernels themselves
  cudaStreamCaptureStatus cs = cudaStreamCaptureStatusNone;
  const bool capturing = cudaStreamIsCapturing((cudaStream_t)stream, &cs) != cudaSuccess ||
                         cs != cudaStreamCaptureStatusNone;
  if (capturing) {
    cudaGetLastError();
    if (knf != g->tuned_nf)
      return set_error(FC2D_ERR_CUDA, "fc2d_group_extend_coeffs: the first call for these function "
                                      "counts cannot be made inside a stream capture");
  }
  for (int i = 0; i < n; ++i) {
    if (n_f[i] < 1 || !f_grid_dev[i] || !fhat_dev[i])
      return set_error(FC2D_ERR_ARG, "fc2d_group_extend_coeffs: bad entry");
    // grow the workspaces now (outside any capture), so that the key below holds the
    // buffers the kernels will use
    fc2d_status st = ensure_plan_workspace(g->plans[i], n_f[i]);
    if (st) return st;
  }
  for (int i = 0; i < n; ++i) {
    kptr.push_back(f_grid_dev[i]);
    kptr.push_back(f_bdry_dev ? f_bdry_dev[i] : nullptr);
    kptr.push_back(fhat_dev[i]);
    kptr.push_back(g->plans[i]->ws.base);
    kptr.push_back(reinterpret_cast<const void*>(g->plans[i]->ws.bytes));
  }
  if (capturing || !g->exec || knf != g->graph_nf || kptr != g->graph_ptr) {
    Call c{n_f, f_grid_dev, f_bdry_dev, fhat_dev};
    fc2d_status st = describe(g, c);
    if (!st && knf != g->tuned_nf) st = tune(g, c);
    if (st) return st;
    const bool again = knf == g->key_nf && kptr == g->key_ptr;
    if (capturing) g->lent = true;
    if (capturing || !again) {
      g->key_nf = knf;
      g->key_ptr = kptr;
      return launch(g, c, g->persistent != 0, (cudaStream_t)stream);
    }
    if ((st = capture(g, c))) return st;
    g->graph_nf = knf;
    g->graph_ptr = kptr;
  }
  g->key_nf = knf;  // a replayed call is the next one's last call too
  g->key_ptr = kptr;
  if (cudaGraphLaunch(g->exec, (cudaStream_t)stream) != cudaSuccess)
    return set_error(FC2D_ERR_CUDA, "fc2d_group: graph launch failed");
  return FC2D_OK;
}

extern "C" fc2d_status fc2d_group_tuning_set(fc2d_group_t g, const int32_t* choice) {
  if (!g) return set_error(FC2D_ERR_ARG, "fc2d_group_tuning_set: null group");
  if (choice && (choice[0] < 0 || choice[0] > 1 || (choice[1] != 256 && choice[1] != 512)))
    return set_error(FC2D_ERR_ARG, "fc2d_group_tuning_set: form 0 or 1, 256 or 512 threads");
  g->forced_form = choice ? choice[0] : -1;
  g->forced_nt = choice ? choice[1] : 0;
  g->tuned_nf.clear();  // the next call tunes anew
  g->key_nf.clear();
  g->graph_nf.clear();
  return FC2D_OK;
}

extern "C" fc2d_status fc2d_group_tuning(fc2d_group_t g, int32_t* choice, float* us) {
  if (!g || !choice || !us) return set_error(FC2D_ERR_ARG, "fc2d_group_tuning: null argument");
  choice[0] = g->persistent;
  choice[1] = g->nt;
  for (int k = 0; k < 4; ++k) us[k] = g->tune_us[k];
  return FC2D_OK;
}

extern "C" void fc2d_group_destroy(fc2d_group_t g) { group_free(g); }
