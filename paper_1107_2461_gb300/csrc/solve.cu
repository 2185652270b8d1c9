// Solve orchestration: the Helmholtz / Laplace inverse on one field of a plan.
//
// TPT (Sec. 3, end): forward transforms along x and y (E_x^{-1}, E_y^{-1}),
// Thomas along z per (x-mode, y-mode) line, back transforms (E_y, E_x).
// TPF (Eq. 29): forward transforms in all three directions, divide by the
// shifted eigenvalue sums (Eq. 26-28), back transforms.
//
// Both are exact inverses of the assembled operator up to rounding; the
// residual r = b - A u is evaluated with the finite-volume stencil and, while
// ||r||/||b|| exceeds the tolerance, a correction A d = r is solved by the same
// direct method and added (iterative refinement).  Every refinement kernel
// reads a device "done" flag and returns at once when the previous check has
// converged, so the whole solve is enqueued without a host round trip.
#include <algorithm>
#include <cmath>
#include <map>
#include <mutex>
#include <tuple>
#include <vector>

#include "fdi_internal.h"
#include "resident.h"
#include "slice_transform.h"

namespace fdi {

#define FDI_TRY(expr)            \
  do {                           \
    fdi_status _s = (expr);      \
    if (_s != FDI_OK) return _s; \
  } while (0)

fdi_status validate_field_args(const fdi_plan* p, int field, double sigma, double lambda) {
  if (!p) return FDI_ERR_INVALID_ARG;
  if (field < 0 || field >= p->nfields) {
    set_error("field not present in this plan");
    return FDI_ERR_INVALID_ARG;
  }
  if (!std::isfinite(sigma) || !std::isfinite(lambda) || sigma < 0.0 || lambda < 0.0) {
    set_error("sigma and lambda must be finite and >= 0");
    return FDI_ERR_INVALID_ARG;
  }
  if (sigma == 0.0 && lambda == 0.0) {
    set_error("sigma = lambda = 0 is the zero operator");
    return FDI_ERR_INVALID_ARG;
  }
  if (sigma == 0.0 && field != FDI_FIELD_CELL) {
    set_error("the Laplace problem (sigma = 0) is defined on the cell field only");
    return FDI_ERR_INVALID_ARG;
  }
  if (sigma == 0.0 && p->cyl && p->fields[0].zero_flux_all) {
    set_error("the zero-flux Laplacian of a cylindrical plan is singular; not handled");
    return FDI_ERR_UNSUPPORTED;
  }
  return FDI_OK;
}

cudaGraph_t capturing_graph(cudaStream_t s) {
  cudaStreamCaptureStatus cap = cudaStreamCaptureStatusNone;
  cudaGraph_t g = nullptr;
  if (cudaStreamGetCaptureInfo(s, &cap, nullptr, &g, nullptr, nullptr, nullptr) != cudaSuccess) {
    cudaGetLastError();  // the legacy stream beside another stream's capture
    return nullptr;
  }
  return cap == cudaStreamCaptureStatusActive ? g : nullptr;
}

fdi_status graph_add_if(cudaStream_t s, cudaGraph_t g, cudaGraphConditionalHandle h, cudaGraph_t* body) {
  const cudaGraphNode_t* deps = nullptr;
  size_t ndeps = 0;
  cudaStreamCaptureStatus cs = cudaStreamCaptureStatusNone;
  cudaGraph_t gg = nullptr;
  FDI_CUDA_TRY(cudaStreamGetCaptureInfo(s, &cs, nullptr, &gg, &deps, nullptr, &ndeps));
  cudaGraphNodeParams cp = {};
  cp.type = cudaGraphNodeTypeConditional;
  cp.conditional.handle = h;
  cp.conditional.type = cudaGraphCondTypeIf;
  cp.conditional.size = 1;
  cudaGraphNode_t node = nullptr;
  FDI_CUDA_TRY(cudaGraphAddNode(&node, g, deps, nullptr, ndeps, &cp));
  FDI_CUDA_TRY(cudaStreamUpdateCaptureDependencies(s, &node, nullptr, 1, cudaStreamSetCaptureDependencies));
  *body = cp.conditional.phGraph_out[0];
  return FDI_OK;
}

namespace {

// One direct solve in FP64: out (+)= A^{-1} in.
fdi_status solve_once_f64(fdi_plan* p, int field, double sigma, double lambda, const double* in, double* out,
                          bool accumulate, const int* skip, cudaStream_t s) {
  const Field& f = p->fields[field];
  const int nx = f.n[0], ny = f.n[1], nz = f.n[2];
  double* t0 = p->ws[0];
  double* t1 = p->ws[1];
  double* t2 = p->ws[2];
  const bool small = small_plane_f64(f);
  auto fwd = [&](int d, const double* src, double* dst) {
    return launch_axis_f64(p, f, d, true, src, dst, false, d > 0, skip, s);
  };
  auto back = [&](int d, const double* src, double* dst, bool acc) {
    return launch_axis_f64(p, f, d, false, src, dst, acc, true, skip, s);
  };
  // in -> t1 in the x and y eigenbases
  if (small) {
    FDI_TRY(launch_small_plane(p, f, true, in, t1, false, false, skip, s));
  } else {
    FDI_TRY(fwd(0, in, t0));
    FDI_TRY(fwd(1, t0, t1));
  }
  // t1 -> z
  double* z = t0;
  if (p->thomas_axis == 2) {
    FDI_TRY(launch_thomas_f64(p, f, sigma, lambda, field, t1, t0, t2, skip, s));
  } else if (p->cyl) {
    // cylindrical TPF (Eq. 45-46): the radial transform of theta mode j uses
    // that mode's own eigenbasis, the divide its own eigenvalues
    FDI_TRY(launch_modes_f64(p, t1, t0, p->cyl_Eri, nz, nx, ny, skip, s));
    FDI_TRY(launch_divide_modes_f64(p, f, sigma, lambda, t0, skip, s));
    FDI_TRY(launch_modes_f64(p, t0, t1, p->cyl_Er, nz, nx, ny, skip, s));
    z = t1;
  } else if (small_z_f64(f)) {
    FDI_TRY(launch_small_z(p, f, sigma, lambda, t1, skip, s));
    z = t1;
  } else {
    FDI_TRY(fwd(2, t1, t0));
    FDI_TRY(launch_divide_f64(p, f, sigma, lambda, t0, skip, s));
    FDI_TRY(back(2, t0, t1, false));
    z = t1;
  }
  // z -> out
  if (small) return launch_small_plane(p, f, false, z, out, accumulate, true, skip, s);
  double* y = z == t0 ? t1 : t0;
  FDI_TRY(back(1, z, y, false));
  FDI_TRY(back(0, y, out, accumulate));
  return FDI_OK;
}

}  // namespace

namespace {

fdi_status field_solve_internal(fdi_plan* p, int field, double sigma, double lambda, const double* rhs, double* out,
                                cudaStream_t s) {
  if (p->prec != FDI_PREC_FP64) return mixed_field_solve(p, field, sigma, lambda, rhs, out, s);
  const Field& f = p->fields[field];
  const double* b = rhs;
  if (out == rhs) {
    FDI_CUDA_TRY(cudaMemcpyAsync(p->ws[4], rhs, f.P * sizeof(double), cudaMemcpyDeviceToDevice, s));
    b = p->ws[4];
  }
  const bool singular = sigma == 0.0 && f.zero_flux_all;
  if (singular) FDI_TRY(launch_mean_f64(p, f, b, s));
  double* r = p->ws[3];
  // round 0 solves for b, later ones add the correction for r; every round ends
  // with the residual and its check (which also sets the next round's graph
  // condition)
  auto enqueue_round = [&](int round, cudaStream_t st, cudaGraphConditionalHandle next_round) -> fdi_status {
    const int* skip = round == 0 ? nullptr : &p->d_status->done;
    FDI_TRY(solve_once_f64(p, field, sigma, lambda, round == 0 ? b : r, out, round > 0, skip, st));
    return launch_residual_f64(p, f, sigma, lambda, b, out, r, singular, round == 0, next_round, skip, st);
  };
  // Eagerly every round is enqueued and returns at once after convergence.  In
  // a captured solve each correction round sits in a conditional node nested in
  // the one before it, so a converged solve launches nothing more (a 16^3 solve
  // went from 80 to 58 us with its residual's reduction folded in, 64^3 from 127
  // to 105 us).
  // Only in the graphs that field_solve_entry and batch_solve keep.  In a caller's
  // own capture the rounds stay ordinary launches (a graph with conditional nodes
  // cannot be used everywhere a plain one can), and in the Krylov loop's WHILE
  // body too: there, with the solves joined from side streams right after their
  // conditional nodes, a replay never finished (the GPU idle, the host waiting).
  cudaGraph_t g = (p->max_refine >= 1 && p->own_capture) ? capturing_graph(s) : nullptr;
  if (!g) {
    for (int round = 0; round <= p->max_refine; ++round) FDI_TRY(enqueue_round(round, s, 0));
    return FDI_OK;
  }
  cudaGraphConditionalHandle h = 0;
  FDI_CUDA_TRY(cudaGraphConditionalHandleCreate(&h, g, 0, cudaGraphCondAssignDefault));
  FDI_TRY(enqueue_round(0, s, h));
  // ordinary launches inside the conditional bodies
  struct NoPdl {
    fdi_plan* p;
    bool was;
    explicit NoPdl(fdi_plan* q) : p(q), was(q->pdl) { p->pdl = false; }
    ~NoPdl() { p->pdl = was; }
  } no_pdl(p);
  cudaGraph_t body = nullptr;
  FDI_TRY(graph_add_if(s, g, h, &body));
  for (int round = 1; round <= p->max_refine; ++round) {
    cudaGraphConditionalHandle hn = 0;
    if (round < p->max_refine)
      FDI_CUDA_TRY(cudaGraphConditionalHandleCreate(&hn, body, 0, cudaGraphCondAssignDefault));
    FDI_CUDA_TRY(cudaStreamBeginCaptureToGraph(p->cstream, body, nullptr, nullptr, 0, cudaStreamCaptureModeRelaxed));
    fdi_status st = enqueue_round(round, p->cstream, hn);
    cudaGraph_t next_body = nullptr;
    if (st == FDI_OK && hn) st = graph_add_if(p->cstream, body, hn, &next_body);
    cudaGraph_t done_graph = nullptr;
    const cudaError_t e = cudaStreamEndCapture(p->cstream, &done_graph);
    FDI_TRY(st);
    FDI_CUDA_TRY(e);
    body = next_body;
  }
  return FDI_OK;
}

}  // namespace

fdi_status field_solve(fdi_plan* p, int field, double sigma, double lambda, const double* rhs, double* out,
                       cudaStream_t s) {
  FDI_TRY(validate_field_args(p, field, sigma, lambda));
  if (!rhs || !out) return FDI_ERR_INVALID_ARG;
  if (p->tstage[0] == nullptr) return field_solve_internal(p, field, sigma, lambda, rhs, out, s);
  // Thomas along x or y: solve on the copy with that axis outermost
  FDI_TRY(launch_axis_permute(p, rhs, p->tstage[0], true, s));
  FDI_TRY(field_solve_internal(p, field, sigma, lambda, p->tstage[0], p->tstage[1], s));
  return launch_axis_permute(p, p->tstage[1], out, false, s);
}

// Autotuned Thomas configurations per (grid shape, precision),
// applied to plans created later with the same shape.
namespace {
struct TuneKey {
  int n0, n1, n2, prec, grid;
  bool operator<(const TuneKey& o) const {
    return std::tie(n0, n1, n2, prec, grid) < std::tie(o.n0, o.n1, o.n2, o.prec, o.grid);
  }
};
std::mutex g_tune_mu;
std::map<TuneKey, int> g_tune;
TuneKey tune_key(const fdi_plan* p) { return TuneKey{p->n[0], p->n[1], p->n[2], (int)p->prec, (int)p->grid}; }
}  // namespace

void forget_batch_graph(const fdi_plan* p);

void remember_tuning(const fdi_plan* p) {
  std::lock_guard<std::mutex> lk(g_tune_mu);
  g_tune[tune_key(p)] = p->thomas_tl;
}

void apply_tuning(fdi_plan* p) {
  std::lock_guard<std::mutex> lk(g_tune_mu);
  auto it = g_tune.find(tune_key(p));
  if (it != g_tune.end()) p->thomas_tl = it->second;
}

void invalidate_graph(fdi_plan* p) {
  for (fdi_plan::GraphSlot& g : p->gslots) {
    if (g.exec) cudaGraphExecDestroy(g.exec);
    g = fdi_plan::GraphSlot{};
  }
  if (p->kgraph) cudaGraphExecDestroy(p->kgraph);
  p->kgraph = nullptr;
  p->kgraph_precond = -1;
  forget_batch_graph(p);
}

namespace {

// The stream a call on s is captured on: s itself, or for the default streams
// (which cannot be captured; a graph can be launched on them) one of the plan's.
// A 75 x 50 x 67 mixed solve on the default stream takes 176 us launch by launch
// and 139 us as a graph.
cudaStream_t capture_stream(fdi_plan* p, cudaStream_t s) {
  if (s != nullptr && s != cudaStreamLegacy && s != cudaStreamPerThread) return s;
  if (!p->gstream && cudaStreamCreateWithFlags(&p->gstream, cudaStreamNonBlocking) != cudaSuccess) {
    cudaGetLastError();
    p->gstream = nullptr;
  }
  return p->gstream;
}

// marks plans whose launches go into one of the library's own graphs
struct OwnCapture {
  fdi_plan* const* plans;
  int count;
  OwnCapture(fdi_plan* const* q, int n) : plans(q), count(n) { set(true); }
  ~OwnCapture() { set(false); }
  void set(bool on) {
    for (int i = 0; i < count; ++i) plans[i]->own_capture = on;
  }
};

// While the library builds one of its graphs: another thread's capture (in the
// global mode that PyTorch takes by default) forbids the stream creation and the
// instantiation meant here and would be invalidated by them.  Nothing done in
// this scope touches a stream of that capture.
struct BesideCaptures {
  cudaStreamCaptureMode mode = cudaStreamCaptureModeRelaxed;
  BesideCaptures() { cudaThreadExchangeStreamCaptureMode(&mode); }
  ~BesideCaptures() { cudaThreadExchangeStreamCaptureMode(&mode); }
};

bool same_key(const fdi_plan::GraphKey& a, const fdi_plan::GraphKey& b) {
  return a.field == b.field && a.sigma == b.sigma && a.lambda == b.lambda && a.rhs == b.rhs && a.out == b.out &&
         a.s == b.s;
}

}  // namespace

// Field solve through the graph cache: the first call with new arguments runs
// eagerly, the second identical call is captured (stream capture of the same
// launch sequence) and every later identical call is one graph launch.  The
// cache keeps the graphs of the last few distinct argument sets.  Timed plans
// need their events, so they run eagerly.  A call on a stream that its caller is
// capturing neither reads nor fills the cache: the launches themselves go into
// the caller's graph (a kept graph would become a child of it, where conditional
// nodes are not allowed, and no capture can begin inside another).
fdi_status field_solve_entry(fdi_plan* p, int field, double sigma, double lambda, const double* rhs, double* out,
                             cudaStream_t s) {
  if (!p) return FDI_ERR_INVALID_ARG;
  p->launches = 0;
  p->kloop_body_launches = 0;
  if (!p->use_graphs || p->timing || capturing_graph(s)) return field_solve(p, field, sigma, lambda, rhs, out, s);
  fdi_plan::GraphKey key;
  key.field = field;
  key.sigma = sigma;
  key.lambda = lambda;
  key.rhs = rhs;
  key.out = out;
  key.s = s;
  fdi_plan::GraphSlot* g = nullptr;
  for (fdi_plan::GraphSlot& c : p->gslots)
    if (c.valid && same_key(key, c.key)) g = &c;
  if (g && g->exec) {
    g->last_use = ++p->gclock;
    FDI_CUDA_TRY(cudaGraphLaunch(g->exec, s));
    p->launches = g->launches;
    return FDI_OK;
  }
  if (!g) {
    // first call with these arguments: eager; remember the key in a free or
    // the least recently used slot
    g = &p->gslots[0];
    for (fdi_plan::GraphSlot& c : p->gslots) {
      if (!c.valid) {
        g = &c;
        break;
      }
      if (c.last_use < g->last_use) g = &c;
    }
    if (g->exec) cudaGraphExecDestroy(g->exec);
    *g = fdi_plan::GraphSlot{};
    fdi_status st = field_solve(p, field, sigma, lambda, rhs, out, s);
    if (st == FDI_OK) {
      g->key = key;
      g->valid = true;
      g->last_use = ++p->gclock;
    }
    return st;
  }
  // second call with these arguments: capture, instantiate, launch
  g->last_use = ++p->gclock;
  const BesideCaptures beside;
  const cudaStream_t cs = capture_stream(p, s);
  if (!cs) return field_solve(p, field, sigma, lambda, rhs, out, s);
  FDI_CUDA_TRY(cudaStreamBeginCapture(cs, cudaStreamCaptureModeThreadLocal));
  fdi_status st;
  {
    OwnCapture own(&p, 1);
    st = field_solve(p, field, sigma, lambda, rhs, out, cs);
  }
  cudaGraph_t gr = nullptr;
  cudaError_t e = cudaStreamEndCapture(cs, &gr);
  if (st != FDI_OK || e != cudaSuccess || gr == nullptr) {
    if (gr) cudaGraphDestroy(gr);
    cudaGetLastError();
    *g = fdi_plan::GraphSlot{};
    if (st != FDI_OK) return st;
    return field_solve(p, field, sigma, lambda, rhs, out, s);  // capture refused: eager
  }
  const long long n_launch = p->launches;
  cudaGraphExec_t ex = nullptr;
  e = cudaGraphInstantiate(&ex, gr, 0);
  cudaGraphDestroy(gr);
  if (e != cudaSuccess) {
    cudaGetLastError();
    *g = fdi_plan::GraphSlot{};
    return field_solve(p, field, sigma, lambda, rhs, out, s);
  }
  g->exec = ex;
  g->launches = n_launch;
  FDI_CUDA_TRY(cudaGraphLaunch(g->exec, s));
  p->launches = n_launch;
  return FDI_OK;
}

namespace {

// ---- batched solves: independent plans run concurrently on a pool of streams ----

constexpr int kBatchStreams = 32;

struct StreamPool {
  cudaStream_t st[kBatchStreams] = {};
  cudaEvent_t done[kBatchStreams] = {};
  cudaEvent_t fork = nullptr;
  bool ok = false;
};

std::mutex g_pool_mu;
std::map<int, StreamPool> g_pools;

StreamPool* stream_pool() {
  int dev = 0;
  if (cudaGetDevice(&dev) != cudaSuccess) return nullptr;
  std::lock_guard<std::mutex> lk(g_pool_mu);
  StreamPool& sp = g_pools[dev];
  if (!sp.ok) {
    for (int k = 0; k < kBatchStreams; ++k) {
      if (cudaStreamCreateWithFlags(&sp.st[k], cudaStreamNonBlocking) != cudaSuccess) return nullptr;
      if (cudaEventCreateWithFlags(&sp.done[k], cudaEventDisableTiming) != cudaSuccess) return nullptr;
    }
    if (cudaEventCreateWithFlags(&sp.fork, cudaEventDisableTiming) != cudaSuccess) return nullptr;
    sp.ok = true;
  }
  return &sp;
}

// Fork from s onto the pool, one stream per distinct plan (a plan appearing
// twice keeps one stream, so its workspace is used in order), join back on s.
fdi_status enqueue_batch(StreamPool* sp, fdi_plan* const* plans, const double* lambdas, const double* const* rhs,
                         double* const* out, int count, cudaStream_t s) {
  FDI_CUDA_TRY(cudaEventRecord(sp->fork, s));
  std::vector<int> lane(count, -1);
  bool used[kBatchStreams] = {false};
  // small grids: resident launches of up to kResMaxJobs solves on pool stream
  // 0 (a plan repeated in the batch goes to a later launch, in order); the
  // other plans one stream each on streams 1...
  std::vector<char> res(count, 0);
  for (int i = 0; i < count; ++i)
    res[i] = (plans[i]->tstage[0] == nullptr && resident_eligible(plans[i], FDI_FIELD_CELL) &&
              validate_field_args(plans[i], FDI_FIELD_CELL, 1.0, lambdas[i]) == FDI_OK) ? 1 : 0;
  {
    std::vector<char> taken(count, 0);
    for (;;) {
      std::vector<ResJob> jobs;
      std::vector<fdi_plan*> in_launch;
      for (int i = 0; i < count && (int)jobs.size() < kResMaxJobs; ++i) {
        if (!res[i] || taken[i]) continue;
        bool dup = false;
        for (fdi_plan* q : in_launch) dup = dup || q == plans[i];
        for (int j = 0; j < i && !dup; ++j) dup = res[j] && !taken[j] && plans[j] == plans[i];
        if (dup) continue;
        ResJob job;
        FDI_TRY(resident_describe(plans[i], FDI_FIELD_CELL, 1.0, lambdas[i], rhs[i], out[i], &job));
        jobs.push_back(job);
        in_launch.push_back(plans[i]);
        taken[i] = 1;
        plans[i]->launches = 0;
      }
      if (jobs.empty()) break;
      if (!used[0]) {
        FDI_CUDA_TRY(cudaStreamWaitEvent(sp->st[0], sp->fork, 0));
        used[0] = true;
      }
      FDI_TRY(resident_launch(in_launch[0], jobs.data(), (int)jobs.size(), sp->st[0]));
    }
  }
  int next = 0;
  for (int i = 0; i < count; ++i) {
    if (res[i]) continue;
    for (int j = 0; j < i; ++j)
      if (plans[j] == plans[i]) {
        lane[i] = lane[j];
        break;
      }
    if (lane[i] < 0) lane[i] = 1 + (next++) % (kBatchStreams - 1);
    const int k = lane[i];
    if (!used[k]) {
      FDI_CUDA_TRY(cudaStreamWaitEvent(sp->st[k], sp->fork, 0));
      used[k] = true;
    }
    plans[i]->launches = 0;
    FDI_TRY(field_solve(plans[i], FDI_FIELD_CELL, 1.0, lambdas[i], rhs[i], out[i], sp->st[k]));
  }
  for (int k = 0; k < kBatchStreams; ++k)
    if (used[k]) {
      FDI_CUDA_TRY(cudaEventRecord(sp->done[k], sp->st[k]));
      FDI_CUDA_TRY(cudaStreamWaitEvent(s, sp->done[k], 0));
    }
  return FDI_OK;
}

// Graph of a whole batch: captured on the second call with identical
// arguments, then replayed as one launch.  The last few distinct batches keep
// theirs (least recently used replaced): a program that alternates between a
// few batches otherwise enqueues thousands of launches each time (64 solves: 4.2
// ms, bound by the host, against 3.5 ms as a graph).
constexpr int kBatchGraphs = 4;
struct BatchGraph {
  std::vector<fdi_plan*> plans;
  std::vector<double> lambdas;
  std::vector<const double*> rhs;
  std::vector<double*> out;
  cudaStream_t s = nullptr;
  cudaGraphExec_t exec = nullptr;
  std::vector<long long> launches;
  unsigned long long last_use = 0;  // 0: empty slot
};

std::mutex g_batch_mu;
BatchGraph g_batches[kBatchGraphs];
unsigned long long g_batch_clock = 0;

void drop_batch(BatchGraph& g) {
  if (g.exec) cudaGraphExecDestroy(g.exec);
  g = BatchGraph();
}

bool same_batch(const BatchGraph& g, fdi_plan* const* plans, const double* lambdas, const double* const* rhs,
                double* const* out, int count, cudaStream_t s) {
  if ((int)g.plans.size() != count || g.s != s) return false;
  for (int i = 0; i < count; ++i)
    if (g.plans[i] != plans[i] || g.lambdas[i] != lambdas[i] || g.rhs[i] != rhs[i] || g.out[i] != out[i]) return false;
  return true;
}

}  // namespace

// drop the batch graph if it involves this plan (plan destroyed or changed)
void forget_batch_graph(const fdi_plan* p) {
  std::lock_guard<std::mutex> lk(g_batch_mu);
  for (BatchGraph& g : g_batches)
    if (std::find(g.plans.begin(), g.plans.end(), p) != g.plans.end()) drop_batch(g);
}

fdi_status batch_solve(fdi_plan* const* plans, const double* lambdas, const double* const* rhs, double* const* out,
                       int count, cudaStream_t s) {
  StreamPool* sp = stream_pool();
  if (!sp) {
    set_error("could not create the batch stream pool");
    return FDI_ERR_CUDA;
  }
  bool graphs = capturing_graph(s) == nullptr;  // a caller's capture gets the launches (field_solve_entry)
  for (int i = 0; i < count; ++i) graphs = graphs && plans[i]->use_graphs && !plans[i]->timing;
  std::lock_guard<std::mutex> lk(g_batch_mu);
  if (!graphs) return enqueue_batch(sp, plans, lambdas, rhs, out, count, s);
  BatchGraph* g = nullptr;
  for (BatchGraph& c : g_batches)
    if (c.last_use && same_batch(c, plans, lambdas, rhs, out, count, s)) g = &c;
  if (g) {
    g->last_use = ++g_batch_clock;
    if (!g->exec) {
      // second identical call: capture the fork / solves / join
      const BesideCaptures beside;
      const cudaStream_t cs = capture_stream(plans[0], s);
      if (!cs) return enqueue_batch(sp, plans, lambdas, rhs, out, count, s);
      FDI_CUDA_TRY(cudaStreamBeginCapture(cs, cudaStreamCaptureModeThreadLocal));
      fdi_status st;
      {
        OwnCapture own(plans, count);
        st = enqueue_batch(sp, plans, lambdas, rhs, out, count, cs);
      }
      cudaGraph_t gr = nullptr;
      cudaError_t e = cudaStreamEndCapture(cs, &gr);
      cudaGraphExec_t ex = nullptr;
      if (st == FDI_OK && e == cudaSuccess && gr) e = cudaGraphInstantiate(&ex, gr, 0);
      if (gr) cudaGraphDestroy(gr);
      if (st != FDI_OK || e != cudaSuccess || !ex) {
        cudaGetLastError();
        drop_batch(*g);
        if (st != FDI_OK) return st;
        return enqueue_batch(sp, plans, lambdas, rhs, out, count, s);
      }
      g->exec = ex;
      g->launches.assign(count, 0);
      for (int i = 0; i < count; ++i) g->launches[i] = plans[i]->launches;
    }
    FDI_CUDA_TRY(cudaGraphLaunch(g->exec, s));
    for (int i = 0; i < count; ++i) plans[i]->launches = g->launches[i];
    return FDI_OK;
  }
  // new arguments: run eagerly and remember them in the least recently used slot
  fdi_status st = enqueue_batch(sp, plans, lambdas, rhs, out, count, s);
  if (st != FDI_OK) return st;
  g = &g_batches[0];
  for (BatchGraph& c : g_batches)
    if (c.last_use < g->last_use) g = &c;
  drop_batch(*g);
  g->plans.assign(plans, plans + count);
  g->lambdas.assign(lambdas, lambdas + count);
  g->rhs.assign(rhs, rhs + count);
  g->out.assign(out, out + count);
  g->s = s;
  g->last_use = ++g_batch_clock;
  return FDI_OK;
}

}  // namespace fdi

using namespace fdi;

extern "C" {

fdi_status fdi_field_solve(fdi_plan* plan, fdi_field field, double sigma, double lambda, const double* rhs,
                           double* out, fdi_stream_t stream) {
  fdi_status st = validate_field_args(plan, (int)field, sigma, lambda);
  if (st != FDI_OK) return st;
  return field_solve_entry(plan, (int)field, sigma, lambda, rhs, out, (cudaStream_t)stream);
}

fdi_status fdi_helmholtz_solve(fdi_plan* plan, double lambda, const double* rhs, double* out,
                               fdi_stream_t stream) {
  fdi_status st = validate_field_args(plan, FDI_FIELD_CELL, 1.0, lambda);
  if (st != FDI_OK) return st;
  return field_solve_entry(plan, FDI_FIELD_CELL, 1.0, lambda, rhs, out, (cudaStream_t)stream);
}

fdi_status fdi_laplace_solve(fdi_plan* plan, const double* rhs, double* out, fdi_stream_t stream) {
  fdi_status st = validate_field_args(plan, FDI_FIELD_CELL, 0.0, 1.0);
  if (st != FDI_OK) return st;
  return field_solve_entry(plan, FDI_FIELD_CELL, 0.0, 1.0, rhs, out, (cudaStream_t)stream);
}

fdi_status fdi_helmholtz_solve_batched(fdi_plan* const* plans, const double* lambdas, const double* const* rhs,
                                       double* const* out, int count, fdi_stream_t stream) {
  if (count < 0 || (count > 0 && (!plans || !lambdas || !rhs || !out))) return FDI_ERR_INVALID_ARG;
  for (int i = 0; i < count; ++i) {
    fdi_status st = validate_field_args(plans[i], FDI_FIELD_CELL, 1.0, lambdas[i]);
    if (st != FDI_OK) return st;
    if (!rhs[i] || !out[i]) return FDI_ERR_INVALID_ARG;
  }
  if (count == 0) return FDI_OK;
  return batch_solve(plans, lambdas, rhs, out, count, (cudaStream_t)stream);
}

fdi_status fdi_plan_set_thomas_config(fdi_plan* plan, int lines_per_cta) {
  if (!plan || (lines_per_cta != 2 && lines_per_cta != 3 && lines_per_cta != 4 && lines_per_cta != 64 &&
                lines_per_cta != 128))
    return FDI_ERR_INVALID_ARG;
  if (lines_per_cta == 4 && plan->prec != FDI_PREC_FP64) {
    // FP64 recurrence with cached line factors: a cache in every workspace
    long long q = 0;
    for (int fi = 0; fi < plan->nfields; ++fi) q = std::max(q, plan->fields[fi].P);
    FDI_TRY(alloc_thomas_cache(plan, q));
    for (int c = 0; c < plan->nextra; ++c) {
      SlotSwap guard(plan, &plan->extra[c]);
      FDI_TRY(alloc_thomas_cache(plan, q));
    }
  }
  plan->thomas_tl = lines_per_cta;
  invalidate_graph(plan);
  return FDI_OK;
}

fdi_status fdi_plan_autotune(fdi_plan* plan, double lambda, const double* rhs, double* out, int reps,
                             int* thomas_tl_out, fdi_stream_t stream) {
  fdi_status st = validate_field_args(plan, FDI_FIELD_CELL, 1.0, lambda);
  if (st != FDI_OK) return st;
  if (!rhs || !out || rhs == out || reps < 1 || reps > 1000) return FDI_ERR_INVALID_ARG;
  cudaStream_t s = (cudaStream_t)stream;
  if (plan->prec != FDI_PREC_FP64) {
    const int tls[4] = {2, 3, 64, 128};
    cudaEvent_t e0 = nullptr, e1 = nullptr;
    FDI_CUDA_TRY(cudaEventCreate(&e0));
    FDI_CUDA_TRY(cudaEventCreate(&e1));
    float best = 0.f;
    int best_t = plan->thomas_tl;
    const bool timing = plan->timing;
    plan->timing = false;
    {
      for (int ti = 0; ti < 4 && st == FDI_OK; ++ti) {
        plan->thomas_tl = tls[ti];
        st = field_solve(plan, FDI_FIELD_CELL, 1.0, lambda, rhs, out, s);  // warm-up
        if (st != FDI_OK) break;
        cudaEventRecord(e0, s);
        for (int r = 0; r < reps && st == FDI_OK; ++r) st = field_solve(plan, FDI_FIELD_CELL, 1.0, lambda, rhs, out, s);
        cudaEventRecord(e1, s);
        if (cudaEventSynchronize(e1) != cudaSuccess) {
          set_error("autotune: timing event failed");
          st = FDI_ERR_CUDA;
          break;
        }
        float ms = 0.f;
        cudaEventElapsedTime(&ms, e0, e1);
        if (best == 0.f || ms < best) {
          best = ms;
          best_t = tls[ti];
        }
      }
    }
    plan->timing = timing;
    cudaEventDestroy(e0);
    cudaEventDestroy(e1);
    plan->thomas_tl = best_t;
    invalidate_graph(plan);
    if (st != FDI_OK) return st;
    remember_tuning(plan);
  }
  if (thomas_tl_out) *thomas_tl_out = plan->thomas_tl;
  return FDI_OK;
}

fdi_status fdi_plan_set_graphs(fdi_plan* plan, int on) {
  if (!plan) return FDI_ERR_INVALID_ARG;
  plan->use_graphs = on != 0;
  invalidate_graph(plan);
  return FDI_OK;
}

}  // extern "C"
