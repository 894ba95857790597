// C-ABI of gradsolve-gb300 (declared in include/gs.h): argument checking, the
// device-resident record, the reusable workspace of gs_solve_grad, and the
// kernel launches. No exception or abort crosses this boundary.
#include <algorithm>
#include <cmath>
#include <cstdio>
#include <cstring>
#include <mutex>
#include <new>
#include <chrono>
#include <thread>
#include <vector>

#include "../../include/gs.h"
#include "gs_internal.h"

using namespace gs;

namespace {

struct ProblemInfo {
  int d, P, stiff, n_shared;
};

bool problem_info(int pid, ProblemInfo* out) {
  switch (pid) {
    case GS_LORENZ: *out = {3, 3, 0, 0}; return true;
    case GS_VDP: *out = {2, 1, 0, 0}; return true;
    case GS_ROBERTSON: *out = {3, 3, 1, 0}; return true;
    case GS_HIRES: *out = {8, 12, 1, 0}; return true;
    case GS_LINEAR: *out = {2, 4, 0, 0}; return true;
    case GS_LV_UDE: *out = {2, 2, 0, 354}; return true;
    case GS_NEURAL_ROBERTSON: *out = {3, 2, 1, 353}; return true;
  }
  return false;
}


// Expected accepted steps per trajectory at rtol 1e-6, used for the first arena
// size and the choice of the record layout; an underestimate costs one rerun.
int step_guess(int pid) {
  switch (pid) {
    case GS_LORENZ: return 48;
    case GS_VDP: return 100;
    case GS_LV_UDE: return 40;
    case GS_ROBERTSON: return 110;
    case GS_HIRES: return 210;
  }
  return 256;
}
// The same for a tolerance rtol and a method: a method of error order q takes
// ~rtol^(-1/(q+1)) steps (q = 4 for Tsit5 and Rodas5P, 6 for Verner7, 2 for
// Rosenbrock23), Verner7 about 0.65 and Rosenbrock23 about 6 times the steps of
// Tsit5 / Rodas5P at rtol 1e-6.
int step_guess(int pid, double rtol, int method) {
  double base = step_guess(pid), expo = 0.2;
  if (method == GS_METHOD_VERNER7) {
    base *= 0.65;
    expo = 1.0 / 7.0;
  } else if (method == GS_METHOD_ROSENBROCK23) {
    base *= 6.0;
    expo = 1.0 / 3.0;
  }
  const double scale = std::pow(1e-6 / (rtol > 0.0 ? rtol : 1e-6), expo);
  const double g = base * (scale < 1.0 ? 1.0 : scale);
  return (int)std::ceil(g);
}

// Stored-stage records (k = 1): the doubles a step and a side step store (the
// kernels' StageData payloads), and the segment [prev, t, y[d], h, step payload]
// rounded up to a 16-byte multiple. Tsit5: Y_1..Y_5 (a side step also Y_6);
// Verner7: Y_1..Y_8 (a side step also its save state); Rodas5P: U_0..U_7, the
// LU factors, pivot reciprocals and pivots (the stage inputs and the save state
// are rebuilt from them); Rosenbrock23: k1, u2 and the LU of W (Y1 and the save
// state rebuilt).
int stage_step_payload(int method, int d, int pid) {
  if (pid == GS_NEURAL_ROBERTSON) return NRG_STAGE_DOUBLES;  // with the network's activations
  switch (method) {
    case GS_METHOD_RODAS5P: return 10 * d + d * d;
    case GS_METHOD_ROSENBROCK23: return 4 * d + d * d;
    case GS_METHOD_VERNER7: return 8 * d;
  }
  return 5 * d;  // Tsit5
}
int stage_side_payload(int method, int d, int pid) {
  const bool rebuilt = method == GS_METHOD_RODAS5P || method == GS_METHOD_ROSENBROCK23;  // save state rebuilt
  return stage_step_payload(method, d, pid) + (rebuilt ? 0 : d);
}
int stage_segw_of(int method, int d, int pid) { return ((3 + d + stage_step_payload(method, d, pid)) + 1) & ~1; }

// Counters that the kernels update; one small device block per record.
struct Counters {
  unsigned long long work_fwd;
  unsigned long long work_rev;
  unsigned long long work_jvp;
  unsigned long long arena_top;
  int overflow;
  int any_failed;
  int tc_error;  // a tensor-core product's completion wait ran out in the reverse sweep
};

}  // namespace

// What decides the sizes of a record's buffers (besides the device).
struct RecordKey {
  int problem, method, precision, k, stages, n_save;
  int64_t n;
  double rtol;
  bool operator==(const RecordKey& o) const {
    return problem == o.problem && method == o.method && precision == o.precision && k == o.k && stages == o.stages &&
           n_save == o.n_save && n == o.n && rtol == o.rtol;
  }
};

struct gs_record {
  RecordKey key = {};
  int device = 0;
  int problem = 0, method = GS_METHOD_TSIT5, precision = GS_FP64;
  int d = 0, P = 0, k = 0, segw = 0;
  int arena_block = 32;  // arena slots the record kernel reserves per 32 trajectories at a time
  int64_t n = 0;
  double t0 = 0, t1 = 0, rtol = 0, atol = 0;
  int n_save = 0;
  double save_t[MAX_SAVE_HOST] = {0};
  // device buffers
  double* arena = nullptr;
  long long arena_cap = 0;
  long long* head = nullptr;
  int32_t* S = nullptr;
  int32_t* natt = nullptr;
  int32_t* status = nullptr;
  double* y_final = nullptr;
  int32_t* order = nullptr;  // scratch of the sweep's step-count sort (workspaces, ensembles up to ORDER_MAX)
  int64_t order_cap = 0;
  void* wpart = nullptr;  // per-warp shared-weight gradient partials (shared-weight problems)
  // Stored stages (gs_solve_grad's workspace, Tsit5 FP64, k = 1): segments also
  // hold each step's stage data, side_stg (n x n_save x payload) the side steps'.
  int stages = 0;
  int packed = 0;  // FP32-mixed segments in the packed layout (gs_solve_grad's workspaces)
  double* side_stg = nullptr;
  size_t side_cap = 0;  // doubles
  // chunk staging of a chunked FP32-mixed gs_solve_grad (inputs and outputs of one chunk)
  double* chunk_buf = nullptr;
  size_t chunk_cap = 0;  // doubles
  Counters* ctr = nullptr;
  Counters* ctr_host = nullptr;  // pinned
  int64_t n_cap = 0;             // capacity of the per-trajectory arrays
  long long nseg_total = 0;      // segments the record holds
  mutable size_t bytes = 0;
  // forward-order segment index, built on the first forward-mode call
  mutable long long* fwd_base = nullptr;
  mutable long long* fwd_seg = nullptr;
  cudaEvent_t ev[4] = {nullptr, nullptr, nullptr, nullptr};  // kernel timing (optional)
  // A handle's last use on each stream (the streams' ids, which are never used again), for
  // the pool; once not all of them are known (a captured use, too many streams) it does not
  // enter the pool.
  struct Use {
    unsigned long long stream;
    cudaEvent_t done;
  };
  mutable std::mutex use_mu;
  mutable std::vector<Use> uses;
  mutable bool uses_known = true;
};

// A solve context: its own reusable record workspace, so that calls on
// different contexts (and streams) run concurrently.
struct gs_context {
  gs_record* ws = nullptr;
  std::mutex mu;
  int device = 0;
};

namespace {

gs_status cuda_fail(cudaError_t e) {
  if (e == cudaErrorMemoryAllocation) return GS_ERR_OOM;
  return GS_ERR_CUDA;
}

bool pool_drain();

// cudaMalloc; if it fails, once more after the pool of freed records has given
// its memory back.
template <class T>
cudaError_t dev_alloc(T** p, size_t bytes) {
  cudaError_t e = cudaMalloc(p, bytes);
  if (e == cudaErrorMemoryAllocation) {
    cudaGetLastError();
    if (pool_drain()) e = cudaMalloc(p, bytes);
  }
  return e;
}

void free_arrays(gs_record* r) {
  cudaFree(r->head);
  cudaFree(r->S);
  cudaFree(r->natt);
  cudaFree(r->status);
  cudaFree(r->y_final);
  cudaFree(r->order);
  r->order = nullptr;
  r->order_cap = 0;
  r->head = nullptr;
  r->S = r->natt = r->status = nullptr;
  r->y_final = nullptr;
  r->n_cap = 0;
}

constexpr int kMaxDim = 8;  // largest state dimension of the registry

size_t record_bytes(const gs_record* r) {
  return (size_t)r->arena_cap * r->segw * sizeof(double) + r->side_cap * sizeof(double) +
         (size_t)r->n_cap * (sizeof(long long) + 3 * sizeof(int32_t) + kMaxDim * sizeof(double)) +
         (r->order ? (ORDER_WORDS + (size_t)r->order_cap) * sizeof(int32_t) : 0) +
         sizeof(Counters);
}

// Ensures per-trajectory arrays for n trajectories of dimension d.
gs_status ensure_arrays(gs_record* r, int64_t n, int d) {
  (void)d;
  if (r->n_cap >= n && r->head) return GS_OK;
  free_arrays(r);
  const int64_t m = n > 0 ? n : 1;
  d = kMaxDim;  // y(t1) sized for any problem, so a reused workspace never reallocates for d
  cudaError_t e;
  if ((e = dev_alloc(&r->head, m * sizeof(long long))) != cudaSuccess) return cuda_fail(e);
  if ((e = dev_alloc(&r->S, m * sizeof(int32_t))) != cudaSuccess) return cuda_fail(e);
  if ((e = dev_alloc(&r->natt, m * sizeof(int32_t))) != cudaSuccess) return cuda_fail(e);
  if ((e = dev_alloc(&r->status, m * sizeof(int32_t))) != cudaSuccess) return cuda_fail(e);
  if ((e = dev_alloc(&r->y_final, m * d * sizeof(double))) != cudaSuccess) return cuda_fail(e);
  r->n_cap = m;
  return GS_OK;
}

gs_status ensure_arena(gs_record* r, long long segs, int segw) {
  if (r->arena && r->arena_cap >= segs && r->segw == segw) return GS_OK;
  cudaFree(r->arena);
  r->arena = nullptr;
  r->arena_cap = 0;
  cudaError_t e = dev_alloc(&r->arena, (size_t)segs * segw * sizeof(double));
  if (e != cudaSuccess) return cuda_fail(e);
  r->arena_cap = segs;
  return GS_OK;
}

gs_status ensure_counters(gs_record* r) {
  if (r->ctr) return GS_OK;
  cudaError_t e = dev_alloc(&r->ctr, sizeof(Counters));
  if (e != cudaSuccess) return cuda_fail(e);
  e = cudaMallocHost(&r->ctr_host, sizeof(Counters));
  if (e != cudaSuccess) return cuda_fail(e);
  return GS_OK;
}

gs_status ensure_events(gs_record* r) {
  for (int i = 0; i < 4; ++i)
    if (!r->ev[i] && cudaEventCreate(&r->ev[i]) != cudaSuccess) return GS_ERR_CUDA;
  return GS_OK;
}

void destroy(gs_record* r) {
  if (!r) return;
  for (int i = 0; i < 4; ++i)
    if (r->ev[i]) cudaEventDestroy(r->ev[i]);
  for (const gs_record::Use& u : r->uses) cudaEventDestroy(u.done);
  free_arrays(r);
  cudaFree(r->arena);
  cudaFree(r->fwd_base);
  cudaFree(r->fwd_seg);
  cudaFree(r->side_stg);
  cudaFree(r->chunk_buf);
  cudaFree(r->ctr);
  cudaFree(r->wpart);
  cudaFreeHost(r->ctr_host);
  delete r;
}

// Freed records of at most POOL_RECORD_BYTES, the shared-weight problems' partials
// included, kept for the next gs_forward_record of the same call signature (a
// training loop records and frees one per step; allocating and freeing its buffers
// took 0.45 ms of a 2.0 ms step at 10007 Lorenz trajectories). The limits bound what
// the library holds beside the caller's allocator, 256 MB in all; with 10 saves a
// Lorenz record stays below them up to about 12300 trajectories, with 50 saves a Van
// der Pol record up to about 7100. At most POOL_RECORDS of them; the oldest is
// released for a newer one, and all of them when an allocation fails. The call that
// takes a record waits for the uses it was freed with (an event per stream): a free
// itself waits for nothing, and unlike a wait for the device neither breaks a capture
// that another stream has under way.
constexpr size_t POOL_RECORD_BYTES = size_t(128) << 20;
constexpr size_t POOL_RECORDS = 2;
constexpr size_t POOL_STREAMS = 8;
std::mutex g_pool_mu;
std::vector<gs_record*> g_pool;  // oldest first

// Notes that work on record r has been queued on stream s.
void note_use(const gs_record* r, cudaStream_t s) {
  std::lock_guard<std::mutex> lock(r->use_mu);
  if (!r->uses_known) return;
  r->uses_known = false;
  cudaStreamCaptureStatus capture = cudaStreamCaptureStatusActive;
  unsigned long long id = 0;
  if (cudaStreamIsCapturing(s, &capture) != cudaSuccess || capture != cudaStreamCaptureStatusNone) return;
  if (cudaStreamGetId(s, &id) != cudaSuccess) return;
  cudaEvent_t done = nullptr;
  for (const gs_record::Use& u : r->uses)
    if (u.stream == id) done = u.done;
  if (!done) {
    if (r->uses.size() >= POOL_STREAMS) return;
    if (cudaEventCreateWithFlags(&done, cudaEventDisableTiming) != cudaSuccess) return;
    try {
      r->uses.push_back({id, done});
    } catch (...) {
      cudaEventDestroy(done);
      return;
    }
  }
  r->uses_known = cudaEventRecord(done, s) == cudaSuccess;
}

gs_record* pool_take(const RecordKey& key) {
  int dev = 0;
  if (cudaGetDevice(&dev) != cudaSuccess) return nullptr;
  gs_record* r = nullptr;
  {
    std::lock_guard<std::mutex> lock(g_pool_mu);
    for (size_t i = 0; i < g_pool.size() && !r; ++i)
      if (g_pool[i]->device == dev && g_pool[i]->key == key) {
        r = g_pool[i];
        g_pool.erase(g_pool.begin() + i);
      }
  }
  if (!r) return nullptr;
  for (const gs_record::Use& u : r->uses)
    if (cudaEventSynchronize(u.done) != cudaSuccess) {
      destroy(r);
      return nullptr;
    }
  cudaFree(r->fwd_base);
  cudaFree(r->fwd_seg);
  r->fwd_base = r->fwd_seg = nullptr;
  return r;
}

bool pool_put(gs_record* r) {  // false: the caller releases it
  if (!r || !r->arena) return false;
  const size_t partials = r->wpart ? (size_t)ude_max_warps() * WPART_BYTES_PER_WARP : 0;
  if (record_bytes(r) + partials > POOL_RECORD_BYTES) return false;
  int dev = 0;
  if (!r->uses_known || cudaGetDevice(&dev) != cudaSuccess || dev != r->device) return false;
  gs_record* old = nullptr;
  try {
    std::lock_guard<std::mutex> lock(g_pool_mu);
    if (g_pool.size() >= POOL_RECORDS) {
      old = g_pool.front();
      g_pool.erase(g_pool.begin());
    }
    g_pool.push_back(r);
  } catch (...) {
    destroy(old);
    return false;
  }
  destroy(old);
  return true;
}

bool pool_drain() {  // whether anything was released
  std::vector<gs_record*> all;
  {
    std::lock_guard<std::mutex> lock(g_pool_mu);
    all.swap(g_pool);
  }
  for (gs_record* r : all) destroy(r);
  return !all.empty();
}

struct Call {
  int problem;
  ProblemInfo pi;
  int method, precision, k;
  int64_t max_steps;
  double h0;
  int32_t* step_counts;
  float* kernel_ms;
  double timeout_ms;
  int32_t* record_info;
  int control;
  int record_stages;
};

// Kernel launches by method.
cudaError_t launch_forward_m(int method, int problem, int precision, const FwdArgs& a, cudaStream_t s) {
  if (method == GS_METHOD_RODAS5P) return launch_rodas_forward(problem, precision, a, s);
  if (method == GS_METHOD_ROSENBROCK23) return launch_ros23_forward(problem, precision, a, s);
  if (method == GS_METHOD_VERNER7) return launch_vern7_forward(problem, precision, a, s);
  return launch_tsit5_forward(problem, precision, a, s);
}
cudaError_t launch_reverse_m(int method, int problem, int precision, const RevArgs& a, cudaStream_t s) {
  if (method == GS_METHOD_RODAS5P) return launch_rodas_reverse(problem, precision, a, s);
  if (method == GS_METHOD_ROSENBROCK23) return launch_ros23_reverse(problem, precision, a, s);
  if (method == GS_METHOD_VERNER7) return launch_vern7_reverse(problem, precision, a, s);
  return launch_tsit5_reverse(problem, precision, a, s);
}

// Waits for the work queued on s, polling with a deadline when timeout_ms > 0.
gs_status wait_stream(cudaStream_t s, double timeout_ms) {
  if (!(timeout_ms > 0.0)) return cudaStreamSynchronize(s) == cudaSuccess ? GS_OK : GS_ERR_CUDA;
  const auto start = std::chrono::steady_clock::now();
  for (;;) {
    const cudaError_t e = cudaStreamQuery(s);
    if (e == cudaSuccess) return GS_OK;
    if (e != cudaErrorNotReady) return GS_ERR_CUDA;
    const double ms = std::chrono::duration<double, std::milli>(std::chrono::steady_clock::now() - start).count();
    if (ms > timeout_ms) return GS_ERR_TIMEOUT;
    std::this_thread::sleep_for(std::chrono::microseconds(20));
  }
}

gs_status check_common(int problem_id, int64_t n, const double* params, const double* y0, const float* shared_w,
                       double t0, double t1, const double* save_t, int n_save, double rtol, double atol,
                       const gs_options* opt, Call* c) {
  if (!problem_info(problem_id, &c->pi)) return GS_ERR_UNKNOWN_PROBLEM;
  c->problem = problem_id;
  if (n < 0) return GS_ERR_INVALID_ARG;
  if (n > 0 && (!params || !y0)) return GS_ERR_INVALID_ARG;
  if (c->pi.n_shared > 0 && n > 0 && !shared_w) return GS_ERR_INVALID_ARG;
  if (!std::isfinite(t0) || !std::isfinite(t1) || !(t1 > t0)) return GS_ERR_INVALID_ARG;
  if (n_save < 0 || n_save > MAX_SAVE_HOST || (n_save > 0 && !save_t)) return GS_ERR_INVALID_ARG;
  for (int s = 0; s < n_save; ++s) {
    if (!std::isfinite(save_t[s]) || !(save_t[s] > t0) || save_t[s] > t1) return GS_ERR_INVALID_ARG;
    if (s > 0 && !(save_t[s] > save_t[s - 1])) return GS_ERR_INVALID_ARG;
  }
  if (!std::isfinite(rtol) || !std::isfinite(atol) || rtol < 0 || atol < 0 || (rtol == 0 && atol == 0))
    return GS_ERR_INVALID_ARG;
  gs_options o;
  gs_default_options(&o);
  if (opt) o = *opt;
  if (o.precision != GS_FP64 && o.precision != GS_FP32_MIXED) return GS_ERR_INVALID_ARG;
  int method = o.method == GS_METHOD_AUTO ? (c->pi.stiff ? GS_METHOD_RODAS5P : GS_METHOD_TSIT5) : o.method;
  if (method != GS_METHOD_TSIT5 && method != GS_METHOD_RODAS5P && method != GS_METHOD_ROSENBROCK23 &&
      method != GS_METHOD_VERNER7)
    return GS_ERR_INVALID_ARG;
  if (o.ckpt_k < 0 || o.ckpt_k > KMAX_HOST) return GS_ERR_INVALID_ARG;
  if (c->pi.n_shared > 0 && o.ckpt_k > 1) return GS_ERR_INVALID_ARG;  // shared weights: every state stored
  if (o.max_steps < 0 || !std::isfinite(o.h0) || o.h0 < 0) return GS_ERR_INVALID_ARG;
  c->method = method;
  c->precision = o.precision;
  c->k = o.ckpt_k;  // 0: chosen in setup_record from the free device memory
  c->max_steps = o.max_steps > 0 ? o.max_steps : 1000000;
  c->h0 = o.h0;
  c->step_counts = o.step_counts;
  c->kernel_ms = o.kernel_ms;
  if (!std::isfinite(o.timeout_ms) || o.timeout_ms < 0) return GS_ERR_INVALID_ARG;
  c->timeout_ms = o.timeout_ms;
  c->record_info = o.record_info;
  if (o.control != GS_CONTROL_FAST && o.control != GS_CONTROL_FP64) return GS_ERR_INVALID_ARG;
  if (o.control == GS_CONTROL_FP64 && (method != GS_METHOD_TSIT5 || c->pi.n_shared > 0)) return GS_ERR_INVALID_ARG;
  c->control = o.control;
  if (o.record_stages != 0 && o.record_stages != 1) return GS_ERR_INVALID_ARG;
  c->record_stages = o.record_stages;
  if (method == GS_METHOD_TSIT5 && !tsit5_supports(problem_id, o.precision)) return GS_ERR_INVALID_ARG;
  if (method == GS_METHOD_RODAS5P && !rodas_supports(problem_id, o.precision)) return GS_ERR_INVALID_ARG;
  if (method == GS_METHOD_ROSENBROCK23 && !ros23_supports(problem_id, o.precision)) return GS_ERR_INVALID_ARG;
  if (method == GS_METHOD_VERNER7 && !vern7_supports(problem_id, o.precision)) return GS_ERR_INVALID_ARG;
  return GS_OK;
}

// Enqueues the record kernel into r (counters zeroed first, statuses to `status`).
gs_status enqueue_record(gs_record* r, const Call& c, int64_t n, const double* params, const double* y0,
                         const float* shared_w, double* y_save, int32_t* status, cudaStream_t s) {
  FwdArgs a;
  std::memset(&a, 0, sizeof(a));
  a.n = n;
  a.params = params;
  a.y0 = y0;
  a.shared_w = shared_w;
  a.t0 = r->t0;
  a.t1 = r->t1;
  a.rtol = r->rtol;
  a.atol = r->atol;
  a.h0 = c.h0;
  a.control = c.control;
  a.max_steps = c.max_steps;
  a.n_save = r->n_save;
  std::memcpy(a.save_t, r->save_t, sizeof(double) * r->n_save);
  a.y_save = y_save;
  a.step_counts = c.step_counts;
  a.k = r->k;
  a.segw = r->segw;
  a.arena_block = r->arena_block;
  a.stages = r->stages;
  a.side_stg = r->stages ? r->side_stg : nullptr;
  cudaError_t e = cudaMemsetAsync(r->ctr, 0, sizeof(Counters), s);
  if (e != cudaSuccess) return cuda_fail(e);
  a.arena = r->arena;
  a.arena_cap = r->arena_cap;
  a.arena_top = &r->ctr->arena_top;
  a.overflow = &r->ctr->overflow;
  a.any_failed = &r->ctr->any_failed;
  a.head = r->head;
  a.S = r->S;
  a.natt = r->natt;
  a.status = status;
  a.y_final = r->y_final;
  a.work = &r->ctr->work_fwd;
  if (c.kernel_ms) cudaEventRecord(r->ev[0], s);
  e = r->packed ? launch_packed_forward(c.problem, a, s) : launch_forward_m(c.method, c.problem, c.precision, a, s);
  if (e != cudaSuccess) return GS_ERR_CUDA;
  if (c.kernel_ms) cudaEventRecord(r->ev[1], s);
  return GS_OK;
}

// Brings the counters to the host and waits for the work queued on s.
gs_status wait_counters(gs_record* r, const Call& c, cudaStream_t s) {
  const cudaError_t e = cudaMemcpyAsync(r->ctr_host, r->ctr, sizeof(Counters), cudaMemcpyDeviceToHost, s);
  if (e != cudaSuccess) return GS_ERR_CUDA;
  return wait_stream(s, c.timeout_ms);
}

// After a record whose arena was large enough.
void record_done(gs_record* r, const Call& c) {
  if (c.kernel_ms) cudaEventElapsedTime(&c.kernel_ms[0], r->ev[0], r->ev[1]);
  if (c.record_info) {
    c.record_info[0] = r->k;
    c.record_info[1] = r->stages;
  }
  r->nseg_total = (long long)r->ctr_host->arena_top;
}

// The arena was too small: size it to the demand just measured (+1/8), as a
// compact record if the stored-stage one does not fit.
gs_status grow_arena(gs_record* r) {
  const long long need = (long long)r->ctr_host->arena_top;
  if (r->packed && need + need / 8 + 1024 >= (1ll << 31)) {  // past a packed segment's 32-bit index
    r->packed = 0;
    r->segw = segw_of(r->d, r->k);
    cudaFree(r->arena);  // (its capacity counts packed segments)
    r->arena = nullptr;
    r->arena_cap = 0;
  }
  gs_status st = ensure_arena(r, need + need / 8 + 1024, r->segw);
  if (st == GS_ERR_OOM && r->stages) {
    r->stages = 0;
    r->segw = segw_of(r->d, r->k);
    st = ensure_arena(r, need + need / 8 + 1024, r->segw);
  }
  return st;
}

// Runs the record kernel into r, growing the arena until it fits.
gs_status run_record(gs_record* r, const Call& c, int64_t n, const double* params, const double* y0,
                     const float* shared_w, double* y_save, int32_t* status, cudaStream_t s) {
  for (int attempt = 0; attempt < 3; ++attempt) {
    gs_status st = enqueue_record(r, c, n, params, y0, shared_w, y_save, status, s);
    if (st == GS_OK) st = wait_counters(r, c, s);
    if (st != GS_OK) return st;
    if (!r->ctr_host->overflow) {
      record_done(r, c);
      return GS_OK;
    }
    if ((st = grow_arena(r)) != GS_OK) return st;
  }
  return GS_ERR_OOM;
}

// Whether a call with k = 1 records packed segments (own: gs_solve_grad's workspace).
// A packed segment's index has 31 bits; with more segments than expected the rerun is
// in the general layout. Van der Pol 3000001 / 2^22 trajectories, general / packed ms:
// 14.3 / 9.0, 19.8 / 12.4.
bool packed_call(const Call& c, int64_t n, double rtol, bool own) {
  return own && c.precision == GS_FP32_MIXED && c.method == GS_METHOD_TSIT5 && packed_supports(c.problem) &&
         (double)n * step_guess(c.problem, rtol, c.method) < 1.5e9;
}

// Checkpoint interval when the caller leaves it to the library: k = 1 (every
// accepted state stored, nothing recomputed in the reverse sweep) if the
// expected record takes at most half of the free device memory, else a
// 128-byte segment of 14 - d steps (one checkpoint per 14 - d steps).
int auto_ckpt_k(const gs_record* r, const Call& c, int64_t n, double rtol, bool own) {
  const int problem = c.problem, d = c.pi.d;
  const int segw = packed_call(c, n, rtol, own) ? PACKED_SEGW_HOST : segw_of(d, 1);
  if (r->arena && r->segw == segw && r->arena_cap >= (n > 0 ? n : 1) * (long long)(step_guess(problem) + 1))
    return 1;  // held from an earlier call of this size, in this call's layout
  size_t free_b = 0, total_b = 0;
  if (cudaMemGetInfo(&free_b, &total_b) != cudaSuccess) free_b = 0;
  const size_t held = (size_t)r->arena_cap * r->segw * sizeof(double);  // reusable by this record
  const double want = 1.25 * (double)(n > 0 ? n : 1) * step_guess(problem) * segw_of(d, 1) * sizeof(double);
  if (want <= 0.5 * (double)(free_b + held)) return 1;
  return 14 - d > 1 ? 14 - d : 1;
}

// Whether r already holds a stored-stage record for this ensemble (a workspace
// used again): nothing would be allocated, so the free memory, which takes a
// driver call to learn, does not matter.
bool holds_stages(const gs_record* r, const Call& c, int64_t n, int n_save, double rtol) {
  const long long m = n > 0 ? n : 1;
  return r->arena && r->segw == stage_segw_of(c.method, c.pi.d, c.problem) &&
         r->arena_cap >= m * (step_guess(c.problem, rtol, c.method) + 1) &&
         r->side_cap >= (size_t)m * (size_t)(n_save > 0 ? n_save : 1) * (size_t)stage_side_payload(c.method, c.pi.d, c.problem);
}

// Stored stages when the caller allows them (gs_solve_grad), the method and
// precision support them (Tsit5, Rodas5P, Rosenbrock23 or Verner7, FP64, no
// shared weights, a segment within MAX_STAGE_SEGW doubles), k is automatic, and
// the expected record with its side-step stages takes at most 70% of the free
// device memory (plus what this workspace already holds).
// The neural Robertson's lane-group form stores them too, in gs_solve_grad's own
// workspace (allow_net; record handles of shared-weight problems stay compact).
bool choose_stages(const gs_record* r, const Call& c, int64_t n, int n_save, double rtol, bool allow_net = false) {
  if (c.method != GS_METHOD_TSIT5 && c.method != GS_METHOD_RODAS5P && c.method != GS_METHOD_VERNER7 &&
      c.method != GS_METHOD_ROSENBROCK23)
    return false;
  if (c.precision != GS_FP64 || c.k > 1) return false;
  if (c.pi.n_shared > 0) {
    if (!allow_net || c.problem != GS_NEURAL_ROBERTSON || c.method != GS_METHOD_RODAS5P || n > NR_GROUP_STAGES_MAX)
      return false;
  } else if (stage_segw_of(c.method, c.pi.d, c.problem) > MAX_STAGE_SEGW) {
    return false;
  }
  if (holds_stages(r, c, n, n_save, rtol)) return true;
  size_t free_b = 0, total_b = 0;
  if (cudaMemGetInfo(&free_b, &total_b) != cudaSuccess) return false;
  const double held = (double)r->arena_cap * r->segw * sizeof(double) + (double)r->side_cap * sizeof(double);
  const double m = (double)(n > 0 ? n : 1);
  const double want =
      m * (1.1 * step_guess(c.problem, rtol, c.method) + 1.0) * stage_segw_of(c.method, c.pi.d, c.problem) * sizeof(double) +
      m * n_save * (double)stage_side_payload(c.method, c.pi.d, c.problem) * sizeof(double);
  return want <= 0.7 * ((double)free_b + held);
}

gs_status setup_record(gs_record* r, const Call& c, int64_t n, double t0, double t1, const double* save_t,
                       int n_save, double rtol, double atol, bool allow_stages = false, bool own = false) {  // own: gs_solve_grad's workspace
  cudaGetDevice(&r->device);
  r->problem = c.problem;
  r->method = c.method;
  r->precision = c.precision;
  r->d = c.pi.d;
  r->P = c.pi.P;
  r->stages = (allow_stages && choose_stages(r, c, n, n_save, rtol, own)) ? 1 : 0;
  r->k = r->stages ? 1 : (c.k > 0 ? c.k : (c.pi.n_shared > 0 ? 1 : auto_ckpt_k(r, c, n, rtol, own)));
  if (c.pi.n_shared > 0 && !r->wpart) {
    const cudaError_t e = dev_alloc(&r->wpart, (size_t)ude_max_warps() * WPART_BYTES_PER_WARP);
    if (e != cudaSuccess) return cuda_fail(e);
  }
  r->n = n;
  r->t0 = t0;
  r->t1 = t1;
  r->rtol = rtol;
  r->atol = atol;
  r->n_save = n_save;
  if (n_save) std::memcpy(r->save_t, save_t, sizeof(double) * n_save);
  gs_status st = ensure_counters(r);
  if (st != GS_OK) return st;
  if (c.kernel_ms && (st = ensure_events(r)) != GS_OK) return st;
  st = ensure_arrays(r, n, r->d);
  if (st != GS_OK) return st;
  if (own && c.precision == GS_FP64 && c.pi.n_shared == 0 && n <= ORDER_MAX && r->order_cap < n) {
    cudaFree(r->order);
    r->order = nullptr;
    r->order_cap = 0;
    if (dev_alloc(&r->order, (ORDER_WORDS + n) * sizeof(int32_t)) == cudaSuccess) {
      r->order_cap = n;
    } else {  // no room: the sweep takes the trajectories as they come
      r->order = nullptr;
      cudaGetLastError();
    }
  }
  if (r->stages) {
    const size_t need = (size_t)(n > 0 ? n : 1) * (size_t)(n_save > 0 ? n_save : 1) *
                        (size_t)stage_side_payload(c.method, r->d, c.problem);
    if (r->side_cap < need) {
      cudaFree(r->side_stg);
      r->side_stg = nullptr;
      r->side_cap = 0;
      const cudaError_t e = dev_alloc(&r->side_stg, need * sizeof(double));
      if (e != cudaSuccess) {
        r->stages = 0;  // fall back to the compact record
        r->k = c.k > 0 ? c.k : (c.pi.n_shared > 0 ? 1 : auto_ckpt_k(r, c, n, rtol, own));
      } else {
        r->side_cap = need;
      }
    }
  }
  r->packed = r->k == 1 && packed_call(c, n, rtol, own);
  const int segw = r->stages ? stage_segw_of(c.method, r->d, c.problem) : (r->packed ? PACKED_SEGW_HOST : segw_of(r->d, r->k));
  if (r->segw != segw) {
    cudaFree(r->arena);
    r->arena = nullptr;
    r->arena_cap = 0;
    r->segw = segw;
  }
  // Expected segments, plus the unused tails of the record kernel's slot blocks: 32
  // trajectories (one warp, or the warps of their lane groups) reserve about an eighth
  // of their expected segments at a time (32 to ARENA_BLOCK_HOST slots), and leave less
  // than that unused.
  const long long m = n > 0 ? n : 1;
  const long long per_traj = (step_guess(c.problem, rtol, c.method) + r->k - 1) / r->k + 1;
  const long long warps = std::min<long long>((m + 31) / 32, 4096 * 4);
  long long blk = 32;
  while (blk < ARENA_BLOCK_HOST && 8 * 2 * blk <= m * per_traj / warps) blk *= 2;
  r->arena_block = (int)blk;
  const long long slack = warps * blk;
  const long long want = m * per_traj + slack;
  if (r->arena_cap > 0 && r->arena_cap < want / 4) {  // far too small for this ensemble: start over
    cudaFree(r->arena);
    r->arena = nullptr;
    r->arena_cap = 0;
  }
  if (r->arena_cap == 0) {
    st = ensure_arena(r, want, segw);
    if (st == GS_ERR_OOM && r->stages) {  // the stored-stage record does not fit: compact record
      r->stages = 0;
      r->k = c.k > 0 ? c.k : (c.pi.n_shared > 0 ? 1 : auto_ckpt_k(r, c, n, rtol, own));
      r->segw = segw_of(r->d, r->k);
      st = ensure_arena(r, m * ((step_guess(c.problem, rtol, c.method) + r->k - 1) / r->k + 1) + slack, r->segw);
      // (the block size chosen above stays: it depends on the ensemble, not the layout)
    }
    if (st != GS_OK) return st;
  }
  return GS_OK;
}

gs_status launch_reverse(const gs_record* r, const double* params, const float* shared_w,
                         const double* y_save_bar, double* loss, double* params_bar, double* y0_bar,
                         float* shared_w_bar, const int32_t* status, bool fresh_counters, cudaStream_t s) {
  RevArgs a;
  std::memset(&a, 0, sizeof(a));
  a.n = r->n;
  a.params = params;
  a.shared_w = shared_w;
  a.shared_w_bar = shared_w_bar;
  a.t0 = r->t0;
  a.t1 = r->t1;
  a.n_save = r->n_save;
  std::memcpy(a.save_t, r->save_t, sizeof(double) * r->n_save);
  a.y_save_bar = y_save_bar;
  a.loss = loss;
  a.params_bar = params_bar;
  a.y0_bar = y0_bar;
  a.status = status;
  a.arena = r->arena;
  a.arena_cap = r->arena_cap;
  a.head = r->head;
  a.S = r->S;
  a.y_final = r->y_final;
  a.wpart = r->wpart;
  a.order_buf = r->order_cap >= r->n ? r->order : nullptr;  // (workspaces)
  a.work = &r->ctr->work_rev;
  a.k = r->k;
  a.segw = r->segw;
  a.stages = r->stages;
  a.side_stg = r->stages ? r->side_stg : nullptr;
  a.tc_error = &r->ctr->tc_error;
  cudaError_t e = fresh_counters ? cudaSuccess : cudaMemsetAsync(&r->ctr->work_rev, 0, sizeof(unsigned long long), s);
  if (e != cudaSuccess) return GS_ERR_CUDA;
  e = r->packed ? launch_packed_reverse(r->problem, a, s) : launch_reverse_m(r->method, r->problem, r->precision, a, s);
  return e == cudaSuccess ? GS_OK : GS_ERR_CUDA;
}

// Forward-mode replay launches over directions [g0, g1) of the call, at most
// JVP_MAX_DIR per launch; `a` carries everything but the per-launch fields.
gs_status launch_jvp_range(const gs_record* r, JvpArgs a, int g0, int g1, double* loss_out, cudaStream_t s) {
  const int64_t n = r->n;
  const double* pdot = a.params_dot;
  const double* ydot = a.y0_dot;
  double* ldot = a.loss_dot;
  double* ysd = a.y_save_dot;
  for (int g = g0; g < g1; g += JVP_MAX_DIR) {
    const int nd = (g1 - g) < JVP_MAX_DIR ? (g1 - g) : JVP_MAX_DIR;
    a.dir0 = g;
    a.nd = nd;
    a.loss = (g == g0) ? loss_out : nullptr;
    if (!a.basis) {
      const int64_t q = g - g0;
      a.params_dot = pdot ? pdot + q * r->P * n : nullptr;
      a.y0_dot = ydot ? ydot + q * r->d * n : nullptr;
      a.loss_dot = ldot + q * n;
      a.y_save_dot = ysd ? ysd + q * (int64_t)r->n_save * r->d * n : nullptr;
    }
    cudaError_t e = cudaMemsetAsync(&r->ctr->work_jvp, 0, sizeof(unsigned long long), s);
    if (e != cudaSuccess) return GS_ERR_CUDA;
    e = launch_jvp(r->method, r->problem, a, s);
    if (e != cudaSuccess) return GS_ERR_CUDA;
  }
  return GS_OK;
}

// The record's segments in forward order (built once, on the stream of the
// first forward-mode call).
gs_status ensure_fwd_index(const gs_record* r, cudaStream_t s) {
  if (r->fwd_base) return GS_OK;
  long long* base = nullptr;
  long long* seg = nullptr;
  cudaError_t e = dev_alloc(&base, (size_t)r->n * sizeof(long long));
  if (e == cudaSuccess) e = dev_alloc(&seg, (size_t)(r->nseg_total > 0 ? r->nseg_total : 1) * sizeof(long long));
  if (e == cudaSuccess) e = cudaMemsetAsync(&r->ctr->work_jvp, 0, sizeof(unsigned long long), s);
  if (e == cudaSuccess)
    e = launch_fwd_index(r->n, r->head, r->S, r->status, r->arena, r->arena_cap, r->k, r->segw, &r->ctr->work_jvp,
                         base, seg, r->nseg_total, s);
  if (e != cudaSuccess) {
    cudaFree(base);
    cudaFree(seg);
    return cuda_fail(e);
  }
  r->fwd_base = base;
  r->fwd_seg = seg;
  r->bytes += (size_t)(r->n + (r->nseg_total > 0 ? r->nseg_total : 1)) * sizeof(long long);
  return GS_OK;
}

// The parts of the forward-mode arguments that come from the record.
gs_status jvp_common(const gs_record* r, const double* params, const double* y0, cudaStream_t s, JvpArgs* a) {
  if (!params || !y0) return GS_ERR_INVALID_ARG;
  if (!jvp_supports(r->method, r->problem)) return GS_ERR_INVALID_ARG;
  int dev = 0;
  cudaGetDevice(&dev);
  if (dev != r->device) return GS_ERR_INVALID_ARG;
  const gs_status st = ensure_fwd_index(r, s);
  if (st != GS_OK) return st;
  std::memset(a, 0, sizeof(*a));
  a->n = r->n;
  a->params = params;
  a->y0 = y0;
  a->t0 = r->t0;
  a->t1 = r->t1;
  a->n_save = r->n_save;
  std::memcpy(a->save_t, r->save_t, sizeof(double) * r->n_save);
  a->status = r->status;
  a->arena = r->arena;
  a->S = r->S;
  a->fwd_base = r->fwd_base;
  a->fwd_seg = r->fwd_seg;
  a->work = &r->ctr->work_jvp;
  a->k = r->k;
  a->segw = r->segw;
  return GS_OK;
}

bool overlap(const void* x, size_t xb, const void* y, size_t yb) {
  const char *p = static_cast<const char*>(x), *q = static_cast<const char*>(y);
  return p && q && p < q + yb && q < p + xb;
}

// Record then reverse into workspace r (the body of gs_solve_grad[_ctx]). The
// reverse sweep is queued right behind the record, and the host waits once, for
// both: if the arena turned out too small, the sweep has met segment indices past
// its end (which it turns into NaN gradients), and both run again on the grown
// arena. Only calls whose outputs overlap their inputs, or with a wait deadline,
// wait for the record first. At 1024 Lorenz trajectories the round trip between
// the two, the status copy and the memory query were 70 us of an 831 us call.
gs_status solve_grad_in(gs_record* r, const Call& c, int64_t n, const double* params, const double* y0,
                        const float* shared_w, double t0, double t1, const double* save_t, int n_save, double rtol,
                        double atol, cudaStream_t s, double* loss_out, double* params_bar, double* y0_bar,
                        float* shared_w_bar, int32_t* traj_status, bool allow_stages) {
  gs_status st = setup_record(r, c, n, t0, t1, save_t, n_save, rtol, atol, allow_stages, true);
  if (st != GS_OK) return st;
  const size_t nb = (size_t)n * sizeof(double);
  const void* outs[5] = {loss_out, params_bar, y0_bar, shared_w_bar, traj_status};
  const size_t outb[5] = {nb, nb * c.pi.P, nb * c.pi.d, sizeof(float) * c.pi.n_shared, sizeof(int32_t) * (size_t)n};
  const void* ins[3] = {params, y0, shared_w};
  const size_t inb[3] = {nb * c.pi.P, nb * c.pi.d, sizeof(float) * c.pi.n_shared};
  bool apart = c.timeout_ms > 0.0;
  for (int i = 0; i < 5; ++i)
    for (int j = 0; j < 3; ++j) apart = apart || overlap(outs[i], outb[i], ins[j], inb[j]);
  int32_t* status = apart ? r->status : traj_status;
  if (apart && (st = run_record(r, c, n, params, y0, shared_w, nullptr, status, s)) != GS_OK) return st;
  for (int attempt = 0;; ++attempt) {
    if (attempt == 3) return GS_ERR_OOM;
    if (!apart && (st = enqueue_record(r, c, n, params, y0, shared_w, nullptr, status, s)) != GS_OK) return st;
    if (c.kernel_ms) cudaEventRecord(r->ev[2], s);
    st = launch_reverse(r, params, shared_w, nullptr, loss_out, params_bar, y0_bar, shared_w_bar, status, true, s);
    if (st != GS_OK) return st;
    if (c.kernel_ms) cudaEventRecord(r->ev[3], s);
    if (apart && cudaMemcpyAsync(traj_status, r->status, n * sizeof(int32_t), cudaMemcpyDeviceToDevice, s) !=
                     cudaSuccess)
      return GS_ERR_CUDA;
    if ((st = wait_counters(r, c, s)) != GS_OK) return st;
    if (!r->ctr_host->overflow) break;
    if ((st = grow_arena(r)) != GS_OK) return st;
  }
  record_done(r, c);
  if (c.kernel_ms) cudaEventElapsedTime(&c.kernel_ms[1], r->ev[2], r->ev[3]);
  if (r->ctr_host->tc_error) return GS_ERR_CUDA;
  return r->ctr_host->any_failed ? GS_ERR_TRAJ_FAILED : GS_OK;
}

// An FP32-mixed gs_solve_grad of more than two chunks runs chunk by chunk
// (shared-weight problems, step_counts and a wait deadline excepted): the
// record of 2^21 Lorenz trajectories takes ~3.4 GB against ~27 GB at 2^24, and the
// reverse sweep's scattered per-lane segment reads run faster over the smaller
// arena (Lorenz 2^24, rtol 1e-6, measured: 26.7 / 26.2 / 26.0 ms in chunks of 2^20 /
// 2^21 / 2^22; with the general segments 40.7 / 40.4 / 41.4 against 44.0
// ms in one piece). Trajectories are independent, so
// the results equal the one-piece call bit for bit.
//
// The FP64 form, bound by its FP64 pipe, is slower in chunks when the whole
// stored-stage record fits (608 against 603 ms at Lorenz 2^24 in chunks of
// 2^22) and then runs in one piece. An FP64 call whose whole stored-stage
// record would not fit in device memory
// (it then records compactly and its reverse sweep recomputes every stage) but
// a chunk's would, runs in the largest power-of-two chunks (2^18 to 2^23) whose
// stored-stage record fits (gs_solve_grad only; contexts record compactly):
// the reverse sweep then reads the stages instead of recomputing them.
constexpr int64_t MIXED_CHUNK = int64_t(1) << 21;

int64_t solve_chunk(const gs_record* r, const Call& c, int64_t n, int n_save, double rtol, bool allow_stages) {
  if (c.pi.n_shared > 0 || c.step_counts || c.timeout_ms > 0.0) return 0;
  if (c.precision == GS_FP32_MIXED) return n > 2 * MIXED_CHUNK ? MIXED_CHUNK : 0;
  if (!allow_stages || choose_stages(r, c, n, n_save, rtol)) return 0;
  for (int64_t m = int64_t(1) << 23; m >= (int64_t(1) << 18); m >>= 1)
    if (m < n && choose_stages(r, c, m, n_save, rtol)) return m;
  return 0;
}

gs_status solve_grad_chunked(gs_record* r, const Call& c, int64_t n, int64_t ch, const double* params,
                             const double* y0, double t0, double t1, const double* save_t, int n_save, double rtol,
                             double atol, cudaStream_t s, double* loss_out, double* params_bar, double* y0_bar,
                             int32_t* traj_status, bool allow_stages) {
  const int P = c.pi.P, d = c.pi.d;
  const size_t need = (size_t)(2 * (P + d)) * (size_t)ch;  // [P + d][ch] in, [P + d][ch] out
  if (r->chunk_cap < need) {
    cudaFree(r->chunk_buf);
    r->chunk_buf = nullptr;
    r->chunk_cap = 0;
    if (dev_alloc(&r->chunk_buf, need * sizeof(double)) != cudaSuccess) {
      cudaGetLastError();  // no staging: the one-piece call
      return solve_grad_in(r, c, n, params, y0, nullptr, t0, t1, save_t, n_save, rtol, atol, s, loss_out,
                           params_bar, y0_bar, nullptr, traj_status, allow_stages);
    }
    r->chunk_cap = need;
  }
  double* in_p = r->chunk_buf;             // [P][ch]
  double* in_y = in_p + (size_t)P * ch;    // [d][ch]
  double* out_p = in_y + (size_t)d * ch;   // [P][ch]
  double* out_y = out_p + (size_t)P * ch;  // [d][ch]
  float kms[2] = {0.0f, 0.0f}, sum[2] = {0.0f, 0.0f};
  Call cc = c;
  if (c.kernel_ms) cc.kernel_ms = kms;
  bool failed = false;
  const size_t pitch = (size_t)n * sizeof(double);
  for (int64_t k0 = 0; k0 < n; k0 += ch) {
    const int64_t nc = std::min(ch, n - k0);
    const size_t w = (size_t)nc * sizeof(double);
    if (cudaMemcpy2DAsync(in_p, w, params + k0, pitch, w, P, cudaMemcpyDeviceToDevice, s) != cudaSuccess ||
        cudaMemcpy2DAsync(in_y, w, y0 + k0, pitch, w, d, cudaMemcpyDeviceToDevice, s) != cudaSuccess)
      return GS_ERR_CUDA;
    const gs_status st = solve_grad_in(r, cc, nc, in_p, in_y, nullptr, t0, t1, save_t, n_save, rtol, atol, s,
                                       loss_out ? loss_out + k0 : nullptr, params_bar ? out_p : nullptr,
                                       y0_bar ? out_y : nullptr, nullptr, traj_status + k0, allow_stages);
    if (st == GS_ERR_TRAJ_FAILED)
      failed = true;
    else if (st != GS_OK)
      return st;
    if (params_bar &&
        cudaMemcpy2DAsync(params_bar + k0, pitch, out_p, w, w, P, cudaMemcpyDeviceToDevice, s) != cudaSuccess)
      return GS_ERR_CUDA;
    if (y0_bar && cudaMemcpy2DAsync(y0_bar + k0, pitch, out_y, w, w, d, cudaMemcpyDeviceToDevice, s) != cudaSuccess)
      return GS_ERR_CUDA;
    sum[0] += kms[0];
    sum[1] += kms[1];
  }
  const gs_status ws = wait_stream(s, 0.0);
  if (ws != GS_OK) return ws;
  if (c.kernel_ms) {
    c.kernel_ms[0] = sum[0];
    c.kernel_ms[1] = sum[1];
  }
  return failed ? GS_ERR_TRAJ_FAILED : GS_OK;
}

// gs_solve_grad's reusable record, one per device.
std::mutex g_ws_mu;
std::vector<gs_record*> g_ws;

gs_record* workspace(int dev) {
  if ((int)g_ws.size() <= dev) g_ws.resize(dev + 1, nullptr);
  if (!g_ws[dev]) g_ws[dev] = new (std::nothrow) gs_record();
  return g_ws[dev];
}

// gs_solve_grad_host's device staging, one per device (guarded by g_ws_mu):
// two input and two output chunk slots, a copy stream per direction, a
// compute stream and the events that order them.
struct HostPipe {
  cudaStream_t comp = nullptr, h2d = nullptr, d2h = nullptr;
  cudaEvent_t in_ready[2] = {nullptr, nullptr}, out_ready[2] = {nullptr, nullptr},
              out_free[2] = {nullptr, nullptr};
  double* in[2] = {nullptr, nullptr};   // [P + d][chunk]
  double* out[2] = {nullptr, nullptr};  // [1 + P + d][chunk] doubles, then [chunk] int32 status
  size_t in_bytes = 0, out_bytes = 0;
};
std::vector<HostPipe*> g_pipe;

gs_status host_pipe(int dev, size_t in_bytes, size_t out_bytes, HostPipe** out) {
  if ((int)g_pipe.size() <= dev) g_pipe.resize(dev + 1, nullptr);
  if (!g_pipe[dev]) {
    HostPipe* hp = new (std::nothrow) HostPipe();
    if (!hp) return GS_ERR_OOM;
    if (cudaStreamCreateWithFlags(&hp->comp, cudaStreamNonBlocking) != cudaSuccess ||
        cudaStreamCreateWithFlags(&hp->h2d, cudaStreamNonBlocking) != cudaSuccess ||
        cudaStreamCreateWithFlags(&hp->d2h, cudaStreamNonBlocking) != cudaSuccess)
      return GS_ERR_CUDA;
    for (int i = 0; i < 2; ++i)
      if (cudaEventCreateWithFlags(&hp->in_ready[i], cudaEventDisableTiming) != cudaSuccess ||
          cudaEventCreateWithFlags(&hp->out_ready[i], cudaEventDisableTiming) != cudaSuccess ||
          cudaEventCreateWithFlags(&hp->out_free[i], cudaEventDisableTiming) != cudaSuccess)
        return GS_ERR_CUDA;
    g_pipe[dev] = hp;
  }
  HostPipe* hp = g_pipe[dev];
  if (hp->in_bytes < in_bytes || hp->out_bytes < out_bytes) {
    for (int i = 0; i < 2; ++i) {
      cudaFree(hp->in[i]);
      cudaFree(hp->out[i]);
      hp->in[i] = hp->out[i] = nullptr;
    }
    hp->in_bytes = hp->out_bytes = 0;
    for (int i = 0; i < 2; ++i)
      if (dev_alloc(&hp->in[i], in_bytes) != cudaSuccess || dev_alloc(&hp->out[i], out_bytes) != cudaSuccess) {
        cudaGetLastError();
        return GS_ERR_OOM;
      }
    hp->in_bytes = in_bytes;
    hp->out_bytes = out_bytes;
  }
  *out = hp;
  return GS_OK;
}

// Rows [rows][n] of a host SoA array, trajectories [k0, k0 + nc), to or from a
// device [rows][nc] block: one strided copy.
cudaError_t copy_rows(void* dst, size_t dpitch, const void* src, size_t spitch, size_t width, int rows,
                      cudaMemcpyKind kind, cudaStream_t s) {
  if (rows <= 0 || width == 0) return cudaSuccess;
  return cudaMemcpy2DAsync(dst, dpitch, src, spitch, width, (size_t)rows, kind, s);
}

}  // namespace

extern "C" {

const char* gs_status_string(gs_status s) {
  switch (s) {
    case GS_OK: return "ok";
    case GS_ERR_INVALID_ARG: return "invalid argument";
    case GS_ERR_UNKNOWN_PROBLEM: return "unknown problem id";
    case GS_ERR_OOM: return "device out of memory";
    case GS_ERR_CUDA: return "CUDA error";
    case GS_ERR_TRAJ_FAILED: return "one or more trajectories failed (see traj_status)";
    case GS_ERR_TIMEOUT: return "timed out waiting for the device";
  }
  return "unknown status";
}

gs_status gs_default_options(gs_options* opt) {
  if (!opt) return GS_ERR_INVALID_ARG;
  std::memset(opt, 0, sizeof(*opt));
  opt->precision = GS_FP64;
  opt->method = GS_METHOD_AUTO;
  return GS_OK;
}

gs_status gs_problem_info(int problem_id, int* d, int* P, int* stiff, int* n_shared) {
  ProblemInfo pi;
  if (!problem_info(problem_id, &pi)) return GS_ERR_UNKNOWN_PROBLEM;
  if (d) *d = pi.d;
  if (P) *P = pi.P;
  if (stiff) *stiff = pi.stiff;
  if (n_shared) *n_shared = pi.n_shared;
  return GS_OK;
}

gs_status gs_forward_record(int problem_id, int64_t n, const double* params, const double* y0,
                            const float* shared_w, double t0, double t1, const double* save_t, int n_save,
                            double rtol, double atol, const gs_options* opt, gs_stream stream,
                            double* y_save_out, int32_t* traj_status, gs_record** rec_out) {
  if (!rec_out) return GS_ERR_INVALID_ARG;
  *rec_out = nullptr;
  Call c;
  gs_status st = check_common(problem_id, n, params, y0, shared_w, t0, t1, save_t, n_save, rtol, atol, opt, &c);
  if (st != GS_OK) return st;
  if (n > 0 && !traj_status) return GS_ERR_INVALID_ARG;
  c.timeout_ms = 0.0;  // the record handle owns the work: wait for it
  const RecordKey key = {c.problem, c.method, c.precision, c.k, c.record_stages, n_save, n, rtol};
  gs_record* r = pool_take(key);
  if (!r) r = new (std::nothrow) gs_record();
  if (!r) return GS_ERR_OOM;
  r->key = key;
  st = setup_record(r, c, n, t0, t1, save_t, n_save, rtol, atol, c.record_stages == 1);
  if (st != GS_OK) { destroy(r); return st; }
  cudaStream_t s = (cudaStream_t)stream;
  if (n > 0) {
    st = run_record(r, c, n, params, y0, shared_w, y_save_out, r->status, s);
    if (st != GS_OK) { destroy(r); return st; }
    cudaError_t e = cudaMemcpyAsync(traj_status, r->status, n * sizeof(int32_t), cudaMemcpyDeviceToDevice, s);
    if (e == cudaSuccess) e = cudaStreamSynchronize(s);
    if (e != cudaSuccess) { destroy(r); return GS_ERR_CUDA; }
  }
  r->bytes = record_bytes(r);
  *rec_out = r;
  return (n > 0 && r->ctr_host->any_failed) ? GS_ERR_TRAJ_FAILED : GS_OK;
}

gs_status gs_reverse(const gs_record* rec, const double* params, const double* y0, const float* shared_w,
                     const double* y_save_bar, double* loss_out, double* params_bar, double* y0_bar,
                     float* shared_w_bar, gs_stream stream) {
  (void)y0;
  if (!rec) return GS_ERR_INVALID_ARG;
  if (rec->n == 0) return GS_OK;
  if (!params) return GS_ERR_INVALID_ARG;
  ProblemInfo pi;
  problem_info(rec->problem, &pi);
  if (pi.n_shared > 0 && !shared_w) return GS_ERR_INVALID_ARG;
  int dev = 0;
  cudaGetDevice(&dev);
  if (dev != rec->device) return GS_ERR_INVALID_ARG;
  const gs_status st = launch_reverse(rec, params, shared_w, y_save_bar, loss_out, params_bar, y0_bar, shared_w_bar,
                                      rec->status, false, (cudaStream_t)stream);
  note_use(rec, (cudaStream_t)stream);
  return st;
}

gs_status gs_replay_jvp(const gs_record* rec, const double* params, const double* y0, int n_dir,
                        const double* params_dot, const double* y0_dot, double* loss_out, double* loss_dot,
                        double* y_save_dot, gs_stream stream) {
  if (!rec) return GS_ERR_INVALID_ARG;
  if (n_dir < 1 || !loss_dot) return GS_ERR_INVALID_ARG;
  if (rec->n == 0) return GS_OK;
  JvpArgs a;
  const gs_status st = jvp_common(rec, params, y0, (cudaStream_t)stream, &a);
  if (st != GS_OK) return st;
  a.params_dot = params_dot;
  a.y0_dot = y0_dot;
  a.loss_dot = loss_dot;
  a.y_save_dot = y_save_dot;
  const gs_status sl = launch_jvp_range(rec, a, 0, n_dir, loss_out, (cudaStream_t)stream);
  note_use(rec, (cudaStream_t)stream);
  return sl;
}

gs_status gs_forward_grad(const gs_record* rec, const double* params, const double* y0, double* loss_out,
                          double* params_bar, double* y0_bar, gs_stream stream) {
  if (!rec) return GS_ERR_INVALID_ARG;
  if (!params_bar && !y0_bar) return GS_ERR_INVALID_ARG;
  if (rec->n == 0) return GS_OK;
  JvpArgs a;
  const gs_status st = jvp_common(rec, params, y0, (cudaStream_t)stream, &a);
  if (st != GS_OK) return st;
  a.basis = 1;
  a.grad_p = params_bar;
  a.grad_y = y0_bar;
  const int g0 = params_bar ? 0 : rec->P;
  const int g1 = y0_bar ? rec->P + rec->d : rec->P;
  const gs_status sl = launch_jvp_range(rec, a, g0, g1, loss_out, (cudaStream_t)stream);
  note_use(rec, (cudaStream_t)stream);
  return sl;
}

gs_status gs_record_refresh(gs_record* rec, const double* params, const double* y0, const float* shared_w,
                            gs_stream stream) {
  if (!rec) return GS_ERR_INVALID_ARG;
  if (rec->n == 0) return GS_OK;
  if (!params || !y0) return GS_ERR_INVALID_ARG;
  ProblemInfo pi;
  problem_info(rec->problem, &pi);
  if (pi.n_shared > 0 && !shared_w) return GS_ERR_INVALID_ARG;
  if (rec->stages) return GS_ERR_INVALID_ARG;  // its stored stage data would go stale
  int dev = 0;
  cudaGetDevice(&dev);
  if (dev != rec->device) return GS_ERR_INVALID_ARG;
  RevArgs a;
  std::memset(&a, 0, sizeof(a));
  a.n = rec->n;
  a.params = params;
  a.shared_w = shared_w;
  a.status = rec->status;
  a.arena = rec->arena;
  a.arena_cap = rec->arena_cap;
  a.head = rec->head;
  a.S = rec->S;
  a.k = rec->k;
  a.segw = rec->segw;
  const cudaStream_t s = (cudaStream_t)stream;
  const cudaError_t e =
      (rec->method == GS_METHOD_RODAS5P)
          ? launch_rodas_refresh(rec->problem, rec->precision, a, rec->arena, rec->y_final, y0, s)
      : (rec->method == GS_METHOD_ROSENBROCK23)
          ? launch_ros23_refresh(rec->problem, rec->precision, a, rec->arena, rec->y_final, y0, s)
      : (rec->method == GS_METHOD_VERNER7)
          ? launch_vern7_refresh(rec->problem, rec->precision, a, rec->arena, rec->y_final, y0, s)
          : launch_tsit5_refresh(rec->problem, rec->precision, a, rec->arena, rec->y_final, y0, s);
  note_use(rec, s);
  return e == cudaSuccess ? GS_OK : GS_ERR_CUDA;
}

gs_status gs_solve_grad(int problem_id, int64_t n, const double* params, const double* y0,
                        const float* shared_w, double t0, double t1, const double* save_t, int n_save,
                        double rtol, double atol, const gs_options* opt, gs_stream stream, double* loss_out,
                        double* params_bar, double* y0_bar, float* shared_w_bar, int32_t* traj_status) {
  Call c;
  gs_status st = check_common(problem_id, n, params, y0, shared_w, t0, t1, save_t, n_save, rtol, atol, opt, &c);
  if (st != GS_OK) return st;
  if (n == 0) return GS_OK;
  if (!traj_status) return GS_ERR_INVALID_ARG;
  int dev = 0;
  cudaGetDevice(&dev);
  std::lock_guard<std::mutex> lock(g_ws_mu);
  gs_record* r = workspace(dev);
  if (!r) return GS_ERR_OOM;
  if (const int64_t ch = solve_chunk(r, c, n, n_save, rtol, true))
    return solve_grad_chunked(r, c, n, ch, params, y0, t0, t1, save_t, n_save, rtol, atol, (cudaStream_t)stream,
                              loss_out, params_bar, y0_bar, traj_status, true);
  return solve_grad_in(r, c, n, params, y0, shared_w, t0, t1, save_t, n_save, rtol, atol, (cudaStream_t)stream,
                       loss_out, params_bar, y0_bar, shared_w_bar, traj_status, true);
}

gs_status gs_solve_grad_host(int problem_id, int64_t n, const double* params, const double* y0,
                             const float* shared_w, double t0, double t1, const double* save_t, int n_save,
                             double rtol, double atol, const gs_options* opt, int64_t chunk, double* loss_out,
                             double* params_bar, double* y0_bar, float* shared_w_bar, int32_t* traj_status) {
  Call c;
  gs_status st = check_common(problem_id, n, params, y0, shared_w, t0, t1, save_t, n_save, rtol, atol, opt, &c);
  if (st != GS_OK) return st;
  if (chunk < 0 || (opt && opt->step_counts)) return GS_ERR_INVALID_ARG;
  if (n == 0) return GS_OK;
  if (!traj_status) return GS_ERR_INVALID_ARG;
  const int P = c.pi.P, d = c.pi.d;
  int64_t ch = chunk > 0 ? chunk : ((int64_t)1 << 21);
  if (c.pi.n_shared > 0 || ch > n) ch = n;  // a shared-weight gradient sums the whole ensemble: one chunk
  const int64_t nchunks = (n + ch - 1) / ch;
  int dev = 0;
  cudaGetDevice(&dev);
  std::lock_guard<std::mutex> lock(g_ws_mu);
  gs_record* r = workspace(dev);
  if (!r) return GS_ERR_OOM;
  HostPipe* hp = nullptr;
  const size_t in_bytes = (size_t)(P + d) * ch * sizeof(double);
  const size_t out_bytes = (size_t)(1 + P + d) * ch * sizeof(double) + (size_t)ch * sizeof(int32_t);
  if ((st = host_pipe(dev, in_bytes, out_bytes, &hp)) != GS_OK) return st;
  const size_t hp_row = (size_t)n * sizeof(double), hs_row = (size_t)n * sizeof(int32_t);

  auto upload = [&](int64_t ci) -> cudaError_t {
    const int64_t k0 = ci * ch, nc = std::min(ch, n - k0);
    const int slot = (int)(ci & 1);
    double* din = hp->in[slot];
    const size_t w = (size_t)nc * sizeof(double);
    cudaError_t e = copy_rows(din, w, params + k0, hp_row, w, P, cudaMemcpyHostToDevice, hp->h2d);
    if (e == cudaSuccess)
      e = copy_rows(din + (size_t)P * nc, w, y0 + k0, hp_row, w, d, cudaMemcpyHostToDevice, hp->h2d);
    if (e == cudaSuccess) e = cudaEventRecord(hp->in_ready[slot], hp->h2d);
    return e;
  };
  auto download = [&](int64_t ci) -> cudaError_t {
    const int64_t k0 = ci * ch, nc = std::min(ch, n - k0);
    const int slot = (int)(ci & 1);
    const double* dout = hp->out[slot];
    const size_t w = (size_t)nc * sizeof(double);
    cudaError_t e = cudaStreamWaitEvent(hp->d2h, hp->out_ready[slot], 0);
    if (e == cudaSuccess && loss_out)
      e = copy_rows(loss_out + k0, hp_row, dout, w, w, 1, cudaMemcpyDeviceToHost, hp->d2h);
    if (e == cudaSuccess && params_bar)
      e = copy_rows(params_bar + k0, hp_row, dout + nc, w, w, P, cudaMemcpyDeviceToHost, hp->d2h);
    if (e == cudaSuccess && y0_bar)
      e = copy_rows(y0_bar + k0, hp_row, dout + (size_t)(1 + P) * nc, w, w, d, cudaMemcpyDeviceToHost, hp->d2h);
    if (e == cudaSuccess)
      e = copy_rows(traj_status + k0, hs_row, dout + (size_t)(1 + P + d) * nc, (size_t)nc * sizeof(int32_t),
                    (size_t)nc * sizeof(int32_t), 1, cudaMemcpyDeviceToHost, hp->d2h);
    if (e == cudaSuccess) e = cudaEventRecord(hp->out_free[slot], hp->d2h);
    return e;
  };

  gs_status result = GS_OK;
  cudaError_t e = upload(0);
  for (int64_t ci = 0; ci < nchunks && e == cudaSuccess; ++ci) {
    const int64_t nc = std::min(ch, n - ci * ch);
    const int slot = (int)(ci & 1);
    // the next chunk's inputs go to the other slot, whose previous solve has returned
    if (ci + 1 < nchunks && (e = upload(ci + 1)) != cudaSuccess) break;
    if ((e = cudaStreamWaitEvent(hp->comp, hp->in_ready[slot], 0)) != cudaSuccess) break;
    if (ci >= 2 && (e = cudaStreamWaitEvent(hp->comp, hp->out_free[slot], 0)) != cudaSuccess) break;
    double* din = hp->in[slot];
    double* dout = hp->out[slot];
    const gs_status cs = solve_grad_in(r, c, nc, din, din + (size_t)P * nc, shared_w, t0, t1, save_t, n_save, rtol,
                                       atol, hp->comp, dout, dout + nc, dout + (size_t)(1 + P) * nc, shared_w_bar,
                                       reinterpret_cast<int32_t*>(dout + (size_t)(1 + P + d) * nc), true);
    if (cs == GS_ERR_TRAJ_FAILED) {
      result = GS_ERR_TRAJ_FAILED;
    } else if (cs != GS_OK) {
      result = cs;
      break;
    }
    if ((e = cudaEventRecord(hp->out_ready[slot], hp->comp)) != cudaSuccess) break;
    if ((e = download(ci)) != cudaSuccess) break;
  }
  const cudaError_t e1 = cudaStreamSynchronize(hp->h2d);
  const cudaError_t e2 = cudaStreamSynchronize(hp->d2h);
  const cudaError_t e3 = cudaStreamSynchronize(hp->comp);
  if (result != GS_OK && result != GS_ERR_TRAJ_FAILED) return result;
  if (e != cudaSuccess || e1 != cudaSuccess || e2 != cudaSuccess || e3 != cudaSuccess) return GS_ERR_CUDA;
  return result;
}

gs_status gs_solve(int problem_id, int64_t n, const double* params, const double* y0, const float* shared_w,
                   double t0, double t1, const double* save_t, int n_save, double rtol, double atol,
                   const gs_options* opt, gs_stream stream, double* y_save_out, double* y_final_out,
                   int32_t* traj_status) {
  Call c;
  gs_status st = check_common(problem_id, n, params, y0, shared_w, t0, t1, save_t, n_save, rtol, atol, opt, &c);
  if (st != GS_OK) return st;
  if (n == 0) return GS_OK;
  if (!traj_status || !y_final_out) return GS_ERR_INVALID_ARG;
  int dev = 0;
  cudaGetDevice(&dev);
  std::lock_guard<std::mutex> lock(g_ws_mu);
  gs_record* r = workspace(dev);
  if (!r) return GS_ERR_OOM;
  if ((st = ensure_counters(r)) != GS_OK) return st;
  if (c.kernel_ms && (st = ensure_events(r)) != GS_OK) return st;
  FwdArgs a;
  std::memset(&a, 0, sizeof(a));
  a.n = n;
  a.params = params;
  a.y0 = y0;
  a.shared_w = shared_w;
  a.t0 = t0;
  a.t1 = t1;
  a.rtol = rtol;
  a.atol = atol;
  a.h0 = c.h0;
  a.control = c.control;
  a.max_steps = c.max_steps;
  a.n_save = n_save;
  if (n_save) std::memcpy(a.save_t, save_t, sizeof(double) * n_save);
  a.y_save = y_save_out;
  a.step_counts = c.step_counts;
  a.k = 0;  // nothing recorded: no arena, no per-trajectory record arrays
  a.segw = 0;
  a.arena_top = &r->ctr->arena_top;
  a.overflow = &r->ctr->overflow;
  a.any_failed = &r->ctr->any_failed;
  a.status = traj_status;
  a.y_final = y_final_out;
  a.work = &r->ctr->work_fwd;
  const cudaStream_t s = (cudaStream_t)stream;
  cudaError_t e = cudaMemsetAsync(r->ctr, 0, sizeof(Counters), s);
  if (e != cudaSuccess) return cuda_fail(e);
  if (c.kernel_ms) cudaEventRecord(r->ev[0], s);
  e = launch_forward_m(c.method, c.problem, c.precision, a, s);
  if (e != cudaSuccess) return GS_ERR_CUDA;
  if (c.kernel_ms) cudaEventRecord(r->ev[1], s);
  e = cudaMemcpyAsync(r->ctr_host, r->ctr, sizeof(Counters), cudaMemcpyDeviceToHost, s);
  if (e != cudaSuccess) return GS_ERR_CUDA;
  if ((st = wait_stream(s, c.timeout_ms)) != GS_OK) return st;
  if (c.kernel_ms) cudaEventElapsedTime(&c.kernel_ms[0], r->ev[0], r->ev[1]);
  return r->ctr_host->any_failed ? GS_ERR_TRAJ_FAILED : GS_OK;
}

gs_status gs_context_create(gs_context** ctx) {
  if (!ctx) return GS_ERR_INVALID_ARG;
  *ctx = nullptr;
  gs_context* c = new (std::nothrow) gs_context();
  if (!c) return GS_ERR_OOM;
  c->ws = new (std::nothrow) gs_record();
  if (!c->ws) {
    delete c;
    return GS_ERR_OOM;
  }
  if (cudaGetDevice(&c->device) != cudaSuccess) {
    delete c->ws;
    delete c;
    return GS_ERR_CUDA;
  }
  *ctx = c;
  return GS_OK;
}

gs_status gs_context_destroy(gs_context* ctx) {
  if (!ctx) return GS_OK;
  destroy(ctx->ws);
  delete ctx;
  return GS_OK;
}

gs_status gs_context_bytes(const gs_context* ctx, size_t* bytes) {
  if (!ctx || !bytes) return GS_ERR_INVALID_ARG;
  *bytes = record_bytes(ctx->ws);
  return GS_OK;
}

gs_status gs_solve_grad_ctx(gs_context* ctx, int problem_id, int64_t n, const double* params, const double* y0,
                            const float* shared_w, double t0, double t1, const double* save_t, int n_save,
                            double rtol, double atol, const gs_options* opt, gs_stream stream, double* loss_out,
                            double* params_bar, double* y0_bar, float* shared_w_bar, int32_t* traj_status) {
  if (!ctx) return GS_ERR_INVALID_ARG;
  Call c;
  gs_status st = check_common(problem_id, n, params, y0, shared_w, t0, t1, save_t, n_save, rtol, atol, opt, &c);
  if (st != GS_OK) return st;
  if (n == 0) return GS_OK;
  if (!traj_status) return GS_ERR_INVALID_ARG;
  int dev = 0;
  cudaGetDevice(&dev);
  if (dev != ctx->device) return GS_ERR_INVALID_ARG;
  std::lock_guard<std::mutex> lock(ctx->mu);
  // contexts record compactly: with stored stages the request server's
  // latencies measured worse (0.8 load, 1000 requests: p50 60 / p99 1015 ms
  // against 43 / 865 ms), the stage records of concurrent small launches
  // costing more than their faster reverse sweeps save
  if (const int64_t ch = solve_chunk(ctx->ws, c, n, n_save, rtol, false))
    return solve_grad_chunked(ctx->ws, c, n, ch, params, y0, t0, t1, save_t, n_save, rtol, atol,
                              (cudaStream_t)stream, loss_out, params_bar, y0_bar, traj_status, false);
  return solve_grad_in(ctx->ws, c, n, params, y0, shared_w, t0, t1, save_t, n_save, rtol, atol,
                       (cudaStream_t)stream, loss_out, params_bar, y0_bar, shared_w_bar, traj_status, false);
}

gs_status gs_record_bytes(const gs_record* rec, size_t* bytes) {
  if (!rec || !bytes) return GS_ERR_INVALID_ARG;
  *bytes = rec->bytes;
  return GS_OK;
}

gs_status gs_record_stats(const gs_record* rec, int64_t* n, int64_t* accepted, int64_t* attempted) {
  if (!rec) return GS_ERR_INVALID_ARG;
  if (n) *n = rec->n;
  if (!accepted && !attempted) return GS_OK;
  std::vector<int32_t> S(rec->n), A(rec->n);
  if (rec->n > 0) {
    if (cudaMemcpy(S.data(), rec->S, rec->n * sizeof(int32_t), cudaMemcpyDeviceToHost) != cudaSuccess ||
        cudaMemcpy(A.data(), rec->natt, rec->n * sizeof(int32_t), cudaMemcpyDeviceToHost) != cudaSuccess)
      return GS_ERR_CUDA;
  }
  int64_t sa = 0, sb = 0;
  for (int64_t i = 0; i < rec->n; ++i) { sa += S[i]; sb += A[i]; }
  if (accepted) *accepted = sa;
  if (attempted) *attempted = sb;
  return GS_OK;
}

gs_status gs_record_export_mesh(const gs_record* rec, int64_t* offsets, double* h) {
  if (!rec || !offsets) return GS_ERR_INVALID_ARG;
  const int64_t n = rec->n;
  std::vector<int32_t> S(n), st(n);
  std::vector<long long> head(n);
  if (n > 0) {
    if (cudaMemcpy(S.data(), rec->S, n * sizeof(int32_t), cudaMemcpyDeviceToHost) != cudaSuccess ||
        cudaMemcpy(head.data(), rec->head, n * sizeof(long long), cudaMemcpyDeviceToHost) != cudaSuccess ||
        cudaMemcpy(st.data(), rec->status, n * sizeof(int32_t), cudaMemcpyDeviceToHost) != cudaSuccess)
      return GS_ERR_CUDA;
  }
  offsets[0] = 0;
  for (int64_t i = 0; i < n; ++i) offsets[i + 1] = offsets[i] + (st[i] == GS_TRAJ_OK ? S[i] : 0);
  if (!h || n == 0) return GS_OK;
  std::vector<double> arena((size_t)rec->arena_cap * rec->segw);
  if (cudaMemcpy(arena.data(), rec->arena, arena.size() * sizeof(double), cudaMemcpyDeviceToHost) != cudaSuccess)
    return GS_ERR_CUDA;
  for (int64_t i = 0; i < n; ++i) {
    if (st[i] != GS_TRAJ_OK) continue;
    // walk segments last to first; the last holds S - (nseg-1) k steps
    const int Sk = S[i];
    int m = Sk - ((Sk - 1) / rec->k) * rec->k;
    long long seg = head[i];
    int64_t end = offsets[i + 1];
    while (seg >= 0) {
      const double* sp = arena.data() + (size_t)seg * rec->segw;
      for (int j = m - 1; j >= 0; --j) h[--end] = sp[2 + rec->d + j];
      long long prev;
      std::memcpy(&prev, sp, sizeof(prev));
      seg = prev;
      m = rec->k;
    }
    if (end != offsets[i]) return GS_ERR_CUDA;  // inconsistent record
  }
  return GS_OK;
}

gs_status gs_record_free(gs_record* rec) {
  if (!pool_put(rec)) destroy(rec);
  return GS_OK;
}

}  // extern "C"
