// C ABI of the batched analyses: plan (shape classes, item table, unit lists, workspace layout, twiddle
// tables), autotuner (CTA sizes of the passes, timed on scratch data of the batch's shapes), and the
// analysis itself, replayed as one CUDA graph.
//
// Items of one grid shape form a class.  A class runs the split passes (k_split.cuh) with one launch per
// pass over the units of its items: forward rows (anomalies and innovations), columns, inverse rows.  The
// kernels take the pointers of an item from a device table, so that new pointers need a new table and no
// new graph.  The classes are issued on kLanes graph branches, largest first, each to the branch with the
// least work.  256 mixed analyses, 32 to 1024 points a side, FP32: 7.9 ms; 12.32 with the 103 analyses of
// at least 512 x 256 points on plans of their own, whose kernels each filled a fraction of the SMs, and the others in
// seven persistent launches whose units were serial over the members; 8.6 to 10.4 (then 8.07) cut into chunks of
// 48 to 160 MB, whose spectra stay in L2.
#include <algorithm>
#include <cmath>
#include <cstring>
#include <map>
#include <string>
#include <utility>
#include <vector>

#include "../../include/fftenkf.h"
#include "common.cuh"

using namespace fftenkf;

namespace fftenkf {
void set_last_error(const std::string& msg);
}  // namespace fftenkf

namespace {
fftenkf_status bfail(fftenkf_status s, const std::string& m) {
  set_last_error(m);
  return s;
}
size_t rup(size_t x, size_t a) { return (x + a - 1) / a * a; }
constexpr int kLanes = 8;
constexpr int kBatchPasses = 7;   // reported passes: mean, anomaly rows, statistics, gain, innovation rows, update, inverse rows
enum Stage { kRows, kCols, kInv, kStages };
// the stage that a reported pass is part of
Stage stage_of(int pass) { return (pass == 1 || pass == 4) ? kRows : (pass == 6) ? kInv : kCols; }
const int kCandBt[2] = {256, 128};

bool batch_line(int n) { return n >= 16 && n <= 1024 && line_supported(n) && row_line_supported(n); }

struct ShapeClass {
  int ny, nx, n_max;            // shape, largest member count
  double cost;
  int first[kStages], units[kStages];   // its units in the unit list of the batch
};
}  // namespace

struct fftenkf_batch_s {
  int count = 0, storage = 0;
  std::vector<fftenkf_dims> dims;
  std::vector<SplitItem> items;        // host copy (pointers of the last bound call)
  std::vector<size_t> off_A, off_W;    // workspace regions
  std::vector<ShapeClass> shapes;           // largest first
  SplitItem* d_items = nullptr;
  uint2* d_units = nullptr;
  float2* d_tw = nullptr;
  std::map<std::pair<int, int>, size_t> off_tw;   // (line length, V) -> stage twiddles
  std::map<int, size_t> off_x;                    // nx -> real-FFT twiddles
  int* d_status = nullptr;
  size_t ws_bytes = 0;
  void* own_ws = nullptr;
  int bt[kStages] = {256, 256, 256};
  cudaStream_t lane[kLanes] = {};
  cudaEvent_t ev_fork = nullptr, ev_lane[kLanes] = {};
  cudaEvent_t ev_read = nullptr;       // after the last launch that reads the item table
  cudaStream_t cap = nullptr;
  cudaGraphExec_t exec = nullptr;
  char* bound_ws = nullptr;
  bool items_dirty = true;             // the device table does not hold `items`
};

// The host's item table to the device, ordered on s and after the last analysis, which may be running on
// another stream and reads the table.  (The copy is pageable: the runtime stages the host table before
// it returns.)
static cudaError_t upload_items(fftenkf_batch b, cudaStream_t s) {
  cudaError_t e = cudaStreamWaitEvent(s, b->ev_read, 0);
  if (e == cudaSuccess)
    e = cudaMemcpyAsync(b->d_items, b->items.data(), b->count * sizeof(SplitItem), cudaMemcpyHostToDevice, s);
  return e;
}

static SplitParams class_params(fftenkf_batch b, const ShapeClass& c) {
  SplitParams q;
  memset(&q, 0, sizeof(q));
  q.ny = c.ny; q.nx = c.nx; q.L = c.nx / 2; q.M = 1; q.n_obs = 1; q.storage = b->storage;
  q.table = b->d_items;
  q.anomalies = 1;
  q.innovations = kInnovation;
  q.twL = b->d_tw + b->off_tw[{q.L, split_row_V(q.L)}];
  q.twX = b->d_tw + b->off_x[c.nx];
  q.twY = b->d_tw + b->off_tw[{c.ny, plan_V(c.ny, split_col_sel(c.ny, false))}];
  q.inv_G = (float)(1.0 / ((double)c.ny * (double)c.nx));
  q.status = b->d_status;
  return q;
}

static cudaError_t run_stage(fftenkf_batch b, const ShapeClass& c, int stage, cudaStream_t s) {
  SplitParams q = class_params(b, c);
  q.units = b->d_units + c.first[stage];
  q.n_units = c.units[stage];
  q.threads = b->bt[stage];
  if (stage == kRows) return launch_row_split(q, s);
  if (stage == kInv) return launch_row_inv_split(q, s);
  q.groups = split_col_groups(c.ny, 1, 1, c.n_max, q.threads);
  return launch_col_split(q, s);
}

// The whole batch on stream s: the classes on the lanes, forked from s and joined back.
static fftenkf_status run_all(fftenkf_batch b, cudaStream_t s) {
  const int lanes = std::min((int)b->shapes.size(), kLanes);
  cudaError_t e = cudaEventRecord(b->ev_fork, s);
  double load[kLanes] = {};
  for (int l = 0; l < lanes && e == cudaSuccess; ++l) e = cudaStreamWaitEvent(b->lane[l], b->ev_fork, 0);
  for (const ShapeClass& c : b->shapes) {
    int l = 0;
    for (int q = 1; q < lanes; ++q)
      if (load[q] < load[l]) l = q;
    load[l] += c.cost;
    for (int stage = 0; stage < kStages && e == cudaSuccess; ++stage) e = run_stage(b, c, stage, b->lane[l]);
  }
  for (int l = 0; l < lanes && e == cudaSuccess; ++l) {
    e = cudaEventRecord(b->ev_lane[l], b->lane[l]);
    if (e == cudaSuccess) e = cudaStreamWaitEvent(s, b->ev_lane[l], 0);
  }
  return e == cudaSuccess ? FFTENKF_OK : bfail(FFTENKF_ECUDA, std::string("batched passes: ") + cudaGetErrorString(e));
}

// Classes, unit lists (uploaded) and the workspace layout.
static cudaError_t build_units(fftenkf_batch b) {
  std::map<std::pair<int, int>, std::vector<int>> classes;
  for (int i = 0; i < b->count; ++i) classes[{b->dims[i].ny, b->dims[i].nx}].push_back(i);
  std::vector<uint2> units;
  auto add_class = [&](int ny, int nx, const std::vector<int>& ids) {
    ShapeClass c{};
    c.ny = ny;
    c.nx = nx;
    const unsigned tiles = (unsigned)(ny / split_row_tile(nx / 2));
    for (int i : ids) {
      c.n_max = std::max(c.n_max, b->dims[i].n_members);
      c.cost += (double)b->dims[i].n_members * ny * nx;
    }
    for (int stage = 0; stage < kStages; ++stage) {
      c.first[stage] = (int)units.size();
      for (int i : ids) {
        const unsigned N = (unsigned)b->dims[i].n_members;
        const unsigned n = stage == kRows ? 2 * N * tiles : stage == kInv ? N * tiles : (unsigned)(nx / 2 + 1);
        for (unsigned u = 0; u < n; ++u) units.push_back(make_uint2((unsigned)i, u));
      }
      c.units[stage] = (int)units.size() - c.first[stage];
    }
    b->shapes.push_back(c);
  };
  for (const auto& cl : classes) add_class(cl.first.first, cl.first.second, cl.second);
  std::stable_sort(b->shapes.begin(), b->shapes.end(), [](const ShapeClass& x, const ShapeClass& y) { return x.cost > y.cost; });
  cudaError_t e = cudaMalloc(&b->d_units, units.size() * sizeof(uint2));
  if (e == cudaSuccess) e = cudaMemcpy(b->d_units, units.data(), units.size() * sizeof(uint2), cudaMemcpyHostToDevice);
  return e;
}

extern "C" fftenkf_status fftenkf_plan_batched(fftenkf_batch* out, int count, const fftenkf_dims* dims) {
  set_last_error("");
  if (!out || !dims || count <= 0) return bfail(FFTENKF_EINVAL, "null argument or empty batch");
  *out = nullptr;
  const int storage = dims[0].storage;
  for (int i = 0; i < count; ++i) {
    const fftenkf_dims& d = dims[i];
    if (d.n_blocks != 1) return bfail(FFTENKF_EUNSUPPORTED, "batched analyses have one (observed) block each");
    if (d.storage != storage) return bfail(FFTENKF_EINVAL, "all batched analyses share one storage type");
    if (d.storage != FFTENKF_F32 && d.storage != FFTENKF_BF16) return bfail(FFTENKF_EINVAL, "unknown storage");
    if (d.n_members < 2) return bfail(FFTENKF_EUNSUPPORTED, "need at least 2 members");
    if (d.nx % 2 || !batch_line(d.nx / 2) || !batch_line(d.ny))
      return bfail(FFTENKF_EUNSUPPORTED, "batched sizes: ny and nx/2 in {2^a, 3*2^a} between 16 and 1024");
  }
  fftenkf_batch b = new fftenkf_batch_s();
  b->count = count;
  b->storage = storage;
  b->dims.assign(dims, dims + count);
  b->items.resize(count);
  // twiddle tables, one per distinct line plan
  std::vector<float2> tw;
  auto root = [&](long long e, long long n) {
    const double ang = 2.0 * M_PI * (double)e / (double)n;
    tw.push_back(make_float2((float)std::cos(ang), (float)-std::sin(ang)));
  };
  auto stage_table = [&](int n, int V) {
    if (b->off_tw.count({n, V})) return;
    b->off_tw[{n, V}] = tw.size();
    for (int i = 0; i < twiddle_count(n, V); ++i) root(twiddle_exponent(n, V, i), n);
    if (tw.size() % 2) tw.push_back(make_float2(0.f, 0.f));
  };
  size_t off = 0;
  b->off_A.resize(count);
  b->off_W.resize(count);
  for (int i = 0; i < count; ++i) {
    const int ny = dims[i].ny, nx = dims[i].nx, L = nx / 2, N = dims[i].n_members;
    stage_table(L, split_row_V(L));
    stage_table(ny, plan_V(ny, split_col_sel(ny, false)));
    if (!b->off_x.count(nx)) {
      b->off_x[nx] = tw.size();
      for (int k = 0; k <= L; ++k) root(k, nx);
      if (tw.size() % 2) tw.push_back(make_float2(0.f, 0.f));
    }
    SplitItem& it = b->items[i];
    memset(&it, 0, sizeof(it));
    it.N = N;
    it.inv_sqrt_N = (float)(1.0 / std::sqrt((double)N));
    it.scale = (float)(1.0 / ((double)(N - 1) * (double)ny * (double)nx));
    const size_t lines = (size_t)N * L * ny * sizeof(float2);
    b->off_A[i] = off; off = rup(off + lines, 256);
    b->off_W[i] = off; off = rup(off + lines, 256);
  }
  b->ws_bytes = off;
  cudaError_t e = cudaMalloc(&b->d_tw, tw.size() * sizeof(float2));
  if (e == cudaSuccess) e = cudaMemcpy(b->d_tw, tw.data(), tw.size() * sizeof(float2), cudaMemcpyHostToDevice);
  if (e == cudaSuccess) e = cudaMalloc(&b->d_status, sizeof(int));
  if (e == cudaSuccess) e = cudaMemset(b->d_status, 0, sizeof(int));
  if (e == cudaSuccess) e = cudaMalloc(&b->d_items, count * sizeof(SplitItem));
  if (e == cudaSuccess) e = build_units(b);
  if (e == cudaSuccess) e = cudaStreamCreateWithFlags(&b->cap, cudaStreamNonBlocking);
  if (e == cudaSuccess) e = cudaEventCreateWithFlags(&b->ev_fork, cudaEventDisableTiming);
  if (e == cudaSuccess) e = cudaEventCreateWithFlags(&b->ev_read, cudaEventDisableTiming);
  for (int l = 0; l < kLanes && e == cudaSuccess; ++l) {
    e = cudaStreamCreateWithFlags(&b->lane[l], cudaStreamNonBlocking);
    if (e == cudaSuccess) e = cudaEventCreateWithFlags(&b->ev_lane[l], cudaEventDisableTiming);
  }
  if (e != cudaSuccess) {
    fftenkf_batch_destroy(b);
    return bfail(FFTENKF_ENOMEM, "batched plan allocation failed");
  }
  *out = b;
  return FFTENKF_OK;
}

extern "C" fftenkf_status fftenkf_batch_destroy(fftenkf_batch b) {
  if (!b) return FFTENKF_OK;
  if (b->exec) cudaGraphExecDestroy(b->exec);
  if (b->cap) cudaStreamDestroy(b->cap);
  for (int l = 0; l < kLanes; ++l) {
    if (b->lane[l]) cudaStreamDestroy(b->lane[l]);
    if (b->ev_lane[l]) cudaEventDestroy(b->ev_lane[l]);
  }
  if (b->ev_fork) cudaEventDestroy(b->ev_fork);
  if (b->ev_read) cudaEventDestroy(b->ev_read);
  if (b->d_units) cudaFree(b->d_units);
  if (b->d_items) cudaFree(b->d_items);
  if (b->d_tw) cudaFree(b->d_tw);
  if (b->d_status) cudaFree(b->d_status);
  if (b->own_ws) cudaFree(b->own_ws);
  delete b;
  return FFTENKF_OK;
}

extern "C" fftenkf_status fftenkf_batch_workspace_size(fftenkf_batch b, size_t* bytes) {
  if (!b || !bytes) return bfail(FFTENKF_EINVAL, "null argument");
  *bytes = b->ws_bytes;
  return FFTENKF_OK;
}

static fftenkf_status bind(fftenkf_batch b, void* const* ens, const float* const* data, const void* const* pert,
                           const double* const* rhat, char* ws) {
  for (int i = 0; i < b->count; ++i) {
    if (!ens[i] || !data[i] || !pert[i] || !rhat[i]) return bfail(FFTENKF_EINVAL, "null item pointer");
    if (((uintptr_t)ens[i] | (uintptr_t)data[i] | (uintptr_t)pert[i] | (uintptr_t)rhat[i]) % 16)
      return bfail(FFTENKF_EINVAL, "item pointers must be 16-byte aligned");
  }
  bool changed = (ws != b->bound_ws);
  for (int i = 0; i < b->count; ++i) {
    SplitItem& it = b->items[i];
    changed |= it.ens != ens[i] || it.data != data[i] || it.pert != pert[i] || it.rhat != rhat[i];
    it.ens = ens[i];
    it.data = data[i];
    it.pert = pert[i];
    it.rhat = rhat[i];
    it.A = reinterpret_cast<float2*>(ws + b->off_A[i]);
    it.W = reinterpret_cast<float2*>(ws + b->off_W[i]);
  }
  b->bound_ws = ws;
  b->items_dirty |= changed;
  return FFTENKF_OK;
}

static fftenkf_status batch_ws(fftenkf_batch b, void* workspace, char** ws) {
  if (workspace) {
    if ((uintptr_t)workspace % 256) return bfail(FFTENKF_EINVAL, "workspace must be 256-byte aligned");
    *ws = static_cast<char*>(workspace);
    return FFTENKF_OK;
  }
  if (!b->own_ws && cudaMalloc(&b->own_ws, b->ws_bytes) != cudaSuccess) {
    b->own_ws = nullptr;
    return bfail(FFTENKF_ENOMEM, "workspace allocation failed");
  }
  *ws = static_cast<char*>(b->own_ws);
  return FFTENKF_OK;
}

extern "C" fftenkf_status fftenkf_analyze_batched(fftenkf_batch b, void* const* ensembles, const float* const* data,
                                                  const void* const* perturbations, const double* const* rhat,
                                                  void* workspace, void* stream) {
  set_last_error("");
  if (!b || !ensembles || !data || !perturbations || !rhat) return bfail(FFTENKF_EINVAL, "null argument");
  char* ws;
  fftenkf_status st = batch_ws(b, workspace, &ws);
  if (st != FFTENKF_OK) return st;
  st = bind(b, ensembles, data, perturbations, rhat, ws);
  if (st != FFTENKF_OK) return st;
  cudaStream_t s = static_cast<cudaStream_t>(stream);
  cudaError_t e = cudaSuccess;
  if (b->items_dirty) {
    e = upload_items(b, s);
    if (e != cudaSuccess) return bfail(FFTENKF_ECUDA, std::string("item table: ") + cudaGetErrorString(e));
  }
  if (!b->exec) {
    cudaGraph_t g = nullptr;
    e = cudaStreamBeginCapture(b->cap, cudaStreamCaptureModeThreadLocal);
    fftenkf_status rs = FFTENKF_OK;
    std::string rmsg;
    if (e == cudaSuccess) {
      rs = run_all(b, b->cap);
      if (rs != FFTENKF_OK) rmsg = fftenkf_last_error();
      e = cudaStreamEndCapture(b->cap, &g);
    }
    if (rs != FFTENKF_OK) {
      if (g) cudaGraphDestroy(g);
      return bfail(rs, "graph capture: " + rmsg);
    }
    if (e == cudaSuccess) e = cudaGraphInstantiate(&b->exec, g, 0);
    if (g) cudaGraphDestroy(g);
    if (e != cudaSuccess) {
      b->exec = nullptr;
      return bfail(FFTENKF_ECUDA, std::string("graph capture: ") + cudaGetErrorString(e));
    }
  }
  e = cudaGraphLaunch(b->exec, s);
  if (e == cudaSuccess) e = cudaEventRecord(b->ev_read, s);
  if (e != cudaSuccess) return bfail(FFTENKF_ECUDA, std::string("graph launch: ") + cudaGetErrorString(e));
  b->items_dirty = false;   // only now: the copy of a call that was refused (s under capture) has not run
  return FFTENKF_OK;
}

// Time the CTA sizes of every stage on scratch inputs of the batch's shapes, the classes one after another, and
// keep the fastest.  The fields are zero; rhat is positive (the byte 0x3f repeated, 4.8e-4): with rhat = 0 every
// denominator would vanish and take the column pass's FP64 branch, which real inputs do not (8 analyses of
// 1024^2, N=5: 0.497 ms instead of 0.487).  Allocates the scratch inputs (one ensemble's worth per item) for the
// duration of the call.
extern "C" fftenkf_status fftenkf_batch_autotune(fftenkf_batch b, void* workspace, void* stream, double* best_ms) {
  set_last_error("");
  if (!b) return bfail(FFTENKF_EINVAL, "null argument");
  char* ws;
  fftenkf_status st = batch_ws(b, workspace, &ws);
  if (st != FFTENKF_OK) return st;
  cudaStream_t s = static_cast<cudaStream_t>(stream);
  const int es = b->storage == FFTENKF_BF16 ? 2 : 4;
  size_t bytes = 0;
  std::vector<size_t> oe(b->count), od(b->count), op(b->count), orh(b->count);
  for (int i = 0; i < b->count; ++i) {
    const fftenkf_dims& d = b->dims[i];
    const size_t G = (size_t)d.ny * d.nx;
    oe[i] = bytes; bytes = rup(bytes + d.n_members * G * es, 256);
    od[i] = bytes; bytes = rup(bytes + G * 4, 256);
    op[i] = bytes; bytes = rup(bytes + d.n_members * G * es, 256);
  }
  const size_t field_bytes = bytes;
  for (int i = 0; i < b->count; ++i) {
    orh[i] = bytes;
    bytes = rup(bytes + (size_t)b->dims[i].ny * (b->dims[i].nx / 2 + 1) * 8, 256);
  }
  char* scratch = nullptr;
  if (cudaMalloc(&scratch, bytes) != cudaSuccess) return bfail(FFTENKF_ENOMEM, "autotune scratch allocation failed");
  cudaMemsetAsync(scratch, 0, field_bytes, s);
  cudaMemsetAsync(scratch + field_bytes, 0x3f, bytes - field_bytes, s);
  std::vector<void*> ens(b->count), pert(b->count);
  std::vector<const float*> dat(b->count);
  std::vector<const double*> rh(b->count);
  for (int i = 0; i < b->count; ++i) {
    ens[i] = scratch + oe[i];
    dat[i] = reinterpret_cast<const float*>(scratch + od[i]);
    pert[i] = scratch + op[i];
    rh[i] = reinterpret_cast<const double*>(scratch + orh[i]);
  }
  std::vector<SplitItem> saved = b->items;
  char* saved_ws = b->bound_ws;
  bind(b, ens.data(), dat.data(), pert.data(), rh.data(), ws);
  cudaError_t e = upload_items(b, s);
  cudaEvent_t e0, e1;
  cudaEventCreate(&e0);
  cudaEventCreate(&e1);
  double total = 0.0;
  for (int stage = 0; stage < kStages && e == cudaSuccess; ++stage) {
    float best = 1e30f;
    int keep = kCandBt[0];
    for (int bt : kCandBt) {
      b->bt[stage] = bt;
      float ms = 0.f;
      for (int rep = 0; rep < 3 && e == cudaSuccess; ++rep) {   // first repetition warms up
        cudaEventRecord(e0, s);
        for (const ShapeClass& c : b->shapes)
          if (e == cudaSuccess) e = run_stage(b, c, stage, s);
        cudaEventRecord(e1, s);
        cudaEventSynchronize(e1);
        float t = 0.f;
        cudaEventElapsedTime(&t, e0, e1);
        if (rep) ms += t;
      }
      if (ms < best) {
        best = ms;
        keep = bt;
      }
    }
    b->bt[stage] = keep;
    total += best / 2.0;
  }
  cudaEventDestroy(e0);
  cudaEventDestroy(e1);
  const cudaError_t se = cudaStreamSynchronize(s);
  if (e == cudaSuccess) e = se;
  cudaMemset(b->d_status, 0, sizeof(int));
  cudaFree(scratch);
  b->items = saved;
  b->bound_ws = saved_ws;
  b->items_dirty = true;
  if (b->exec) {
    cudaGraphExecDestroy(b->exec);
    b->exec = nullptr;
  }
  if (best_ms) *best_ms = total;
  if (e != cudaSuccess) return bfail(FFTENKF_ECUDA, std::string("autotune: ") + cudaGetErrorString(e));
  return FFTENKF_OK;
}

extern "C" fftenkf_status fftenkf_batch_schedule(fftenkf_batch b, int* cta_threads, int* sched, int n) {
  if (!b || !cta_threads || !sched) return bfail(FFTENKF_EINVAL, "null argument");
  for (int p = 0; p < kBatchPasses && p < n; ++p) {
    cta_threads[p] = b->bt[stage_of(p)];
    sched[p] = 0;   // one line plan per length
  }
  return FFTENKF_OK;
}

extern "C" fftenkf_status fftenkf_batch_last_device_status(fftenkf_batch b, void* stream) {
  if (!b) return bfail(FFTENKF_EINVAL, "null argument");
  cudaError_t e = cudaStreamSynchronize(static_cast<cudaStream_t>(stream));
  if (e != cudaSuccess) return bfail(FFTENKF_ECUDA, std::string("stream: ") + cudaGetErrorString(e));
  int word = 0;
  e = cudaMemcpy(&word, b->d_status, sizeof(int), cudaMemcpyDeviceToHost);
  if (e == cudaSuccess) e = cudaMemset(b->d_status, 0, sizeof(int));
  if (e != cudaSuccess) return bfail(FFTENKF_ECUDA, std::string("status word: ") + cudaGetErrorString(e));
  if (word & kStatusNonFinite) return bfail(FFTENKF_ENONFINITE, "non-finite spectral covariance");
  return FFTENKF_OK;
}
