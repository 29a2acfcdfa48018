// libbege C ABI: contexts, handles, memory accounting and job bookkeeping.
// The arithmetic of the search lives in the .cu files; this file validates
// arguments, owns device memory and enqueues the kernels.
#include <cuda_runtime.h>

#include <algorithm>
#include <atomic>
#include <cmath>
#include <cstdint>
#include <cstdio>
#include <cstring>
#include <map>
#include <memory>
#include <mutex>
#include <string>
#include <vector>

#include "bege_batch.h"
#include "bege_internal.h"

namespace {

thread_local std::string g_last_error;

int fail(int code, const std::string& msg) {
  g_last_error = msg;
  return code;
}

int cuda_fail(cudaError_t e, const char* where) {
  return fail(BEGE_ECUDA, std::string(where) + ": " + cudaGetErrorString(e));
}

bool is_pow2(int64_t n) { return n > 0 && (n & (n - 1)) == 0; }

// Restores the caller's current device on scope exit.
struct DeviceGuard {
  int prev = -1;
  bool ok = false;
  explicit DeviceGuard(int dev) {
    if (cudaGetDevice(&prev) != cudaSuccess) prev = -1;
    ok = cudaSetDevice(dev) == cudaSuccess;
  }
  ~DeviceGuard() {
    if (prev >= 0) cudaSetDevice(prev);
  }
};

struct DevBuf {
  void* ptr = nullptr;
  size_t bytes = 0;
};

}  // namespace

namespace bege {
int set_last_error(int code, const std::string& msg) { return fail(code, msg); }
}  // namespace bege

struct PlanHost {
  bege::Geometry g{};
  bege::PlanDev dev{};
  DevBuf tables;
};

struct Segment {
  int64_t n = 0;
  int32_t channel = 0;
  DevBuf D, AB;
  std::shared_ptr<PlanHost> plan;
  bool loaded = false;  // its kernel is known to have finished
};

struct Bank {
  int64_t count = 0, L = 0, Lp = 0;
  DevBuf w;
  bool large = false;  // holds a sample above bege::kLargeSample
};

// What a job needs beside its segment and bank; kept by the context between
// jobs (events included: creating three costs more than a small launch).
struct JobBuffers {
  DevBuf sigma, recs, counter;
  DevBuf exch;  // exchange buffer of the job's correlate kernel (may be absent)
  int64_t sigma_cap = 0;
  uint64_t rec_cap = 0;
  cudaEvent_t done = nullptr;
  cudaEvent_t k_start = nullptr, k_stop = nullptr;  // around the correlate kernel
};

struct Job {
  int32_t seg = -1, bank = -1;
  int64_t k0 = 0, k1 = 0;
  float kappa = 0.f;
  std::unique_ptr<JobBuffers> buf;
  DevBuf proj;        // per-lag maximum over the bank (bege_correlate_max), n_proj words
  int64_t n_proj = 0;
  DevBuf scratch;     // bege_correlate_multi: the group's template-spectrum scratch
  bool counted = false;             // the finished job's counter has been read into
  unsigned long long count[2] = {};  // {tail count, status}
};

struct BatchEntryHost {
  int64_t n = 0;
  int32_t bank = -1;
  int64_t k0 = 0, k1 = 0;
  float kappa = 0.f;
  bool large = false;  // of its bank
};

struct Batch {
  std::vector<BatchEntryHost> entries;
  std::vector<bege::BatchSeg> segs_host;
  DevBuf y, D, AB, segs, items, jobs, queue, sigma, recs, counters;
  std::vector<size_t> sigma_off;  // per entry, in floats
  uint64_t cap = 0;               // tail records per entry
  int n_items = 0, n_jobs = 0;
  int32_t plan = 0, order = 0;
  int64_t chunk = 256;
  bege::BatchArgs args{};
  cudaStream_t cs = nullptr;      // capture stream
  cudaGraph_t graph = nullptr;
  cudaGraphExec_t exec = nullptr;
  cudaEvent_t done = nullptr, t0 = nullptr, t1 = nullptr;
  bool ran = false;
};

struct bege_ctx {
  int device = 0;
  int sms = 0;
  bege_config cfg{};
  std::mutex mu;
  uint64_t bytes = 0;
  int32_t next_id = 1;
  std::map<int64_t, std::shared_ptr<PlanHost>> plans;  // by N
  std::map<int32_t, std::unique_ptr<Segment>> segs;
  std::map<int32_t, std::unique_ptr<Bank>> banks;
  std::map<int32_t, std::unique_ptr<Job>> jobs;
  std::map<int32_t, std::unique_ptr<Batch>> batches;
  std::vector<std::unique_ptr<JobBuffers>> pool;
  std::map<int64_t, bege::CorrConfig> configs;  // chosen launch shape per N

  // Segment buffers (spectrum, coefficients, staged strain) of released
  // segments, all idle, for the next segment of that length: cudaMalloc and
  // cudaFree of these few buffers took 10 us of a small search, and 100 us
  // where the driver gave back and fetched a whole block each time.  At most
  // kSpareBytes, and given back whenever an allocation would not fit.
  static constexpr uint64_t kSpareBytes = 4u << 20;
  std::vector<DevBuf> spare;
  uint64_t spare_bytes = 0;

  int alloc(DevBuf* b, size_t bytes) {
    if (cfg.hbm_budget_bytes && this->bytes + bytes > cfg.hbm_budget_bytes) drop_spare();
    if (cfg.hbm_budget_bytes && this->bytes + bytes > cfg.hbm_budget_bytes)
      return fail(BEGE_EBUDGET, "device allocation of " + std::to_string(bytes) +
                                    " bytes exceeds the HBM budget");
    void* p = nullptr;
    cudaError_t e = cudaMalloc(&p, bytes ? bytes : 16);
    if (e != cudaSuccess) {
      cudaGetLastError();
      drop_spare();
      e = cudaMalloc(&p, bytes ? bytes : 16);
    }
    if (e != cudaSuccess) {
      cudaGetLastError();
      return fail(BEGE_ENOMEM, std::string("cudaMalloc: ") + cudaGetErrorString(e));
    }
    b->ptr = p;
    b->bytes = bytes;
    this->bytes += bytes;
    return BEGE_OK;
  }
  void release(DevBuf* b) {
    if (b->ptr) {
      exchange_refused = SIZE_MAX;
      cudaFree(b->ptr);
      bytes -= b->bytes;
    }
    b->ptr = nullptr;
    b->bytes = 0;
  }
  // As alloc and release, by way of the spare buffers.  keep: no work that
  // uses the buffer is unfinished.
  int take(DevBuf* b, size_t bytes) {
    for (size_t i = 0; i < spare.size(); ++i) {
      if (spare[i].bytes == bytes) {
        *b = spare[i];
        spare[i] = spare.back();
        spare.pop_back();
        spare_bytes -= bytes;
        return BEGE_OK;
      }
    }
    return alloc(b, bytes);
  }
  void keep(DevBuf* b) {
    if (!b->ptr || spare_bytes + b->bytes > kSpareBytes) {
      release(b);
      return;
    }
    spare_bytes += b->bytes;
    spare.push_back(*b);
    *b = DevBuf{};
  }
  // Exchange buffers of the correlate kernel (at most 40 MB each) belong to a
  // job from its launch to its release and are idle between jobs, for
  // whichever comes next: as many exist as jobs were ever held at once, at
  // most kExchangeBytes in all, and idle ones are given back with the spare
  // buffers.  A size that the device refused is not asked for again before
  // the context has given memory back.
  static constexpr uint64_t kExchangeBytes = 160u << 20;
  std::vector<DevBuf> idle_exchange;
  uint64_t exchange_bytes = 0;  // idle and in use
  size_t exchange_refused = SIZE_MAX;
  void drop_exchange(DevBuf* b) {
    exchange_bytes -= b->bytes;
    release(b);
  }
  // b: of a job not launched yet, on stream s.  Null under capture: the
  // allocation would end it, and its graph may run after the job's release.
  float4* take_exchange(JobBuffers* b, size_t need, cudaStream_t s) {
    if (need == 0 || cfg.hbm_budget_bytes) return nullptr;
    cudaStreamCaptureStatus capture = cudaStreamCaptureStatusNone;
    if (cudaStreamIsCapturing(s, &capture) != cudaSuccess) {
      cudaGetLastError();
      return nullptr;
    }
    if (capture != cudaStreamCaptureStatusNone) return nullptr;
    auto best = idle_exchange.end();
    uint64_t idle = 0;
    for (auto i = idle_exchange.begin(); i != idle_exchange.end(); ++i) {
      idle += i->bytes;
      if (i->bytes >= need && (best == idle_exchange.end() || i->bytes < best->bytes)) best = i;
    }
    if (best != idle_exchange.end()) {
      b->exch = *best;
      idle_exchange.erase(best);
    } else {
      if (need >= exchange_refused || exchange_bytes - idle + need > kExchangeBytes) return nullptr;
      while (exchange_bytes + need > kExchangeBytes) {  // the idle ones are too small
        drop_exchange(&idle_exchange.back());
        idle_exchange.pop_back();
      }
      void* p = nullptr;
      if (cudaMalloc(&p, need) != cudaSuccess) {
        cudaGetLastError();
        exchange_refused = need;
        return nullptr;
      }
      b->exch = {p, need};
      this->bytes += need;
      exchange_bytes += need;
    }
    return static_cast<float4*>(b->exch.ptr);
  }
  // b: of a finished job
  void give_back(std::unique_ptr<JobBuffers> b) {
    if (b->exch.ptr) idle_exchange.push_back(b->exch);
    b->exch = DevBuf{};
    pool.push_back(std::move(b));
  }
  void drop_spare() {
    for (DevBuf& b : idle_exchange) drop_exchange(&b);
    idle_exchange.clear();
    for (DevBuf& b : spare) release(&b);
    spare.clear();
    spare_bytes = 0;
  }
  void free_buffers(JobBuffers* b) {
    release(&b->sigma);
    release(&b->recs);
    release(&b->counter);
    drop_exchange(&b->exch);
    for (cudaEvent_t e : {b->done, b->k_start, b->k_stop})
      if (e) cudaEventDestroy(e);
    b->done = b->k_start = b->k_stop = nullptr;
  }
};

namespace {

int get_plan(bege_ctx* ctx, int64_t n, std::shared_ptr<PlanHost>* out) {
  auto it = ctx->plans.find(n);
  if (it != ctx->plans.end()) {
    *out = it->second;
    return BEGE_OK;
  }
  auto p = std::make_shared<PlanHost>();
  p->g = bege::make_geometry(n);
  const bege::Geometry& g = p->g;
  int rc = ctx->alloc(&p->tables, (size_t)bege::plan_floats2(g) * sizeof(float2));
  if (rc) return rc;
  float2* const base = static_cast<float2*>(p->tables.ptr);
  cudaError_t e = bege::launch_plan_tables(g, base, nullptr);
  if (e == cudaSuccess) e = cudaStreamSynchronize(nullptr);  // read by kernels of any stream
  if (e != cudaSuccess) {
    ctx->release(&p->tables);
    return cuda_fail(e, "plan tables");
  }
  p->dev = bege::plan_at(g, base);
  ctx->plans[n] = p;
  *out = p;
  return BEGE_OK;
}

// Fixed-point representation of x mod 1 in units of 2^-64 cycles.
unsigned long long frac_to_u64(double x) {
  x -= std::floor(x);
  const double s = std::ldexp(x, 32);
  double hi = std::floor(s);
  const double rem = s - hi;
  double lo = std::nearbyint(std::ldexp(rem, 32));
  if (lo >= 4294967296.0) {
    lo -= 4294967296.0;
    hi += 1.0;
  }
  const unsigned long long h = (unsigned long long)hi & 0xffffffffull;
  return (h << 32) + (unsigned long long)lo;
}

int segment_common(bege_ctx* ctx, const float* y_dev, int64_t n, int32_t channel,
                   cudaStream_t s, int32_t* seg_id) {
  std::shared_ptr<PlanHost> plan;
  int rc = get_plan(ctx, n, &plan);
  if (rc) return rc;
  auto seg = std::make_unique<Segment>();
  seg->n = n;
  seg->channel = channel;
  seg->plan = plan;
  const bege::Geometry& g = plan->g;
  rc = ctx->take(&seg->D, (size_t)(g.H + 1) * sizeof(float2));
  if (rc) return rc;
  rc = ctx->take(&seg->AB, (size_t)g.H * sizeof(float4));
  if (rc) {
    ctx->keep(&seg->D);
    return rc;
  }
  cudaError_t e = bege::launch_segment(plan->dev, y_dev, static_cast<float2*>(seg->D.ptr),
                                       static_cast<float4*>(seg->AB.ptr), ctx->cfg.precision != 0, s);
  if (e != cudaSuccess) {
    ctx->release(&seg->D);
    ctx->release(&seg->AB);
    return cuda_fail(e, "segment kernel");
  }
  const int32_t id = ctx->next_id++;
  ctx->segs[id] = std::move(seg);
  *seg_id = id;
  return BEGE_OK;
}

int take_job_buffers(bege_ctx* ctx, int64_t nsig, uint64_t cap, std::unique_ptr<JobBuffers>* out) {
  for (size_t i = 0; i < ctx->pool.size(); ++i) {
    if (ctx->pool[i]->sigma_cap >= nsig && ctx->pool[i]->rec_cap >= cap) {
      *out = std::move(ctx->pool[i]);
      ctx->pool.erase(ctx->pool.begin() + i);
      return BEGE_OK;
    }
  }
  auto b = std::make_unique<JobBuffers>();
  int rc = ctx->alloc(&b->sigma, (size_t)nsig * sizeof(float));
  if (rc) return rc;
  rc = ctx->alloc(&b->recs, (size_t)cap * sizeof(bege_tail));
  if (rc) {
    ctx->release(&b->sigma);
    return rc;
  }
  rc = ctx->alloc(&b->counter, 16);  // u64 tail count, u32 status
  if (rc) {
    ctx->release(&b->sigma);
    ctx->release(&b->recs);
    return rc;
  }
  cudaError_t e = cudaEventCreateWithFlags(&b->done, cudaEventDisableTiming);
  if (e == cudaSuccess) e = cudaEventCreate(&b->k_start);
  if (e == cudaSuccess) e = cudaEventCreate(&b->k_stop);
  if (e != cudaSuccess) {
    ctx->free_buffers(b.get());
    return cuda_fail(e, "job events");
  }
  b->sigma_cap = nsig;
  b->rec_cap = cap;
  *out = std::move(b);
  return BEGE_OK;
}

// Waits for a job; its {tail count, status} (read from the device once).
int wait_counted(Job* j) {
  cudaError_t e = cudaEventSynchronize(j->buf->done);
  if (e != cudaSuccess) return cuda_fail(e, "job");
  if (!j->counted) {
    e = cudaMemcpy(j->count, j->buf->counter.ptr, 16, cudaMemcpyDeviceToHost);
    if (e != cudaSuccess) return cuda_fail(e, "tail count");
    j->counted = true;
  }
  if (j->count[1] & 0xffffffffull)
    return fail(BEGE_ETIMEDOUT, "a bounded device wait gave up; results of this job are invalid");
  return BEGE_OK;
}

// Waits for a job that is let go.  The event of one enqueued under capture
// cannot be waited for, and that refusal is no error of the launches to come.
void wait_done(Job* j) {
  if (cudaEventSynchronize(j->buf->done) != cudaSuccess) cudaGetLastError();
}

Job* find_job(bege_ctx* ctx, int32_t id) {
  auto it = ctx->jobs.find(id);
  return it == ctx->jobs.end() ? nullptr : it->second.get();
}

}  // namespace

// ---------------------------------------------------------------------------
// Batching form
// ---------------------------------------------------------------------------
static void destroy_batch(bege_ctx* ctx, Batch* b) {
  if (b->done) cudaEventSynchronize(b->done);
  if (b->exec) cudaGraphExecDestroy(b->exec);
  if (b->graph) cudaGraphDestroy(b->graph);
  if (b->done) cudaEventDestroy(b->done);
  if (b->t0) cudaEventDestroy(b->t0);
  if (b->t1) cudaEventDestroy(b->t1);
  if (b->cs) cudaStreamDestroy(b->cs);
  b->exec = nullptr;
  b->graph = nullptr;
  b->done = b->t0 = b->t1 = nullptr;
  b->cs = nullptr;
  for (DevBuf* d : {&b->y, &b->D, &b->AB, &b->segs, &b->items, &b->jobs, &b->queue, &b->sigma,
                    &b->recs, &b->counters})
    ctx->release(d);
}

static int log2i(int64_t n) {
  int k = 0;
  while ((int64_t(1) << k) < n) ++k;
  return k;
}

// Work items of `chunk` templates; order 0: longest segments first,
// order 1: entries interleaved chunk by chunk.
static std::vector<bege::BatchItem> batch_items(const Batch& b, int64_t chunk, int order) {
  std::vector<std::vector<bege::BatchItem>> per(b.entries.size());
  for (size_t e = 0; e < b.entries.size(); ++e)
    for (int64_t k = b.entries[e].k0; k < b.entries[e].k1; k += chunk)
      per[e].push_back({(int)e, 0, k, std::min(k + chunk, b.entries[e].k1)});
  std::vector<bege::BatchItem> out;
  if (order == 0) {
    std::vector<size_t> idx(b.entries.size());
    for (size_t i = 0; i < idx.size(); ++i) idx[i] = i;
    std::stable_sort(idx.begin(), idx.end(), [&](size_t x, size_t y) {
      return b.entries[x].n > b.entries[y].n;
    });
    for (size_t i : idx) out.insert(out.end(), per[i].begin(), per[i].end());
  } else {
    for (size_t r = 0;; ++r) {
      bool any = false;
      for (auto& v : per)
        if (r < v.size()) {
          out.push_back(v[r]);
          any = true;
        }
      if (!any) break;
    }
  }
  return out;
}

// (Re)build the work items for the batch's plan and capture its graph.
static int batch_build(bege_ctx* ctx, Batch* b) {
  if (b->exec) cudaGraphExecDestroy(b->exec);
  if (b->graph) cudaGraphDestroy(b->graph);
  b->exec = nullptr;
  b->graph = nullptr;
  cudaError_t e = cudaSuccess;
  if (b->plan == 0) {
    auto items = batch_items(*b, b->chunk, b->order);
    if (b->items.bytes < items.size() * sizeof(bege::BatchItem)) {
      ctx->release(&b->items);
      int rc = ctx->alloc(&b->items, items.size() * sizeof(bege::BatchItem));
      if (rc) return rc;
    }
    e = cudaMemcpy(b->items.ptr, items.data(), items.size() * sizeof(bege::BatchItem),
                   cudaMemcpyHostToDevice);
    if (e != cudaSuccess) return cuda_fail(e, "batch items");
    b->n_items = (int)items.size();
    b->args.items = static_cast<const bege::BatchItem*>(b->items.ptr);
    b->args.n_items = b->n_items;
  }
  const int clusters = bege::batch_max_clusters();
  if (b->plan == 0 && clusters < 1) return fail(BEGE_ECUDA, "batch kernel does not fit");
  // one uncaptured pass of the attribute setup of every kernel used below
  if (b->plan == 1) {
    for (const auto& en : b->entries) {
      auto pl = ctx->plans[en.n];
      auto ci = ctx->configs.find(en.n);
      const bege::CorrConfig cc = ci != ctx->configs.end() ? ci->second : bege::default_config(pl->g);
      bege::CorrelateArgs a{};
      a.k0 = a.k1 = 0;  // empty range: returns before launching
      bege::launch_correlate(pl->dev, a, cc, b->cs);
    }
  }
  e = cudaStreamBeginCapture(b->cs, cudaStreamCaptureModeRelaxed);
  if (e != cudaSuccess) return cuda_fail(e, "graph capture");
  e = cudaMemsetAsync(b->counters.ptr, 0, b->counters.bytes, b->cs);
  if (e == cudaSuccess) e = cudaMemsetAsync(b->queue.ptr, 0, b->queue.bytes, b->cs);
  if (e == cudaSuccess)
    e = bege::launch_segment_batch(b->args, static_cast<const bege::SegJob*>(b->jobs.ptr),
                                   b->n_jobs, b->cs);
  if (e == cudaSuccess) {
    if (b->plan == 0) e = bege::launch_batch(b->args, std::min(clusters, b->n_items), b->cs);
    for (size_t i = 0; i < b->entries.size() && e == cudaSuccess; ++i) {
      const auto& en = b->entries[i];
      const auto& sg = b->segs_host[i];
      auto pl = ctx->plans[en.n];
      auto ci = ctx->configs.find(en.n);
      const bege::CorrConfig cc =
          ci != ctx->configs.end() ? ci->second : bege::default_config(pl->g);
      bege::CorrelateArgs a{};
      a.AB = sg.AB;
      a.bank = sg.bank;
      a.Lp = sg.Lp;
      a.k0 = sg.k0;
      a.k1 = sg.k1;
      a.kappa = sg.kappa;
      a.sigma = sg.sigma;
      a.recs = sg.recs;
      a.cap = sg.cap;
      a.counter = sg.counter;
      a.dump = nullptr;
      a.max_clusters = 0;
      // no exchange buffer: up to 40 MB would be the batch's as long as it lives
      if (b->plan == 1) e = bege::launch_correlate(pl->dev, a, cc, b->cs);
      if (e == cudaSuccess && en.large) e = bege::launch_range(pl->dev, a, b->cs);
    }
  }
  cudaGraph_t g = nullptr;
  cudaError_t e2 = cudaStreamEndCapture(b->cs, &g);
  if (e != cudaSuccess || e2 != cudaSuccess) {
    if (g) cudaGraphDestroy(g);
    cudaGetLastError();
    return cuda_fail(e != cudaSuccess ? e : e2, "batch graph");
  }
  b->graph = g;
  e = cudaGraphInstantiate(&b->exec, g, 0);
  if (e != cudaSuccess) return cuda_fail(e, "graph instantiate");
  return BEGE_OK;
}

static Batch* find_batch(bege_ctx* ctx, int32_t id) {
  auto it = ctx->batches.find(id);
  return it == ctx->batches.end() ? nullptr : it->second.get();
}

static int batch_wait(Batch* b) {
  if (!b->ran) return fail(BEGE_ENOTREADY, "batch has not been run");
  cudaError_t e = cudaEventSynchronize(b->done);
  if (e != cudaSuccess) return cuda_fail(e, "batch");
  return BEGE_OK;
}

static int batch_run_locked(Batch* b, cudaStream_t s) {
  cudaError_t e = cudaEventRecord(b->t0, s);
  if (e == cudaSuccess) e = cudaGraphLaunch(b->exec, s);
  if (e == cudaSuccess) e = cudaEventRecord(b->t1, s);
  if (e == cudaSuccess) e = cudaEventRecord(b->done, s);
  if (e != cudaSuccess) return cuda_fail(e, "batch run");
  b->ran = true;
  return BEGE_OK;
}

extern "C" {

const char* bege_version(void) { return "bege 0.1 (sm_103a)"; }

const char* bege_last_error(const bege_ctx*) { return g_last_error.c_str(); }

int bege_create(bege_ctx** out, int device, const bege_config* cfg) {
  if (!out) return fail(BEGE_EINVAL, "out is NULL");
  *out = nullptr;
  bege_config c{};
  c.fs = 4096.0;
  c.tail_capacity = 1u << 20;
  if (cfg) {
    c = *cfg;
    if (c.fs == 0.0) c.fs = 4096.0;
    if (c.tail_capacity == 0) c.tail_capacity = 1u << 20;
  }
  if (!(c.fs > 0.0) || !std::isfinite(c.fs)) return fail(BEGE_EINVAL, "fs must be positive");
  if (c.precision < 0 || c.precision > 2)
    return fail(BEGE_EINVAL, "precision must be 0 (FP32), 1 (BF16x3) or 2 (FP16x3)");
  if (c.reserved != 0) return fail(BEGE_EINVAL, "reserved must be 0");
  int ndev = 0;
  cudaError_t e = cudaGetDeviceCount(&ndev);
  if (e != cudaSuccess) return cuda_fail(e, "cudaGetDeviceCount");
  if (device < 0 || device >= ndev) return fail(BEGE_EINVAL, "no such CUDA device");
  DeviceGuard dg(device);
  if (!dg.ok) return fail(BEGE_ECUDA, "cudaSetDevice failed");
  cudaDeviceProp prop;
  e = cudaGetDeviceProperties(&prop, device);
  if (e != cudaSuccess) return cuda_fail(e, "cudaGetDeviceProperties");
  if (prop.major < 10) return fail(BEGE_ECUDA, "libbege needs an sm_103a (Blackwell) GPU");
  auto* ctx = new bege_ctx();
  ctx->device = device;
  ctx->sms = prop.multiProcessorCount;
  ctx->cfg = c;
  *out = ctx;
  return BEGE_OK;
}

int bege_destroy(bege_ctx* ctx) {
  if (!ctx) return fail(BEGE_EINVAL, "ctx is NULL");
  bege::serve_destroy_all(ctx);
  {
    DeviceGuard dg(ctx->device);
    std::lock_guard<std::mutex> lk(ctx->mu);
    for (auto& kv : ctx->jobs) {
      wait_done(kv.second.get());
      ctx->release(&kv.second->proj);
      ctx->release(&kv.second->scratch);
      ctx->free_buffers(kv.second->buf.get());
    }
    for (auto& b : ctx->pool) ctx->free_buffers(b.get());
    ctx->drop_spare();
    for (auto& kv : ctx->batches) destroy_batch(ctx, kv.second.get());
    for (auto& kv : ctx->segs) {
      ctx->release(&kv.second->D);
      ctx->release(&kv.second->AB);
    }
    for (auto& kv : ctx->banks) ctx->release(&kv.second->w);
    for (auto& kv : ctx->plans) ctx->release(&kv.second->tables);
  }
  delete ctx;
  return BEGE_OK;
}

int bege_load_segment(bege_ctx* ctx, const float* strain, int64_t n, int32_t channel,
                      void* stream, int32_t* seg_id) {
  if (!ctx || !strain || !seg_id) return fail(BEGE_EINVAL, "NULL argument");
  if (!is_pow2(n) || n < 1024 || n > (1 << 17))
    return fail(BEGE_EINVAL, "n must be a power of two in [2^10, 2^17]");
  DeviceGuard dg(ctx->device);
  std::lock_guard<std::mutex> lk(ctx->mu);
  cudaStream_t s = static_cast<cudaStream_t>(stream);
  DevBuf tmp;
  int rc = ctx->take(&tmp, (size_t)n * sizeof(float));
  if (rc) return rc;
  cudaError_t e = cudaMemcpyAsync(tmp.ptr, strain, (size_t)n * sizeof(float),
                                  cudaMemcpyHostToDevice, s);
  if (e != cudaSuccess) {
    ctx->release(&tmp);
    return cuda_fail(e, "strain upload");
  }
  rc = segment_common(ctx, static_cast<const float*>(tmp.ptr), n, channel, s, seg_id);
  // the segment kernel reads tmp on stream s; wait before it is reused
  cudaError_t e2 = cudaStreamSynchronize(s);
  if (e2 == cudaSuccess)
    ctx->keep(&tmp);
  else
    ctx->release(&tmp);
  if (rc) return rc;
  if (e2 != cudaSuccess) return cuda_fail(e2, "segment kernel");
  ctx->segs[*seg_id]->loaded = true;
  return BEGE_OK;
}

int bege_load_segment_device(bege_ctx* ctx, const float* strain_dev, int64_t n, int32_t channel,
                             void* stream, int32_t* seg_id) {
  if (!ctx || !strain_dev || !seg_id) return fail(BEGE_EINVAL, "NULL argument");
  if (!is_pow2(n) || n < 1024 || n > (1 << 17))
    return fail(BEGE_EINVAL, "n must be a power of two in [2^10, 2^17]");
  if (reinterpret_cast<uintptr_t>(strain_dev) % 8 != 0)
    return fail(BEGE_EINVAL, "strain_dev must be 8-byte aligned");
  DeviceGuard dg(ctx->device);
  std::lock_guard<std::mutex> lk(ctx->mu);
  return segment_common(ctx, strain_dev, n, channel, static_cast<cudaStream_t>(stream), seg_id);
}

static int define_bank_impl(bege_ctx* ctx, const bege_chirp* params, int64_t count, double tau,
                            double taper_frac, void* stream, int32_t* bank_id, bool symmetric) {
  if (!ctx || !params || !bank_id) return fail(BEGE_EINVAL, "NULL argument");
  if (count <= 0 || count > (int64_t)1 << 31) return fail(BEGE_EINVAL, "count out of range");
  if (!(tau > 0.0) || !std::isfinite(tau)) return fail(BEGE_EINVAL, "tau must be positive");
  if (!(taper_frac >= 0.0 && taper_frac <= 1.0)) return fail(BEGE_EINVAL, "taper_frac in [0,1]");
  const int64_t L = (int64_t)std::llround(tau * ctx->cfg.fs);
  if (L < 1 || L > (1 << 16)) return fail(BEGE_EINVAL, "tau * fs must be in [1, 2^16]");
  std::vector<unsigned long long> ab((size_t)count * 2);
  const double fs = ctx->cfg.fs;
  for (int64_t k = 0; k < count; ++k) {
    if (!std::isfinite(params[k].f0) || !std::isfinite(params[k].fdot))
      return fail(BEGE_EINVAL, "non-finite chirp parameter");
    ab[2 * k] = frac_to_u64(params[k].f0 / fs);
    ab[2 * k + 1] = frac_to_u64(0.5 * params[k].fdot / (fs * fs));
  }
  DeviceGuard dg(ctx->device);
  std::lock_guard<std::mutex> lk(ctx->mu);
  cudaStream_t s = static_cast<cudaStream_t>(stream);
  auto bank = std::make_unique<Bank>();
  bank->count = count;
  bank->L = L;
  bank->Lp = (L + 7) / 8 * 8;
  int rc = ctx->alloc(&bank->w, (size_t)count * bank->Lp * sizeof(float));
  if (rc) return rc;
  DevBuf dab;
  rc = ctx->alloc(&dab, ab.size() * sizeof(unsigned long long));
  if (rc) {
    ctx->release(&bank->w);
    return rc;
  }
  cudaError_t e = cudaMemcpyAsync(dab.ptr, ab.data(), ab.size() * sizeof(unsigned long long),
                                  cudaMemcpyHostToDevice, s);
  if (e == cudaSuccess)
    e = bege::launch_bank_chirp(static_cast<unsigned long long*>(dab.ptr), count, L, bank->Lp,
                                taper_frac, symmetric, static_cast<float*>(bank->w.ptr), s);
  cudaError_t e2 = cudaStreamSynchronize(s);
  ctx->release(&dab);
  if (e != cudaSuccess || e2 != cudaSuccess) {
    ctx->release(&bank->w);
    return cuda_fail(e != cudaSuccess ? e : e2, "bank synthesis");
  }
  const int32_t id = ctx->next_id++;
  ctx->banks[id] = std::move(bank);
  *bank_id = id;
  return BEGE_OK;
}

int bege_define_bank(bege_ctx* ctx, const bege_chirp* params, int64_t count, double tau,
                     double taper_frac, void* stream, int32_t* bank_id) {
  return define_bank_impl(ctx, params, count, tau, taper_frac, stream, bank_id, false);
}

int bege_define_bank_symmetric(bege_ctx* ctx, const bege_chirp* params, int64_t count,
                               double tau, double taper_frac, void* stream, int32_t* bank_id) {
  return define_bank_impl(ctx, params, count, tau, taper_frac, stream, bank_id, true);
}

int bege_define_bank_samples(bege_ctx* ctx, const float* samples, int64_t count, int64_t length,
                             void* stream, int32_t* bank_id) {
  if (!ctx || !samples || !bank_id) return fail(BEGE_EINVAL, "NULL argument");
  if (count <= 0 || count > (int64_t)1 << 31) return fail(BEGE_EINVAL, "count out of range");
  if (length < 1 || length > (1 << 16)) return fail(BEGE_EINVAL, "length must be in [1, 2^16]");
  DeviceGuard dg(ctx->device);
  std::lock_guard<std::mutex> lk(ctx->mu);
  cudaStream_t s = static_cast<cudaStream_t>(stream);
  auto bank = std::make_unique<Bank>();
  bank->count = count;
  bank->L = length;
  bank->Lp = (length + 7) / 8 * 8;
  int rc = ctx->alloc(&bank->w, (size_t)count * bank->Lp * sizeof(float));
  if (rc) return rc;
  cudaError_t e = cudaMemsetAsync(bank->w.ptr, 0, bank->w.bytes, s);
  if (e == cudaSuccess)
    e = cudaMemcpy2DAsync(bank->w.ptr, bank->Lp * sizeof(float), samples, length * sizeof(float),
                          length * sizeof(float), (size_t)count, cudaMemcpyHostToDevice, s);
  DevBuf flag;  // without room for it the bank counts as large
  int large = 1;
  if (e == cudaSuccess && ctx->take(&flag, 16) == BEGE_OK) {
    e = bege::launch_bank_large(static_cast<float*>(bank->w.ptr), count * bank->Lp,
                                static_cast<int*>(flag.ptr), s);
    if (e == cudaSuccess)
      e = cudaMemcpyAsync(&large, flag.ptr, sizeof(int), cudaMemcpyDeviceToHost, s);
  }
  if (e == cudaSuccess) e = cudaStreamSynchronize(s);
  if (e != cudaSuccess) {
    ctx->release(&flag);
    ctx->release(&bank->w);
    return cuda_fail(e, "bank upload");
  }
  ctx->keep(&flag);
  bank->large = large != 0;
  const int32_t id = ctx->next_id++;
  ctx->banks[id] = std::move(bank);
  *bank_id = id;
  return BEGE_OK;
}

static int correlate_impl(bege_ctx* ctx, int32_t seg_id, int32_t bank_id, int64_t k_begin,
                          int64_t k_end, float kappa, cudaStream_t s, float* dump_dev,
                          int32_t* job_id, bool project = false, float kappa_hi = 0.f,
                          bool linear = false) {
  auto si = ctx->segs.find(seg_id);
  if (si == ctx->segs.end()) return fail(BEGE_EINVAL, "unknown segment handle");
  auto bi = ctx->banks.find(bank_id);
  if (bi == ctx->banks.end()) return fail(BEGE_EINVAL, "unknown bank handle");
  Segment* seg = si->second.get();
  Bank* bank = bi->second.get();
  if (k_begin < 0 || k_end > bank->count || k_begin >= k_end)
    return fail(BEGE_EINVAL, "template range outside the bank or empty");
  if (bank->L > seg->n) return fail(BEGE_EINVAL, "template longer than the segment");
  if (ctx->cfg.precision != 0 && (seg->n < (1 << 14) || bank->Lp > 4096))
    return fail(BEGE_EINVAL,
                "the tensor-core precision form needs N >= 2^14 and templates of at most 4096 "
                "samples");
  if (!std::isfinite(kappa) && !(dump_dev && std::isinf(kappa)))
    return fail(BEGE_EINVAL, "kappa must be finite");
  if (kappa < 0.f) return fail(BEGE_EINVAL, "kappa must be >= 0");
  const int64_t nsig = k_end - k_begin;
  auto job = std::make_unique<Job>();
  job->seg = seg_id;
  job->bank = bank_id;
  job->k0 = k_begin;
  job->k1 = k_end;
  job->kappa = kappa;
  int rc = take_job_buffers(ctx, nsig, ctx->cfg.tail_capacity, &job->buf);
  if (rc) return rc;
  if (project) {
    rc = ctx->alloc(&job->proj, (size_t)seg->n * sizeof(unsigned long long));
    if (rc) {
      ctx->pool.push_back(std::move(job->buf));
      return rc;
    }
    job->n_proj = seg->n;
  }
  cudaError_t e = cudaSuccess;
  if (project) e = cudaMemsetAsync(job->proj.ptr, 0, job->proj.bytes, s);
  if (e == cudaSuccess) e = cudaMemsetAsync(job->buf->counter.ptr, 0, 16, s);
  auto ci = ctx->configs.find(seg->n);
  const bege::CorrConfig cc =
      ci != ctx->configs.end() ? ci->second : bege::default_config(seg->plan->g);
  // a context with a budget, or a full device, does without; ahead of the
  // event, for an idle stream passes it while the call still allocates
  float4* exch = nullptr;
  if (e == cudaSuccess && ctx->cfg.precision == 0)
    exch = ctx->take_exchange(job->buf.get(),
                              bege::exchange_bytes(seg->plan->g, cc, nsig, ctx->sms), s);
  if (e == cudaSuccess) e = cudaEventRecord(job->buf->k_start, s);
  if (e == cudaSuccess) {
    bege::CorrelateArgs a{};
    a.AB = static_cast<const float4*>(seg->AB.ptr);
    a.bank = static_cast<const float*>(bank->w.ptr);
    a.Lp = bank->Lp;
    a.k0 = k_begin;
    a.k1 = k_end;
    a.kappa = kappa;
    a.sigma = static_cast<float*>(job->buf->sigma.ptr);
    a.recs = static_cast<bege_tail*>(job->buf->recs.ptr);
    a.cap = job->buf->rec_cap;
    a.counter = static_cast<unsigned long long*>(job->buf->counter.ptr);
    a.dump = dump_dev;
    a.max_clusters = 0;
    a.status = reinterpret_cast<unsigned int*>(static_cast<char*>(job->buf->counter.ptr) + 8);
    a.proj = static_cast<unsigned long long*>(job->proj.ptr);
    a.kappa_hi = kappa_hi;
    a.exch = exch;
    // overlap-save: the window y[n .. n+L-1] of a length-L template stays
    // inside the segment for n <= N - L
    if (linear) a.lag_end = (uint32_t)(seg->n - bank->L + 1);
    if (ctx->cfg.precision != 0) {
      e = bege::launch_correlate_tc(seg->plan->dev, a, ctx->cfg.precision, s);
    } else {
      e = bege::launch_correlate(seg->plan->dev, a, cc, s);
      if (e == cudaSuccess && bank->large) e = bege::launch_range(seg->plan->dev, a, s);
    }
  }
  if (e == cudaSuccess) e = cudaEventRecord(job->buf->k_stop, s);
  if (e == cudaSuccess) e = cudaEventRecord(job->buf->done, s);
  if (e != cudaSuccess) {
    ctx->release(&job->proj);
    ctx->drop_exchange(&job->buf->exch);  // waits for a kernel that may use it
    ctx->pool.push_back(std::move(job->buf));
    return cuda_fail(e, "correlate");
  }
  const int32_t id = ctx->next_id++;
  ctx->jobs[id] = std::move(job);
  *job_id = id;
  return BEGE_OK;
}

int bege_correlate(bege_ctx* ctx, int32_t seg_id, int32_t bank_id, int64_t k_begin,
                   int64_t k_end, float kappa, void* stream, int32_t* job_id) {
  if (!ctx || !job_id) return fail(BEGE_EINVAL, "NULL argument");
  DeviceGuard dg(ctx->device);
  std::lock_guard<std::mutex> lk(ctx->mu);
  return correlate_impl(ctx, seg_id, bank_id, k_begin, k_end, kappa,
                        static_cast<cudaStream_t>(stream), nullptr, job_id);
}

int bege_correlate_multi(bege_ctx* ctx, const int32_t* seg_ids, int32_t n_seg, int32_t bank_id,
                         int64_t k_begin, int64_t k_end, float kappa, void* stream,
                         int32_t* job_ids) {
  if (!ctx || !seg_ids || !job_ids) return fail(BEGE_EINVAL, "NULL argument");
  if (n_seg < 1 || n_seg > bege::kMaxMulti)
    return fail(BEGE_EINVAL, "between 1 and " + std::to_string(bege::kMaxMulti) + " segments");
  DeviceGuard dg(ctx->device);
  std::lock_guard<std::mutex> lk(ctx->mu);
  if (ctx->cfg.precision != 0)
    return fail(BEGE_EINVAL, "the multi-segment search runs the FP32 path (precision 0)");
  auto bi = ctx->banks.find(bank_id);
  if (bi == ctx->banks.end()) return fail(BEGE_EINVAL, "unknown bank handle");
  Bank* bank = bi->second.get();
  if (k_begin < 0 || k_end > bank->count || k_begin >= k_end)
    return fail(BEGE_EINVAL, "template range outside the bank or empty");
  if (!std::isfinite(kappa) || kappa < 0.f) return fail(BEGE_EINVAL, "kappa must be finite, >= 0");
  std::vector<Segment*> segs;
  for (int32_t i = 0; i < n_seg; ++i) {
    auto si = ctx->segs.find(seg_ids[i]);
    if (si == ctx->segs.end()) return fail(BEGE_EINVAL, "unknown segment handle");
    segs.push_back(si->second.get());
  }
  const int64_t n = segs[0]->n;
  for (Segment* sg : segs)
    if (sg->n != n) return fail(BEGE_EINVAL, "the segments must have one length");
  if (n < (1 << 14) || bank->Lp > 4096 || bank->L > n)
    return fail(BEGE_EINVAL, "the multi-segment search needs N >= 2^14 and templates of at "
                             "most 4096 samples");
  int sms = 0;
  cudaError_t e = cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, ctx->device);
  if (e != cudaSuccess) return cuda_fail(e, "device attribute");
  cudaStream_t s = static_cast<cudaStream_t>(stream);
  std::vector<std::unique_ptr<Job>> jobs;
  auto unwind = [&](int rc) {
    for (auto& j : jobs) {
      ctx->release(&j->scratch);
      if (j->buf) ctx->pool.push_back(std::move(j->buf));
    }
    return rc;
  };
  for (int32_t i = 0; i < n_seg; ++i) {
    auto job = std::make_unique<Job>();
    job->seg = seg_ids[i];
    job->bank = bank_id;
    job->k0 = k_begin;
    job->k1 = k_end;
    job->kappa = kappa;
    jobs.push_back(std::move(job));
    Job* j = jobs.back().get();
    int rc = take_job_buffers(ctx, k_end - k_begin, ctx->cfg.tail_capacity, &j->buf);
    if (rc) return unwind(rc);
    e = cudaMemsetAsync(j->buf->counter.ptr, 0, 16, s);
    if (e != cudaSuccess) return unwind(cuda_fail(e, "multi-segment job"));
  }
  int rc = ctx->alloc(&jobs[0]->scratch, bege::multi_scratch_bytes(sms));
  if (rc) return unwind(rc);
  bege::MultiArgs a{};
  a.bank = static_cast<const float*>(bank->w.ptr);
  a.Lp = bank->Lp;
  a.k0 = k_begin;
  a.k1 = k_end;
  a.kappa = kappa;
  a.M = n_seg;
  for (int32_t i = 0; i < n_seg; ++i) {
    a.AB[i] = static_cast<const float4*>(segs[i]->AB.ptr);
    a.sigma[i] = static_cast<float*>(jobs[i]->buf->sigma.ptr);
    a.recs[i] = static_cast<bege_tail*>(jobs[i]->buf->recs.ptr);
    a.cap[i] = jobs[i]->buf->rec_cap;
    a.counter[i] = static_cast<unsigned long long*>(jobs[i]->buf->counter.ptr);
  }
  a.scratch = static_cast<float4*>(jobs[0]->scratch.ptr);
  for (auto& j : jobs)
    if (e == cudaSuccess) e = cudaEventRecord(j->buf->k_start, s);
  if (e == cudaSuccess) e = bege::launch_correlate_multi(segs[0]->plan->dev, a, s);
  for (int32_t i = 0; i < n_seg && bank->large && e == cudaSuccess; ++i) {
    bege::CorrelateArgs one{};
    one.AB = a.AB[i];
    one.bank = a.bank;
    one.Lp = a.Lp;
    one.k0 = a.k0;
    one.k1 = a.k1;
    one.kappa = a.kappa;
    one.sigma = a.sigma[i];
    one.recs = a.recs[i];
    one.cap = a.cap[i];
    one.counter = a.counter[i];
    e = bege::launch_range(segs[i]->plan->dev, one, s);
  }
  for (auto& j : jobs) {
    if (e == cudaSuccess) e = cudaEventRecord(j->buf->k_stop, s);
    if (e == cudaSuccess) e = cudaEventRecord(j->buf->done, s);
  }
  if (e != cudaSuccess) return unwind(cuda_fail(e, "multi-segment correlate"));
  for (int32_t i = 0; i < n_seg; ++i) {
    const int32_t id = ctx->next_id++;
    ctx->jobs[id] = std::move(jobs[i]);
    job_ids[i] = id;
  }
  return BEGE_OK;
}

int bege_correlate_max(bege_ctx* ctx, int32_t seg_id, int32_t bank_id, int64_t k_begin,
                       int64_t k_end, float kappa, void* stream, int32_t* job_id) {
  if (!ctx || !job_id) return fail(BEGE_EINVAL, "NULL argument");
  DeviceGuard dg(ctx->device);
  std::lock_guard<std::mutex> lk(ctx->mu);
  return correlate_impl(ctx, seg_id, bank_id, k_begin, k_end, kappa,
                        static_cast<cudaStream_t>(stream), nullptr, job_id, true);
}

int bege_correlate_band(bege_ctx* ctx, int32_t seg_id, int32_t bank_id, int64_t k_begin,
                        int64_t k_end, float kappa_lo, float kappa_hi, void* stream,
                        int32_t* job_id) {
  if (!ctx || !job_id) return fail(BEGE_EINVAL, "NULL argument");
  if (!std::isfinite(kappa_lo) || !std::isfinite(kappa_hi) || !(kappa_hi > kappa_lo))
    return fail(BEGE_EINVAL, "the band needs finite kappa_lo < kappa_hi");
  DeviceGuard dg(ctx->device);
  std::lock_guard<std::mutex> lk(ctx->mu);
  return correlate_impl(ctx, seg_id, bank_id, k_begin, k_end, kappa_lo,
                        static_cast<cudaStream_t>(stream), nullptr, job_id, false, kappa_hi);
}

int bege_correlate_ex(bege_ctx* ctx, int32_t seg_id, int32_t bank_id, int64_t k_begin,
                      int64_t k_end, const bege_search_opts* opts, void* stream,
                      int32_t* job_id) {
  if (!ctx || !opts || !job_id) return fail(BEGE_EINVAL, "NULL argument");
  const bege_search_opts o = *opts;
  if (!std::isfinite(o.kappa) || !std::isfinite(o.kappa_hi))
    return fail(BEGE_EINVAL, "kappa and kappa_hi must be finite");
  if (o.kappa_hi != 0.f && !(o.kappa_hi > o.kappa))
    return fail(BEGE_EINVAL, "kappa_hi must be 0 (no upper end) or above kappa");
  if ((o.linear != 0 && o.linear != 1) || (o.project != 0 && o.project != 1))
    return fail(BEGE_EINVAL, "linear and project must be 0 or 1");
  DeviceGuard dg(ctx->device);
  std::lock_guard<std::mutex> lk(ctx->mu);
  return correlate_impl(ctx, seg_id, bank_id, k_begin, k_end, o.kappa,
                        static_cast<cudaStream_t>(stream), nullptr, job_id, o.project == 1,
                        o.kappa_hi, o.linear == 1);
}

int bege_fetch_max(bege_ctx* ctx, int32_t job_id, float* snr, int32_t* tmpl, int64_t n) {
  if (!ctx || !snr || !tmpl) return fail(BEGE_EINVAL, "NULL argument");
  DeviceGuard dg(ctx->device);
  std::lock_guard<std::mutex> lk(ctx->mu);
  Job* j = find_job(ctx, job_id);
  if (!j) return fail(BEGE_EINVAL, "unknown job handle");
  if (!j->proj.ptr) return fail(BEGE_EINVAL, "the job was not started by bege_correlate_max");
  if (n != j->n_proj) return fail(BEGE_EINVAL, "n must equal the segment length");
  int rc = wait_counted(j);
  if (rc) return rc;
  std::vector<unsigned long long> w((size_t)n);
  cudaError_t e = cudaMemcpy(w.data(), j->proj.ptr, (size_t)n * sizeof(unsigned long long),
                 cudaMemcpyDeviceToHost);
  if (e != cudaSuccess) return cuda_fail(e, "projection");
  for (int64_t i = 0; i < n; ++i) {
    if (w[i] == 0) {
      snr[i] = 0.f;
      tmpl[i] = -1;
    } else {
      const uint32_t hi = (uint32_t)(w[i] >> 32);
      float v;
      std::memcpy(&v, &hi, sizeof v);
      snr[i] = v;
      tmpl[i] = (int32_t)(~(uint32_t)(w[i] & 0xffffffffull));
    }
  }
  return BEGE_OK;
}

int bege_job_kernel_ms(bege_ctx* ctx, int32_t job_id, float* ms) {
  if (!ctx || !ms) return fail(BEGE_EINVAL, "NULL argument");
  DeviceGuard dg(ctx->device);
  std::lock_guard<std::mutex> lk(ctx->mu);
  Job* j = find_job(ctx, job_id);
  if (!j) return fail(BEGE_EINVAL, "unknown job handle");
  cudaError_t e = cudaEventSynchronize(j->buf->done);
  if (e == cudaSuccess) e = cudaEventElapsedTime(ms, j->buf->k_start, j->buf->k_stop);
  if (e != cudaSuccess) return cuda_fail(e, "kernel time");
  return BEGE_OK;
}

int bege_query(bege_ctx* ctx, int32_t job_id) {
  if (!ctx) return fail(BEGE_EINVAL, "NULL argument");
  DeviceGuard dg(ctx->device);
  std::lock_guard<std::mutex> lk(ctx->mu);
  Job* j = find_job(ctx, job_id);
  if (!j) return fail(BEGE_EINVAL, "unknown job handle");
  cudaError_t e = cudaEventQuery(j->buf->done);
  if (e == cudaErrorNotReady) return BEGE_ENOTREADY;
  if (e != cudaSuccess) return cuda_fail(e, "job");
  return BEGE_OK;
}

int bege_sort_tails(bege_tail* recs, int64_t n) {
  if (n < 0 || (n > 0 && !recs)) return fail(BEGE_EINVAL, "bad record array");
  std::sort(recs, recs + n, [](const bege_tail& x, const bege_tail& y) {
    return x.tmpl != y.tmpl ? x.tmpl < y.tmpl : x.lag < y.lag;
  });
  return BEGE_OK;
}

int bege_fetch_tails(bege_ctx* ctx, int32_t job_id, bege_tail* out, int64_t capacity,
                     int64_t* n_written, int64_t* n_total) {
  if (!ctx || !n_written || !n_total) return fail(BEGE_EINVAL, "NULL argument");
  if (capacity < 0 || (capacity > 0 && !out)) return fail(BEGE_EINVAL, "bad output buffer");
  DeviceGuard dg(ctx->device);
  std::lock_guard<std::mutex> lk(ctx->mu);
  Job* j = find_job(ctx, job_id);
  if (!j) return fail(BEGE_EINVAL, "unknown job handle");
  int rc = wait_counted(j);
  if (rc) return rc;
  const unsigned long long total = j->count[0];
  uint64_t ncopy = total;
  if (ncopy > j->buf->rec_cap) ncopy = j->buf->rec_cap;
  if (ncopy > (uint64_t)capacity) ncopy = (uint64_t)capacity;
  if (ncopy) {
    cudaError_t e = cudaMemcpy(out, j->buf->recs.ptr, ncopy * sizeof(bege_tail),
                               cudaMemcpyDeviceToHost);
    if (e != cudaSuccess) return cuda_fail(e, "tail records");
  }
  *n_written = (int64_t)ncopy;
  *n_total = (int64_t)total;
  if (ncopy < total)
    return fail(BEGE_EOVERFLOW, "more tails (" + std::to_string(total) + ") than copied (" +
                                    std::to_string(ncopy) + ")");
  return BEGE_OK;
}

int bege_get_sigma(bege_ctx* ctx, int32_t job_id, float* out, int64_t count) {
  if (!ctx || !out) return fail(BEGE_EINVAL, "NULL argument");
  DeviceGuard dg(ctx->device);
  std::lock_guard<std::mutex> lk(ctx->mu);
  Job* j = find_job(ctx, job_id);
  if (!j) return fail(BEGE_EINVAL, "unknown job handle");
  if (count != j->k1 - j->k0) return fail(BEGE_EINVAL, "count must equal k_end - k_begin");
  cudaError_t e = cudaEventSynchronize(j->buf->done);
  if (e == cudaSuccess)
    e = cudaMemcpy(out, j->buf->sigma.ptr, (size_t)count * sizeof(float), cudaMemcpyDeviceToHost);
  if (e != cudaSuccess) return cuda_fail(e, "sigma");
  return BEGE_OK;
}

int bege_dump_correlation(bege_ctx* ctx, int32_t seg_id, int32_t bank_id, int64_t k_begin,
                          int64_t k_end, float* out, void* stream) {
  if (!ctx || !out) return fail(BEGE_EINVAL, "NULL argument");
  DeviceGuard dg(ctx->device);
  std::lock_guard<std::mutex> lk(ctx->mu);
  auto si = ctx->segs.find(seg_id);
  if (si == ctx->segs.end()) return fail(BEGE_EINVAL, "unknown segment handle");
  if (k_end <= k_begin) return fail(BEGE_EINVAL, "empty template range");
  const int64_t n = si->second->n;
  cudaStream_t s = static_cast<cudaStream_t>(stream);
  DevBuf d;
  int rc = ctx->alloc(&d, (size_t)(k_end - k_begin) * n * sizeof(float));
  if (rc) return rc;
  int32_t job = -1;
  rc = correlate_impl(ctx, seg_id, bank_id, k_begin, k_end, INFINITY, s,
                      static_cast<float*>(d.ptr), &job);
  if (rc) {
    ctx->release(&d);
    return rc;
  }
  cudaError_t e = cudaStreamSynchronize(s);
  if (e == cudaSuccess)
    e = cudaMemcpy(out, d.ptr, (size_t)(k_end - k_begin) * n * sizeof(float),
                   cudaMemcpyDeviceToHost);
  ctx->release(&d);
  Job* j = find_job(ctx, job);
  if (j) {
    ctx->give_back(std::move(j->buf));
    ctx->jobs.erase(job);
  }
  if (e != cudaSuccess) return cuda_fail(e, "dump");
  return BEGE_OK;
}

int bege_list_configs(bege_ctx* ctx, int64_t n, int32_t* out, int32_t max, int32_t* count) {
  if (!ctx || !count || (max > 0 && !out)) return fail(BEGE_EINVAL, "NULL argument");
  if (!is_pow2(n) || n < 1024 || n > (1 << 17)) return fail(BEGE_EINVAL, "bad segment length");
  bege::CorrConfig c[8];
  const int k = bege::correlate_configs(bege::make_geometry(n), c, 8);
  for (int i = 0; i < k && i < max; ++i) {
    out[2 * i] = c[i].nc;
    out[2 * i + 1] = c[i].threads;
  }
  *count = k;
  return BEGE_OK;
}

int bege_set_config(bege_ctx* ctx, int64_t n, int32_t nc, int32_t threads) {
  if (!ctx) return fail(BEGE_EINVAL, "NULL argument");
  if (!is_pow2(n) || n < 1024 || n > (1 << 17)) return fail(BEGE_EINVAL, "bad segment length");
  const bege::CorrConfig c{nc, threads};
  if (!bege::config_valid(bege::make_geometry(n), c))
    return fail(BEGE_EINVAL, "launch shape not compiled for this length");
  std::lock_guard<std::mutex> lk(ctx->mu);
  ctx->configs[n] = c;
  return BEGE_OK;
}

int bege_get_config(bege_ctx* ctx, int64_t n, int32_t* nc, int32_t* threads) {
  if (!ctx || !nc || !threads) return fail(BEGE_EINVAL, "NULL argument");
  if (!is_pow2(n) || n < 1024 || n > (1 << 17)) return fail(BEGE_EINVAL, "bad segment length");
  std::lock_guard<std::mutex> lk(ctx->mu);
  auto it = ctx->configs.find(n);
  const bege::CorrConfig c =
      it != ctx->configs.end() ? it->second : bege::default_config(bege::make_geometry(n));
  *nc = c.nc;
  *threads = c.threads;
  return BEGE_OK;
}

int bege_autotune(bege_ctx* ctx, int32_t seg_id, int32_t bank_id, int64_t k_begin, int64_t k_end,
                  int32_t reps, void* stream, float* best_ms) {
  if (!ctx || !best_ms || reps < 1) return fail(BEGE_EINVAL, "bad argument");
  DeviceGuard dg(ctx->device);
  std::lock_guard<std::mutex> lk(ctx->mu);
  auto si = ctx->segs.find(seg_id);
  if (si == ctx->segs.end()) return fail(BEGE_EINVAL, "unknown segment handle");
  const int64_t n = si->second->n;
  cudaStream_t s = static_cast<cudaStream_t>(stream);
  bege::CorrConfig cand[8];
  const int nc = bege::correlate_configs(si->second->plan->g, cand, 8);
  float best = 0.f;
  bege::CorrConfig pick = bege::default_config(si->second->plan->g);
  for (int i = 0; i < nc; ++i) {
    ctx->configs[n] = cand[i];
    std::vector<float> t;
    for (int r = 0; r <= reps; ++r) {
      int32_t job = -1;
      int rc = correlate_impl(ctx, seg_id, bank_id, k_begin, k_end, 1e30f, s, nullptr, &job);
      if (rc) return rc;
      Job* j = find_job(ctx, job);
      float ms = 0.f;
      cudaError_t e = cudaEventSynchronize(j->buf->done);
      if (e == cudaSuccess) e = cudaEventElapsedTime(&ms, j->buf->k_start, j->buf->k_stop);
      ctx->give_back(std::move(j->buf));
      ctx->jobs.erase(job);
      if (e != cudaSuccess) return cuda_fail(e, "autotune");
      if (r > 0) t.push_back(ms);
    }
    std::sort(t.begin(), t.end());
    const float med = t[t.size() / 2];
    if (i == 0 || med < best) {
      best = med;
      pick = cand[i];
    }
  }
  ctx->configs[n] = pick;
  *best_ms = best;
  return BEGE_OK;
}

int bege_get_segment_spectrum(bege_ctx* ctx, int32_t seg_id, float* out) {
  if (!ctx || !out) return fail(BEGE_EINVAL, "NULL argument");
  DeviceGuard dg(ctx->device);
  std::lock_guard<std::mutex> lk(ctx->mu);
  auto si = ctx->segs.find(seg_id);
  if (si == ctx->segs.end()) return fail(BEGE_EINVAL, "unknown segment handle");
  cudaError_t e = cudaDeviceSynchronize();
  if (e == cudaSuccess)
    e = cudaMemcpy(out, si->second->D.ptr, si->second->D.bytes, cudaMemcpyDeviceToHost);
  if (e != cudaSuccess) return cuda_fail(e, "segment spectrum");
  return BEGE_OK;
}

int bege_get_bank_samples(bege_ctx* ctx, int32_t bank_id, int64_t k_begin, int64_t k_end,
                          float* out) {
  if (!ctx || !out) return fail(BEGE_EINVAL, "NULL argument");
  DeviceGuard dg(ctx->device);
  std::lock_guard<std::mutex> lk(ctx->mu);
  auto bi = ctx->banks.find(bank_id);
  if (bi == ctx->banks.end()) return fail(BEGE_EINVAL, "unknown bank handle");
  Bank* b = bi->second.get();
  if (k_begin < 0 || k_end > b->count || k_begin >= k_end)
    return fail(BEGE_EINVAL, "row range outside the bank");
  cudaError_t e = cudaDeviceSynchronize();
  if (e == cudaSuccess)
    e = cudaMemcpy2D(out, b->L * sizeof(float),
                     static_cast<const float*>(b->w.ptr) + k_begin * b->Lp, b->Lp * sizeof(float),
                     b->L * sizeof(float), (size_t)(k_end - k_begin), cudaMemcpyDeviceToHost);
  if (e != cudaSuccess) return cuda_fail(e, "bank samples");
  return BEGE_OK;
}

int64_t bege_segment_length(bege_ctx* ctx, int32_t seg_id) {
  if (!ctx) return 0;
  std::lock_guard<std::mutex> lk(ctx->mu);
  auto si = ctx->segs.find(seg_id);
  return si == ctx->segs.end() ? 0 : si->second->n;
}

}  // extern "C"

namespace bege {
int ctx_device(const bege_ctx* ctx) { return ctx->device; }
void ctx_drop_spare(bege_ctx* ctx) {
  DeviceGuard dg(ctx->device);
  std::lock_guard<std::mutex> lk(ctx->mu);
  ctx->drop_spare();
}
int64_t bank_count(bege_ctx* ctx, int32_t bank_id) {
  std::lock_guard<std::mutex> lk(ctx->mu);
  auto bi = ctx->banks.find(bank_id);
  return bi == ctx->banks.end() ? 0 : bi->second->count;
}
}  // namespace bege

extern "C" {

int64_t bege_bank_length(bege_ctx* ctx, int32_t bank_id) {
  if (!ctx) return 0;
  std::lock_guard<std::mutex> lk(ctx->mu);
  auto bi = ctx->banks.find(bank_id);
  return bi == ctx->banks.end() ? 0 : bi->second->L;
}

uint64_t bege_device_bytes(const bege_ctx* ctx) { return ctx ? ctx->bytes : 0; }

int bege_batch_create(bege_ctx* ctx, const bege_batch_entry* entries, int32_t count,
                      uint64_t tail_capacity, void* stream, int32_t* batch_id) {
  if (!ctx || !entries || !batch_id || count <= 0) return fail(BEGE_EINVAL, "bad argument");
  DeviceGuard dg(ctx->device);
  std::lock_guard<std::mutex> lk(ctx->mu);
  cudaStream_t us = static_cast<cudaStream_t>(stream);
  auto b = std::make_unique<Batch>();
  b->cap = tail_capacity ? tail_capacity : ctx->cfg.tail_capacity;
  size_t ny = 0, nD = 0, nAB = 0, nsig = 0;
  for (int32_t i = 0; i < count; ++i) {
    const bege_batch_entry& en = entries[i];
    if (!en.strain || en.reserved != 0 || en.reserved2 != 0.f)
      return fail(BEGE_EINVAL, "batch entry: NULL strain or non-zero reserved field");
    if (en.n != (1 << 14) && en.n != (1 << 15) && en.n != (1 << 16) && en.n != (1 << 17))
      return fail(BEGE_EINVAL, "batch entry: n must be 2^14, 2^15, 2^16 or 2^17");
    auto bi = ctx->banks.find(en.bank_id);
    if (bi == ctx->banks.end()) return fail(BEGE_EINVAL, "batch entry: unknown bank handle");
    if (bi->second->Lp > 4096)
      return fail(BEGE_EINVAL, "batch entry: template longer than 4096 samples");
    if (en.k_begin < 0 || en.k_end > bi->second->count || en.k_begin >= en.k_end)
      return fail(BEGE_EINVAL, "batch entry: template range outside the bank or empty");
    if (!std::isfinite(en.kappa) || en.kappa < 0.f)
      return fail(BEGE_EINVAL, "batch entry: kappa must be finite and >= 0");
    b->entries.push_back({en.n, en.bank_id, en.k_begin, en.k_end, en.kappa, bi->second->large});
    b->sigma_off.push_back(nsig);
    ny += en.n;
    nD += en.n / 2 + 1;
    nAB += en.n / 2;
    nsig += en.k_end - en.k_begin;
  }
  for (int64_t n : {1 << 14, 1 << 15, 1 << 16, 1 << 17}) {
    std::shared_ptr<PlanHost> pl;
    int rc = get_plan(ctx, n, &pl);
    if (rc) return rc;
    b->args.plans[log2i(n) - 14] = pl->dev;
  }
  struct Need {
    DevBuf* d;
    size_t bytes;
  } need[] = {{&b->y, ny * 4}, {&b->D, nD * 8}, {&b->AB, nAB * 16},
              {&b->segs, count * sizeof(bege::BatchSeg)}, {&b->queue, 16},
              {&b->sigma, nsig * 4}, {&b->recs, (size_t)count * b->cap * sizeof(bege_tail)},
              {&b->counters, (size_t)count * 8}};
  for (auto& nd : need) {
    int rc = ctx->alloc(nd.d, nd.bytes);
    if (rc) {
      destroy_batch(ctx, b.get());
      return rc;
    }
  }
  std::vector<bege::SegJob> jobs;
  size_t oy = 0, oD = 0, oAB = 0;
  cudaError_t e = cudaSuccess;
  for (int32_t i = 0; i < count && e == cudaSuccess; ++i) {
    const auto& en = b->entries[i];
    Bank* bank = ctx->banks[en.bank].get();
    float* y = static_cast<float*>(b->y.ptr) + oy;
    float2* D = static_cast<float2*>(b->D.ptr) + oD;
    float4* AB = static_cast<float4*>(b->AB.ptr) + oAB;
    e = cudaMemcpyAsync(y, entries[i].strain, en.n * sizeof(float), cudaMemcpyHostToDevice, us);
    const int S = (int)(en.n / 8192);
    bege::BatchSeg sg{};
    sg.AB = AB;
    sg.bank = static_cast<const float*>(bank->w.ptr);
    sg.Lp = bank->Lp;
    sg.k0 = en.k0;
    sg.k1 = en.k1;
    sg.kappa = en.kappa;
    sg.S = S;
    sg.sigma = static_cast<float*>(b->sigma.ptr) + b->sigma_off[i];
    sg.recs = static_cast<bege_tail*>(b->recs.ptr) + (size_t)i * b->cap;
    sg.cap = b->cap;
    sg.counter = static_cast<unsigned long long*>(b->counters.ptr) + i;
    b->segs_host.push_back(sg);
    for (int r = 0; r < S / 2; ++r) jobs.push_back({y, D, AB, S, r});
    oy += en.n;
    oD += en.n / 2 + 1;
    oAB += en.n / 2;
  }
  if (e == cudaSuccess)
    e = cudaMemcpyAsync(b->segs.ptr, b->segs_host.data(), count * sizeof(bege::BatchSeg),
                        cudaMemcpyHostToDevice, us);
  int rc = BEGE_OK;
  if (e == cudaSuccess) rc = ctx->alloc(&b->jobs, jobs.size() * sizeof(bege::SegJob));
  if (e == cudaSuccess && !rc)
    e = cudaMemcpyAsync(b->jobs.ptr, jobs.data(), jobs.size() * sizeof(bege::SegJob),
                        cudaMemcpyHostToDevice, us);
  if (e == cudaSuccess && !rc) e = cudaStreamSynchronize(us);
  if (e == cudaSuccess && !rc) e = cudaStreamCreateWithFlags(&b->cs, cudaStreamNonBlocking);
  if (e == cudaSuccess && !rc) e = cudaEventCreateWithFlags(&b->done, cudaEventDisableTiming);
  if (e == cudaSuccess && !rc) e = cudaEventCreate(&b->t0);
  if (e == cudaSuccess && !rc) e = cudaEventCreate(&b->t1);
  if (e != cudaSuccess || rc) {
    destroy_batch(ctx, b.get());
    return rc ? rc : cuda_fail(e, "batch setup");
  }
  b->n_jobs = (int)jobs.size();
  b->args.segs = static_cast<const bege::BatchSeg*>(b->segs.ptr);
  b->args.queue = static_cast<unsigned int*>(b->queue.ptr);
  rc = batch_build(ctx, b.get());
  if (rc) {
    destroy_batch(ctx, b.get());
    return rc;
  }
  const int32_t id = ctx->next_id++;
  ctx->batches[id] = std::move(b);
  *batch_id = id;
  return BEGE_OK;
}

int bege_batch_run(bege_ctx* ctx, int32_t batch_id, void* stream) {
  if (!ctx) return fail(BEGE_EINVAL, "NULL argument");
  DeviceGuard dg(ctx->device);
  std::lock_guard<std::mutex> lk(ctx->mu);
  Batch* b = find_batch(ctx, batch_id);
  if (!b) return fail(BEGE_EINVAL, "unknown batch handle");
  return batch_run_locked(b, static_cast<cudaStream_t>(stream));
}

int bege_batch_elapsed_ms(bege_ctx* ctx, int32_t batch_id, float* ms) {
  if (!ctx || !ms) return fail(BEGE_EINVAL, "NULL argument");
  DeviceGuard dg(ctx->device);
  std::lock_guard<std::mutex> lk(ctx->mu);
  Batch* b = find_batch(ctx, batch_id);
  if (!b) return fail(BEGE_EINVAL, "unknown batch handle");
  int rc = batch_wait(b);
  if (rc) return rc;
  cudaError_t e = cudaEventElapsedTime(ms, b->t0, b->t1);
  if (e != cudaSuccess) return cuda_fail(e, "batch time");
  return BEGE_OK;
}

int bege_batch_fetch_tails(bege_ctx* ctx, int32_t batch_id, int32_t entry, bege_tail* out,
                           int64_t capacity, int64_t* n_written, int64_t* n_total) {
  if (!ctx || !n_written || !n_total) return fail(BEGE_EINVAL, "NULL argument");
  if (capacity < 0 || (capacity > 0 && !out)) return fail(BEGE_EINVAL, "bad output buffer");
  DeviceGuard dg(ctx->device);
  std::lock_guard<std::mutex> lk(ctx->mu);
  Batch* b = find_batch(ctx, batch_id);
  if (!b) return fail(BEGE_EINVAL, "unknown batch handle");
  if (entry < 0 || entry >= (int32_t)b->entries.size()) return fail(BEGE_EINVAL, "bad entry");
  int rc = batch_wait(b);
  if (rc) return rc;
  unsigned long long total = 0;
  cudaError_t e = cudaMemcpy(&total, static_cast<unsigned long long*>(b->counters.ptr) + entry,
                             sizeof(total), cudaMemcpyDeviceToHost);
  if (e != cudaSuccess) return cuda_fail(e, "tail count");
  uint64_t ncopy = std::min<uint64_t>(std::min<uint64_t>(total, b->cap), (uint64_t)capacity);
  if (ncopy) {
    e = cudaMemcpy(out, static_cast<bege_tail*>(b->recs.ptr) + (size_t)entry * b->cap,
                   ncopy * sizeof(bege_tail), cudaMemcpyDeviceToHost);
    if (e != cudaSuccess) return cuda_fail(e, "tail records");
  }
  *n_written = (int64_t)ncopy;
  *n_total = (int64_t)total;
  if (ncopy < total) return fail(BEGE_EOVERFLOW, "more tails than copied");
  return BEGE_OK;
}

int bege_batch_get_sigma(bege_ctx* ctx, int32_t batch_id, int32_t entry, float* out,
                         int64_t count) {
  if (!ctx || !out) return fail(BEGE_EINVAL, "NULL argument");
  DeviceGuard dg(ctx->device);
  std::lock_guard<std::mutex> lk(ctx->mu);
  Batch* b = find_batch(ctx, batch_id);
  if (!b) return fail(BEGE_EINVAL, "unknown batch handle");
  if (entry < 0 || entry >= (int32_t)b->entries.size()) return fail(BEGE_EINVAL, "bad entry");
  if (count != b->entries[entry].k1 - b->entries[entry].k0)
    return fail(BEGE_EINVAL, "count must equal k_end - k_begin");
  int rc = batch_wait(b);
  if (rc) return rc;
  cudaError_t e = cudaMemcpy(out, static_cast<float*>(b->sigma.ptr) + b->sigma_off[entry],
                             (size_t)count * sizeof(float), cudaMemcpyDeviceToHost);
  if (e != cudaSuccess) return cuda_fail(e, "sigma");
  return BEGE_OK;
}

int bege_batch_set_plan(bege_ctx* ctx, int32_t batch_id, int32_t plan, int64_t chunk,
                        int32_t order) {
  if (!ctx) return fail(BEGE_EINVAL, "NULL argument");
  if (plan < 0 || plan > 1 || chunk < 1 || order < 0 || order > 1)
    return fail(BEGE_EINVAL, "bad plan");
  DeviceGuard dg(ctx->device);
  std::lock_guard<std::mutex> lk(ctx->mu);
  Batch* b = find_batch(ctx, batch_id);
  if (!b) return fail(BEGE_EINVAL, "unknown batch handle");
  if (b->done) cudaEventSynchronize(b->done);
  b->plan = plan;
  b->chunk = chunk;
  b->order = order;
  return batch_build(ctx, b);
}

int bege_batch_get_plan(bege_ctx* ctx, int32_t batch_id, int32_t* plan, int64_t* chunk,
                        int32_t* order) {
  if (!ctx || !plan || !chunk || !order) return fail(BEGE_EINVAL, "NULL argument");
  std::lock_guard<std::mutex> lk(ctx->mu);
  Batch* b = find_batch(ctx, batch_id);
  if (!b) return fail(BEGE_EINVAL, "unknown batch handle");
  *plan = b->plan;
  *chunk = b->chunk;
  *order = b->order;
  return BEGE_OK;
}

int bege_batch_autotune(bege_ctx* ctx, int32_t batch_id, int32_t reps, void* stream,
                        float* best_ms) {
  if (!ctx || !best_ms || reps < 1) return fail(BEGE_EINVAL, "bad argument");
  DeviceGuard dg(ctx->device);
  std::lock_guard<std::mutex> lk(ctx->mu);
  Batch* b = find_batch(ctx, batch_id);
  if (!b) return fail(BEGE_EINVAL, "unknown batch handle");
  cudaStream_t s = static_cast<cudaStream_t>(stream);
  struct Cand {
    int32_t plan;
    int64_t chunk;
    int32_t order;
  };
  std::vector<Cand> cands;
  for (int64_t c : {64, 128, 256, 512, 1024, 2048})
    for (int32_t o : {0, 1}) cands.push_back({0, c, o});
  cands.push_back({1, b->chunk, 0});
  // the per-segment plan is kept only if it beats the best persistent
  // candidate by more than 1%: within timing noise the single launch wins
  constexpr float kMargin = 0.99f;
  float best = 0.f;
  Cand pick = cands[0];
  for (size_t i = 0; i < cands.size(); ++i) {
    b->plan = cands[i].plan;
    b->chunk = cands[i].chunk;
    b->order = cands[i].order;
    int rc = batch_build(ctx, b);
    if (rc) return rc;
    std::vector<float> t;
    for (int r = 0; r <= reps; ++r) {
      rc = batch_run_locked(b, s);
      if (rc) return rc;
      cudaError_t e = cudaEventSynchronize(b->done);
      float ms = 0.f;
      if (e == cudaSuccess) e = cudaEventElapsedTime(&ms, b->t0, b->t1);
      if (e != cudaSuccess) return cuda_fail(e, "batch autotune");
      if (r > 0) t.push_back(ms);
    }
    std::sort(t.begin(), t.end());
    const float med = t[t.size() / 2];
    const bool better = cands[i].plan == 1 ? med < kMargin * best : med < best;
    if (i == 0 || better) {
      best = med;
      pick = cands[i];
    }
  }
  b->plan = pick.plan;
  b->chunk = pick.chunk;
  b->order = pick.order;
  *best_ms = best;
  return batch_build(ctx, b);
}

int bege_release(bege_ctx* ctx, int32_t handle) {
  if (!ctx) return fail(BEGE_EINVAL, "NULL argument");
  DeviceGuard dg(ctx->device);
  std::lock_guard<std::mutex> lk(ctx->mu);
  auto ji = ctx->jobs.find(handle);
  if (ji != ctx->jobs.end()) {
    wait_done(ji->second.get());
    ctx->release(&ji->second->proj);
    ctx->release(&ji->second->scratch);
    ctx->give_back(std::move(ji->second->buf));
    ctx->jobs.erase(ji);
    return BEGE_OK;
  }
  auto bti = ctx->batches.find(handle);
  if (bti != ctx->batches.end()) {
    destroy_batch(ctx, bti->second.get());
    ctx->batches.erase(bti);
    return BEGE_OK;
  }
  auto si = ctx->segs.find(handle);
  if (si != ctx->segs.end()) {
    // what may still use the segment: its own kernel, jobs not released yet
    if (!si->second->loaded) cudaDeviceSynchronize();
    for (auto& kv : ctx->jobs)
      if (kv.second->seg == handle) wait_done(kv.second.get());
    ctx->keep(&si->second->D);
    ctx->keep(&si->second->AB);
    ctx->segs.erase(si);
    return BEGE_OK;
  }
  auto bi = ctx->banks.find(handle);
  if (bi != ctx->banks.end()) {
    cudaDeviceSynchronize();
    ctx->release(&bi->second->w);
    ctx->banks.erase(bi);
    return BEGE_OK;
  }
  return fail(BEGE_EINVAL, "unknown handle");
}

}  // extern "C"
