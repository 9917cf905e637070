// C ABI of the AET-SGD hot-path library: handle, device memory, and the run
// loop that turns the integer schedule into waves of kernel launches.
#include <cuda_runtime.h>
#include <math.h>
#include <string.h>

#include <chrono>
#include <mutex>
#include <new>
#include <string>
#include <thread>
#include <unordered_map>
#include <vector>

#include "../../include/aet.h"
#include "aet_kernels.h"
#include "aet_rng.h"
#include "aet_schedule.h"

using namespace aet;

namespace {

thread_local std::string g_create_error;

// Device memory of destroyed handles, kept for the next one: cudaMalloc and cudaFree of a handle's dozen arrays cost a
// short job (create, load, run, destroy) more than its run - milliseconds, at times tens of them.  Bounded per process,
// given back to the driver by aet_release_memory and whenever an allocation fails, never grown past the bound; blocks come
// back only after the device has been synchronised, so any stream may use them next.
class DevicePool {
 public:
  void* get(size_t bytes) {
    int dev = 0;
    if (cudaGetDevice(&dev) != cudaSuccess) { cudaGetLastError(); return nullptr; }
    bytes = (bytes + 511) & ~(size_t)511;
    std::lock_guard<std::mutex> lock(mu_);
    size_t best = free_.size();
    for (size_t i = 0; i < free_.size(); ++i)   // smallest block that fits without wasting more than itself
      if (free_[i].dev == dev && free_[i].bytes >= bytes && free_[i].bytes <= 2 * bytes + 65536 &&
          (best == free_.size() || free_[i].bytes < free_[best].bytes)) best = i;
    if (best < free_.size()) {
      const Block b = free_[best];
      free_.erase(free_.begin() + best);
      held_ -= b.bytes;
      live_[b.p] = b;
      return b.p;
    }
    void* p = nullptr;
    if (cudaMalloc(&p, bytes) != cudaSuccess) {
      cudaGetLastError();
      flush();
      if (cudaMalloc(&p, bytes) != cudaSuccess) { cudaGetLastError(); return nullptr; }
    }
    live_[p] = Block{p, bytes, dev};
    return p;
  }
  // The caller has synchronised the device since the block's last use.
  void put(void* p) {
    if (!p) return;
    std::lock_guard<std::mutex> lock(mu_);
    auto it = live_.find(p);
    if (it == live_.end()) return;
    const Block b = it->second;
    live_.erase(it);
    if (b.bytes > kMost) { cudaFree(p); return; }
    while (held_ + b.bytes > kMost || free_.size() >= kMostBlocks) {   // over the bound the oldest go: the next handle is most like the last
      cudaFree(free_.front().p);
      held_ -= free_.front().bytes;
      free_.erase(free_.begin());
    }
    held_ += b.bytes;
    free_.push_back(b);
  }
  void release() {   // everything no handle holds, back to the driver
    std::lock_guard<std::mutex> lock(mu_);
    flush();
  }

 private:
  struct Block { void* p; size_t bytes; int dev; };
  static constexpr size_t kMost = 512ull << 20, kMostBlocks = 128;
  void flush() {
    for (const Block& b : free_) cudaFree(b.p);
    free_.clear();
    held_ = 0;
  }
  std::mutex mu_;
  std::vector<Block> free_;   // in the order they came back
  std::unordered_map<void*, Block> live_;
  size_t held_ = 0;
};
DevicePool& pool() {
  static DevicePool* p = new DevicePool;   // outlives every handle; the driver takes its blocks back with the process
  return *p;
}

// A few pinned blocks for small read-backs, shared by all handles and threads; kept until aet_release_memory.
class PinnedPool {
 public:
  static constexpr size_t kBlock = 64 << 10;
  void* get() {   // null: none to be had, go without
    {
      std::lock_guard<std::mutex> lock(mu_);
      if (!free_.empty()) {
        void* p = free_.back();
        free_.pop_back();
        return p;
      }
      if (made_ >= kMost) return nullptr;
      ++made_;
    }
    void* p = nullptr;
    if (cudaHostAlloc(&p, kBlock, cudaHostAllocPortable) != cudaSuccess) {
      cudaGetLastError();
      std::lock_guard<std::mutex> lock(mu_);
      --made_;
      return nullptr;
    }
    return p;
  }
  void put(void* p) {
    std::lock_guard<std::mutex> lock(mu_);
    free_.push_back(p);
  }
  void release() {
    std::lock_guard<std::mutex> lock(mu_);
    for (void* p : free_) cudaFreeHost(p);
    made_ -= (int)free_.size();
    free_.clear();
  }

 private:
  static constexpr int kMost = 16;
  std::mutex mu_;
  std::vector<void*> free_;
  int made_ = 0;
};
PinnedPool& pinned() {
  static PinnedPool* p = new PinnedPool;
  return *p;
}

// Bump allocator over a few large device chunks: client data sets are many
// small allocations of unknown count, and cudaMalloc per client is slow.
struct Arena {
  std::vector<void*> chunks;
  char* cur = nullptr;
  size_t left = 0;
  // Chunks of 8 to 256 MB: the first as large as the first client's arrays say that all of them will be, so that neither a small
  // job takes much nor a large one many (a chunk costs 0.3 to 0.6 ms), the next ones growing if that was too little.
  static constexpr size_t kLeast = 8ull << 20, kMost = 256ull << 20;
  size_t next = kLeast;
  void expect(size_t bytes) {
    if (chunks.empty()) next = bytes < kLeast ? kLeast : bytes > kMost ? kMost : (bytes + kLeast - 1) / kLeast * kLeast;
  }
  void* alloc(size_t bytes) {
    bytes = (bytes + 255) & ~(size_t)255;
    if (bytes > left) {
      size_t want = bytes > next ? bytes : next;
      if (next < kMost) next = next * 4 < kMost ? next * 4 : kMost;
      void* p = pool().get(want);
      if (!p) return nullptr;
      chunks.push_back(p);
      cur = (char*)p;
      left = want;
    }
    void* r = cur;
    cur += bytes;
    left -= bytes;
    return r;
  }
  void release() {
    for (void* p : chunks) pool().put(p);
    chunks.clear();
    cur = nullptr;
    left = 0;
  }
};

template <class T>
struct DevBuf {  // grow-only device array
  T* p = nullptr;
  size_t cap = 0;
  bool reserve(size_t n) {
    if (n <= cap) return true;
    if (p) { cudaDeviceSynchronize(); release(); }   // an earlier launch may still use the old array
    p = static_cast<T*>(pool().get(n * sizeof(T)));
    if (!p) return false;
    cap = n;
    return true;
  }
  void release() { pool().put(p); p = nullptr; cap = 0; }
};

struct CachedRingPlan {
  bool valid = false, uploaded = false;
  uint32_t rounds_before = 0, n_rounds = 0;
  RingState before, after;
  RingResult sched;
  RingPlan plan;
};

struct CachedPlan {
  bool valid = false, uploaded = false;
  uint32_t rounds_before = 0, n_rounds = 0;
  SchedState before, after;
  SchedResult sched;
  Plan plan;
};

}  // namespace

namespace aet {
// Lets other translation units of the library set the text aet_last_error(NULL) returns.
void set_thread_error(const std::string& msg) { g_create_error = msg; }
}  // namespace aet

struct aet_handle {
  aet_config cfg{};
  int device = 0;
  std::vector<uint32_t> shares;   // copy of cfg.client_shares (cfg.client_shares points here)
  uint32_t P = 0;
  size_t stride = 0;
  bool lr_fast = false;  // 784 -> 10, batch 1, fp32: the specialised kernel
  bool cnn = false;      // model 2: the small convolutional classifier
  MlpShape shape{};
  CnnShape cshape{};
  size_t act_floats() const { return cnn ? cnn_act_floats(cshape) : mlp_act_floats(shape); }
  std::string err;

  SchedState st;
  RingState rst;                  // topology 1
  DelayCache delays;
  CachedPlan cached;
  CachedRingPlan ring_cached;
  // aet_prepare_rounds: schedule and launch plan of the next run computed by a host thread of its own, on copies
  // of the scheduling state; aet_run_rounds takes the result over if it still fits.
  std::thread prep_thread;
  CachedPlan prep;
  CachedRingPlan prep_ring;
  DelayCache prep_delays;
  bool prep_ok = false;
  std::vector<RingTask> last_ring_tasks;
  std::vector<aet_event> log;
  aet_summary total{};

  Arena arena;
  std::vector<ClientData> h_clients;
  std::vector<uint64_t> keys;
  DevBuf<ClientData> d_clients;
  DevBuf<uint64_t> d_keys;
  DevBuf<uint32_t> d_H;
  DevBuf<float> w, w0, snaps, U, work, act, dbg;
  DevBuf<float> node_w;           // topology 1: [n_clients, stride], every node's own model
  DevBuf<RingApplyDesc> d_ring_applies;
  DevBuf<RingOp> d_ring_ops;
  float* w_cur() { return w.p; }   // the server model
  uint32_t* d_status() { return reinterpret_cast<uint32_t*>(w.p + stride); }   // what kernels report, right behind it: read back together
  DevBuf<TaskDesc> d_tasks;
  DevBuf<char> d_plan;            // topology 0: the plan's tasks, sums in flight and updates
  std::vector<char> pack;         // the same on the host, for the copy
  DevBuf<TriggerRec> d_trig;
  DevBuf<ApplyRec> d_alog;
  bool clients_dirty = true, have_w0 = false;

  // most recent run, for the device-record cross-check and aet_get_update_sum
  size_t last_first_event = 0, last_n_events = 0;
  bool last_checked = true;
  std::vector<uint32_t> last_H_before;
  cudaStream_t last_stream = nullptr;

  bool timing = false;
  aet_stats stats{};
  struct Timed { cudaEvent_t a, b; int id; };
  std::vector<Timed> timed;
  std::vector<cudaEvent_t> ev_pool;
};

namespace {

aet_status fail(aet_handle* h, aet_status s, const std::string& msg) {
  if (h) h->err = msg; else g_create_error = msg;
  return s;
}
aet_status cuda_fail(aet_handle* h, cudaError_t e, const char* what) {
  cudaGetLastError();
  return fail(h, AET_ERR_CUDA, std::string(what) + ": " + cudaGetErrorString(e));
}
#define AET_CUDA(h, call)                                         \
  do {                                                            \
    cudaError_t e_ = (call);                                      \
    if (e_ != cudaSuccess) return cuda_fail(h, e_, #call);        \
  } while (0)

uint32_t count_params(const aet_config& c) {
  uint64_t p = 0;
  for (uint32_t l = 0; l < c.n_layers; ++l) p += (uint64_t)c.dims[l] * c.dims[l + 1] + c.dims[l + 1];
  return p > 0xFFFFFFFFull ? 0 : (uint32_t)p;
}

cudaEvent_t get_event(aet_handle* h) {
  if (!h->ev_pool.empty()) { cudaEvent_t e = h->ev_pool.back(); h->ev_pool.pop_back(); return e; }
  cudaEvent_t e = nullptr;
  cudaEventCreate(&e);
  return e;
}

struct KernelTimer {  // records a pair of events around a launch when timing is on
  aet_handle* h; cudaStream_t s; int id; cudaEvent_t a = nullptr;
  KernelTimer(aet_handle* h_, cudaStream_t s_, int id_) : h(h_), s(s_), id(id_) {
    h->stats.launches[id] += 1;
    if (h->timing) { a = get_event(h); cudaEventRecord(a, s); }
  }
  ~KernelTimer() {
    if (h->timing) { cudaEvent_t b = get_event(h); cudaEventRecord(b, s); h->timed.push_back({a, b, id}); }
  }
};

void collect_timings(aet_handle* h) {
  for (auto& t : h->timed) {
    float ms = 0.f;
    if (cudaEventSynchronize(t.b) == cudaSuccess && cudaEventElapsedTime(&ms, t.a, t.b) == cudaSuccess)
      h->stats.kernel_ms[t.id] += ms;
    h->ev_pool.push_back(t.a);
    h->ev_pool.push_back(t.b);
  }
  h->timed.clear();
}

aet_status upload_clients(aet_handle* h, cudaStream_t s) {
  if (!h->clients_dirty) return AET_OK;
  const uint32_t n = h->cfg.n_clients;
  if (!h->d_clients.reserve(n) || !h->d_keys.reserve(n)) return fail(h, AET_ERR_NOMEM, "device allocation failed");
  std::vector<uint64_t>& keys = h->keys;
  keys.resize(n);
  for (uint32_t c = 0; c < n; ++c) keys[c] = stream_key(h->cfg.seed, kStreamSample, c);
  AET_CUDA(h, cudaMemcpyAsync(h->d_clients.p, h->h_clients.data(), n * sizeof(ClientData), cudaMemcpyHostToDevice, s));
  AET_CUDA(h, cudaMemcpyAsync(h->d_keys.p, keys.data(), n * sizeof(uint64_t), cudaMemcpyHostToDevice, s));
  h->clients_dirty = false;
  return AET_OK;
}

// What a status word read from the device says.
aet_status judge_status(aet_handle* h, uint32_t st) {
  if (st) cudaMemset(h->d_status(), 0, sizeof(uint32_t));
  if (st & 1u) return fail(h, AET_ERR_TIMEOUT, "a bounded wait for an asynchronous row copy gave up; results are invalid");
  if (st & 4u) return fail(h, AET_ERR_STATE, "a debug check failed on the device: a label, row number or slot was out of range; results are invalid");
  if (st & 2u) return fail(h, AET_ERR_NUMERIC, "a non-finite value reached the server model (or, with debug checks, sits in a client's rows); results are invalid");
  return AET_OK;
}
// After a synchronisation: did a bounded device-side wait give up?
aet_status check_device_status(aet_handle* h) {
  uint32_t st = 0;
  AET_CUDA(h, cudaMemcpy(&st, h->d_status(), sizeof(st), cudaMemcpyDeviceToHost));
  return judge_status(h, st);
}

// A model out of the device, once the stream is done and the status word is clean; `out` stays untouched on error.  Small
// models come with the status word through pinned memory: one wait instead of three.
aet_status read_model(aet_handle* h, const float* src, float* out, cudaStream_t s) {
  const size_t bytes = (size_t)h->P * sizeof(float);
  cudaPointerAttributes attr{};
  const bool known = cudaPointerGetAttributes(&attr, out) == cudaSuccess;
  cudaGetLastError();
  const bool to_host = known && (attr.type == cudaMemoryTypeHost || attr.type == cudaMemoryTypeUnregistered);
  const size_t row = h->stride * sizeof(float);
  void* pin = to_host && row + 16 <= PinnedPool::kBlock ? pinned().get() : nullptr;
  if (pin) {
    uint32_t* st = reinterpret_cast<uint32_t*>(static_cast<char*>(pin) + row);
    cudaError_t e;
    if (src == h->w_cur()) {
      e = cudaMemcpyAsync(pin, src, row + sizeof(uint32_t), cudaMemcpyDeviceToHost, s);
    } else {
      e = cudaMemcpyAsync(pin, src, bytes, cudaMemcpyDeviceToHost, s);
      if (e == cudaSuccess) e = cudaMemcpyAsync(st, h->d_status(), sizeof(uint32_t), cudaMemcpyDeviceToHost, s);
    }
    const cudaError_t w = cudaStreamSynchronize(s);   // (also before the block goes back)
    if (e == cudaSuccess) e = w;
    aet_status r = e == cudaSuccess ? judge_status(h, *st) : cuda_fail(h, e, "reading a model");
    if (r == AET_OK) memcpy(out, pin, bytes);
    pinned().put(pin);
    return r;
  }
  AET_CUDA(h, cudaStreamSynchronize(s));
  if (aet_status ds = check_device_status(h)) return ds;
  AET_CUDA(h, cudaMemcpyAsync(out, src, bytes, cudaMemcpyDefault, s));
  AET_CUDA(h, cudaStreamSynchronize(s));
  return AET_OK;
}

uint32_t longest_round(const TaskDesc* t, uint32_t n) {   // (the kernels' choice asks for it where there are few)
  uint32_t most = 0;
  for (uint32_t i = 0; n <= 32 && i < n; ++i) most = std::max(most, t[i].n_samples);
  return most;
}

aet_status launch_rounds(aet_handle* h, const RoundLaunch& r, cudaStream_t s) {
  KernelTimer kt(h, s, 0);
  cudaError_t e;
  if (h->lr_fast) {
    e = launch_lr_rounds(r, s);
  } else if (h->cnn) {
    CnnLaunch m;
    m.r = r;
    m.shape = h->cshape;
    m.act = h->act.p;
    m.act_stride = cnn_act_floats(h->cshape);
    e = launch_cnn_rounds(m, s);
  } else {
    MlpLaunch m;
    m.r = r;
    m.shape = h->shape;
    m.work = h->work.p;
    m.act = h->act.p;
    m.act_stride = mlp_act_floats(h->shape);
    e = launch_mlp_rounds(m, s);
  }
  if (e != cudaSuccess) return cuda_fail(h, e, "local-SGD kernel launch");
  return AET_OK;
}

// Waits for the thread aet_prepare_rounds started, if any.
void join_prepare(aet_handle* h) {
  if (h->prep_thread.joinable()) h->prep_thread.join();
}

// Peer-to-peer ring: waves of round-tasks (each from its node's own model), and before every wave
// the Receive step of the nodes about to start; after the last wave every node takes what is left.
aet_status run_ring_rounds(aet_handle* h, uint32_t n_rounds, cudaStream_t s) {
  auto t0 = std::chrono::steady_clock::now();
  CachedRingPlan& cp = h->ring_cached;
  if (h->prep_ok && h->prep_ring.valid && h->prep_ring.rounds_before == h->rst.rounds_done && h->prep_ring.n_rounds == n_rounds &&
      h->prep_ring.before.clock == h->rst.clock && h->prep_ring.before.H == h->rst.H) {
    cp = std::move(h->prep_ring);   // prepared by aet_prepare_rounds for exactly this state
    h->delays = std::move(h->prep_delays);
  }
  h->prep_ok = false;
  if (!(cp.valid && cp.rounds_before == h->rst.rounds_done && cp.n_rounds == n_rounds &&
        cp.before.clock == h->rst.clock && cp.before.H == h->rst.H)) {
    cp.valid = false;
    cp.uploaded = false;
    cp.before = h->rst;
    cp.rounds_before = h->rst.rounds_done;
    cp.n_rounds = n_rounds;
    RingState st = h->rst;
    std::string err;
    if (!simulate_ring(h->cfg, n_rounds, st, h->delays, cp.sched, err)) return fail(h, AET_ERR_CONFIG, err);
    cp.after = st;
    build_ring_plan(h->cfg, h->delays, cp.sched, (h->cfg.flags & AET_FLAG_KEEP_UPDATE_SUMS) != 0, cp.plan);
    cp.valid = true;
  }
  const RingPlan& plan = cp.plan;
  const size_t T = cp.sched.tasks.size();
  h->stats.plan_ms = std::chrono::duration<double, std::milli>(std::chrono::steady_clock::now() - t0).count();

  aet_status st_up = upload_clients(h, s);
  if (st_up != AET_OK) return st_up;
  bool ok = h->U.reserve((size_t)plan.n_u_rows * h->stride) && h->d_tasks.reserve(T) && h->d_trig.reserve(T) &&
            h->d_ring_applies.reserve(plan.applies.size() + 1) && h->d_ring_ops.reserve(plan.ops.size() + 1);
  if (ok && !h->lr_fast) ok = h->act.reserve((size_t)plan.max_wave_tasks * h->act_floats());
  if (!ok) return fail(h, AET_ERR_NOMEM, "device allocation failed");
  if (!cp.uploaded) {   // (a copy from pageable memory has read its source when it returns: no need to wait)
    AET_CUDA(h, cudaMemcpyAsync(h->d_tasks.p, plan.tasks.data(), T * sizeof(TaskDesc), cudaMemcpyHostToDevice, s));
    if (!plan.applies.empty())
      AET_CUDA(h, cudaMemcpyAsync(h->d_ring_applies.p, plan.applies.data(), plan.applies.size() * sizeof(RingApplyDesc), cudaMemcpyHostToDevice, s));
    if (!plan.ops.empty())
      AET_CUDA(h, cudaMemcpyAsync(h->d_ring_ops.p, plan.ops.data(), plan.ops.size() * sizeof(RingOp), cudaMemcpyHostToDevice, s));
    cp.uploaded = true;
  }
  AET_CUDA(h, cudaMemsetAsync(h->d_trig.p, 0, T * sizeof(TriggerRec), s));

  RoundLaunch r{};
  r.tasks = h->d_tasks.p; r.inflight = nullptr; r.clients = h->d_clients.p;
  r.sample_keys = h->d_keys.p; r.snaps = h->node_w.p; r.U = h->U.p; r.w_end = nullptr;
  r.trig = h->d_trig.p; r.status = h->d_status(); r.stride = h->stride; r.l2 = h->cfg.l2;
  r.debug_checks = (h->cfg.flags & AET_FLAG_DEBUG_CHECKS) ? 1u : 0u;
  r.step_by_step = (h->cfg.flags & AET_FLAG_STEPWISE_RECURRENCE) ? 1u : 0u;
  r.n_u_rows = plan.n_u_rows; r.n_snap = h->cfg.n_clients;
  RingApplyLaunch a{};
  a.applies = h->d_ring_applies.p; a.ops = h->d_ring_ops.p; a.U = h->U.p; a.node_w = h->node_w.p;
  a.status = h->d_status(); a.stride = h->stride; a.n_params = h->P;

  const uint32_t n_waves = (uint32_t)plan.wave_off.size() - 1;
  for (uint32_t L = 0; L <= n_waves; ++L) {
    a.lo = plan.apply_off[L]; a.hi = plan.apply_off[L + 1];
    if (a.hi > a.lo) {
      KernelTimer kt(h, s, 1);
      cudaError_t e = launch_ring_apply(a, s);
      if (e != cudaSuccess) return cuda_fail(h, e, "ring receive kernel launch");
    }
    if (L == n_waves) break;
    r.task_begin = plan.wave_off[L];
    r.n_tasks = plan.wave_off[L + 1] - plan.wave_off[L];
    r.longest = longest_round(plan.tasks.data() + r.task_begin, r.n_tasks);
    aet_status rs = launch_rounds(h, r, s);
    if (rs != AET_OK) return rs;
  }
  h->stats.waves = n_waves;

  h->last_first_event = h->log.size();
  h->last_n_events = T;                 // update sums are indexed by round-task here
  h->last_ring_tasks = cp.sched.tasks;
  h->last_checked = false;
  h->last_stream = s;
  h->log.insert(h->log.end(), cp.sched.events.begin(), cp.sched.events.end());
  const aet_summary& q = cp.sched.summary;
  h->total.messages_up += q.messages_up; h->total.model_pulls += q.model_pulls;
  h->total.samples_total += q.samples_total; h->total.messages_if_per_sample += q.messages_if_per_sample;
  h->total.messages_if_constant_b += q.messages_if_constant_b; h->total.t_end_ticks = q.t_end_ticks;
  h->rst = cp.after;
  return AET_OK;
}

}  // namespace

extern "C" {

aet_status aet_create(const aet_config* cfg, aet_handle** out) {
  if (!cfg || !out) return fail(nullptr, AET_ERR_ARG, "null argument");
  std::string err;
  if (cfg->struct_size != sizeof(aet_config)) return fail(nullptr, AET_ERR_ARG, "struct_size does not match sizeof(aet_config)");
  if (!validate_config(*cfg, err)) return fail(nullptr, AET_ERR_CONFIG, err);
  CnnShape cshape{};
  for (int i = 0; i < 8; ++i) cshape.dims[i] = cfg->dims[i];
  cshape.batch = cfg->batch;
  if (cfg->model == 2)
    if (const char* why = cnn_check_shape(cshape)) return fail(nullptr, AET_ERR_CONFIG, why);
  const uint32_t P = cfg->model == 2 ? cnn_n_params(cshape) : count_params(*cfg);
  if (!P) return fail(nullptr, AET_ERR_CONFIG, "model too large");
  if (cfg->dims[cfg->n_layers] > 32) return fail(nullptr, AET_ERR_CONFIG, "at most 32 classes are supported");
  if (cfg->flags & ~(uint32_t)(AET_FLAG_BORROW_DATA | AET_FLAG_DEBUG_CHECKS | AET_FLAG_KEEP_UPDATE_SUMS | AET_FLAG_STEPWISE_RECURRENCE))
    return fail(nullptr, AET_ERR_CONFIG, "unknown bit in flags");
  int dev = 0;
  cudaError_t ce = cudaGetDevice(&dev);
  if (ce != cudaSuccess) { cudaGetLastError(); return fail(nullptr, AET_ERR_CUDA, std::string("no CUDA device: ") + cudaGetErrorString(ce)); }
  aet_handle* h = new (std::nothrow) aet_handle();
  if (!h) return fail(nullptr, AET_ERR_NOMEM, "out of host memory");
  h->cfg = *cfg;
  h->device = dev;
  if (cfg->client_shares) {
    h->shares.assign(cfg->client_shares, cfg->client_shares + cfg->n_clients);
    h->cfg.client_shares = h->shares.data();
  }
  h->P = P;
  h->stride = ((size_t)P + 31) & ~(size_t)31;
  h->lr_fast = cfg->model == 0 && cfg->dims[0] == 784 && cfg->dims[1] == 10 && cfg->batch == 1 && cfg->precision == 0;
  h->shape.n_layers = cfg->n_layers;
  for (int i = 0; i < 8; ++i) h->shape.dims[i] = cfg->dims[i];
  h->shape.batch = cfg->batch;
  h->shape.precision = cfg->precision;
  h->shape.cluster = mlp_pick_cluster(h->shape, cfg->n_clients);
  h->cnn = cfg->model == 2;
  h->cshape = cshape;
  if (!h->lr_fast && !h->cnn && !mlp_tc_eligible(h->shape)) {
    if (const char* why = mlp_check_shape(h->shape)) { delete h; return fail(nullptr, AET_ERR_CONFIG, why); }
  }
  h->h_clients.assign(cfg->n_clients, ClientData{nullptr, nullptr, 0, 0});
  h->st.H.assign(cfg->n_clients, 0);
  bool ok = h->w.reserve(h->stride + 4) && h->w0.reserve(h->stride) &&
            h->d_H.reserve(cfg->n_clients);
  if (ok && !h->lr_fast && !h->cnn) ok = h->work.reserve((size_t)cfg->n_clients * h->stride);
  if (ok && cfg->topology == 1) ok = h->node_w.reserve((size_t)cfg->n_clients * h->stride);
  if (!ok) { aet_destroy(h); return fail(nullptr, AET_ERR_NOMEM, "device allocation failed"); }
  if (cfg->topology == 1 && cudaMemset(h->node_w.p, 0, (size_t)cfg->n_clients * h->stride * sizeof(float)) != cudaSuccess) {
    cudaError_t e = cudaGetLastError();
    aet_destroy(h);
    return fail(nullptr, AET_ERR_CUDA, std::string("cudaMemset: ") + cudaGetErrorString(e));
  }
  if (cudaMemset(h->w.p, 0, (h->stride + 4) * sizeof(float)) != cudaSuccess ||
      cudaMemset(h->w0.p, 0, h->stride * sizeof(float)) != cudaSuccess ||
      cudaMemset(h->d_H.p, 0, cfg->n_clients * sizeof(uint32_t)) != cudaSuccess) {
    cudaError_t e = cudaGetLastError();
    aet_destroy(h);
    return fail(nullptr, AET_ERR_CUDA, std::string("cudaMemset: ") + cudaGetErrorString(e));
  }
  *out = h;
  return AET_OK;
}

aet_status aet_destroy(aet_handle* h) {
  if (!h) return AET_ERR_ARG;
  join_prepare(h);
  int before = h->device;
  cudaGetDevice(&before);
  if (before != h->device) cudaSetDevice(h->device);
  cudaDeviceSynchronize();   // nothing uses the handle's memory any more when it goes back to the pool
  collect_timings(h);
  for (cudaEvent_t e : h->ev_pool) cudaEventDestroy(e);
  h->arena.release();
  h->d_clients.release(); h->d_keys.release(); h->d_H.release();
  h->w.release(); h->w0.release(); h->snaps.release(); h->U.release();
  h->work.release(); h->act.release(); h->dbg.release();
  h->node_w.release(); h->d_ring_applies.release(); h->d_ring_ops.release();
  h->d_tasks.release(); h->d_plan.release();
  h->d_trig.release(); h->d_alog.release();
  cudaGetLastError();
  if (before != h->device) cudaSetDevice(before);
  delete h;
  return AET_OK;
}

aet_status aet_release_memory(void) {
  pool().release();
  pinned().release();
  const cudaError_t e = cudaGetLastError();
  if (e != cudaSuccess) return fail(nullptr, AET_ERR_CUDA, std::string("releasing memory: ") + cudaGetErrorString(e));
  return AET_OK;
}

aet_status aet_reset(aet_handle* h, void* cuda_stream) {
  if (!h) return AET_ERR_ARG;
  join_prepare(h);
  cudaStream_t s = (cudaStream_t)cuda_stream;
  AET_CUDA(h, launch_copy_and_zero(h->w_cur(), h->w0.p, h->stride, h->d_H.p, h->cfg.n_clients, s));
  if (h->cfg.topology == 1)
    for (uint32_t c = 0; c < h->cfg.n_clients; ++c)
      AET_CUDA(h, cudaMemcpyAsync(h->node_w.p + (size_t)c * h->stride, h->w0.p, h->stride * sizeof(float), cudaMemcpyDeviceToDevice, s));
  h->rst = RingState{};
  h->st = SchedState{};
  h->st.H.assign(h->cfg.n_clients, 0);
  h->log.clear();
  h->total = aet_summary{};
  h->last_n_events = 0;
  h->last_checked = true;
  h->last_stream = s;
  return AET_OK;
}

aet_status aet_set_global_model(aet_handle* h, const float* w0, size_t n_params, void* cuda_stream) {
  if (!h || !w0) return h ? fail(h, AET_ERR_ARG, "null argument") : AET_ERR_ARG;
  if (n_params != h->P) return fail(h, AET_ERR_ARG, "n_params does not match the model");
  cudaStream_t s = (cudaStream_t)cuda_stream;
  AET_CUDA(h, cudaMemcpyAsync(h->w_cur(), w0, (size_t)h->P * sizeof(float), cudaMemcpyDefault, s));
  AET_CUDA(h, cudaMemcpyAsync(h->w0.p, h->w_cur(), (size_t)h->P * sizeof(float), cudaMemcpyDeviceToDevice, s));
  if (h->cfg.topology == 1)   // every node starts from it (Algorithm 2: the same initial model for all compute nodes)
    for (uint32_t c = 0; c < h->cfg.n_clients; ++c)
      AET_CUDA(h, cudaMemcpyAsync(h->node_w.p + (size_t)c * h->stride, h->w0.p, h->stride * sizeof(float), cudaMemcpyDeviceToDevice, s));
  AET_CUDA(h, cudaStreamSynchronize(s));
  h->have_w0 = true;
  h->last_stream = s;
  return AET_OK;
}

aet_status aet_load_client_data(aet_handle* h, uint32_t client, const void* x, const int32_t* y,
                                uint32_t n, void* cuda_stream) {
  if (!h) return AET_ERR_ARG;
  if (!x || !y) return fail(h, AET_ERR_ARG, "null data pointer");
  if (client >= h->cfg.n_clients) return fail(h, AET_ERR_ARG, "client index out of range");
  if (n == 0 || n < h->cfg.batch) return fail(h, AET_ERR_ARG, "a client needs at least max(1, batch) samples");
  cudaStream_t s = (cudaStream_t)cuda_stream;
  // a row: the input layer's width, or side * side * c_in values for the convolutional classifier
  const size_t D = h->cfg.model == 2 ? (size_t)h->cfg.dims[0] * h->cfg.dims[0] * h->cfg.dims[1] : h->cfg.dims[0];
  const size_t elems = (size_t)n * D;
  const bool bf16 = h->cfg.precision == 1;
  const bool debug = (h->cfg.flags & AET_FLAG_DEBUG_CHECKS) != 0;
  if ((h->cfg.flags & AET_FLAG_BORROW_DATA) && !bf16) {
    // D_c stays where the caller put it: both arrays must be device memory the kernels can read
    // with 16-byte row copies, and must stay alive and unchanged until aet_destroy.
    cudaPointerAttributes ax{}, ay{};
    const bool okx = cudaPointerGetAttributes(&ax, x) == cudaSuccess &&
                     (ax.type == cudaMemoryTypeDevice || ax.type == cudaMemoryTypeManaged);
    const bool oky = cudaPointerGetAttributes(&ay, y) == cudaSuccess &&
                     (ay.type == cudaMemoryTypeDevice || ay.type == cudaMemoryTypeManaged);
    cudaGetLastError();
    if (!okx || !oky) return fail(h, AET_ERR_ARG, "AET_FLAG_BORROW_DATA needs device pointers");
    if (((uintptr_t)x & 15) || ((D * 4) & 15) || ((uintptr_t)y & 3))
      return fail(h, AET_ERR_ARG, "AET_FLAG_BORROW_DATA needs 16-byte aligned rows");
    if (debug) AET_CUDA(h, launch_validate_data((const float*)x, y, n, (uint32_t)D, h->cfg.dims[h->cfg.n_layers], h->d_status(), s));
    h->h_clients[client] = ClientData{x, y, n, 0};
    h->clients_dirty = true;
    h->last_stream = s;
    return AET_OK;
  }
  h->arena.expect((elems * (bf16 ? 2 : 4) + (size_t)n * sizeof(int32_t) + 512) * h->cfg.n_clients);
  void* dx = h->arena.alloc(elems * (bf16 ? 2 : 4));
  int32_t* dy = (int32_t*)h->arena.alloc((size_t)n * sizeof(int32_t));
  if (!dx || !dy) return fail(h, AET_ERR_NOMEM, "device allocation failed");
  // Page-locked host arrays: the GPU fetches rows and labels itself.  A copy costs 5 us beside its bytes, two of them as much
  // as 500 KB; from 2.5 MB on (measured) the copy engine's higher rate wins, except that bf16 would need an fp32 copy first.
  constexpr size_t kFetchMost = 2 << 20;
  const void *px = nullptr, *py = nullptr;   // the arrays as the device sees them
  if ((bf16 || elems * 4 <= kFetchMost) && elems % 4 == 0) {
    // the whole array page-locked and in one piece as the device sees it: its last byte as far from the first there as here
    auto seen = [](const void* from, size_t bytes) -> const void* {
      cudaPointerAttributes first{}, last{};
      const char* end = static_cast<const char*>(from) + bytes - 1;
      const bool ok = cudaPointerGetAttributes(&first, from) == cudaSuccess && first.type == cudaMemoryTypeHost && first.devicePointer &&
                      cudaPointerGetAttributes(&last, end) == cudaSuccess && last.type == cudaMemoryTypeHost && last.devicePointer &&
                      static_cast<const char*>(last.devicePointer) - static_cast<const char*>(first.devicePointer) == (ptrdiff_t)bytes - 1;
      cudaGetLastError();
      return ok ? first.devicePointer : nullptr;
    };
    const void* sx = seen(x, elems * 4);
    const void* sy = sx ? seen(y, (size_t)n * sizeof(int32_t)) : nullptr;
    if (sx && sy && !((uintptr_t)sx & 15) && !((uintptr_t)sy & 3)) {
      px = sx;
      py = sy;
    }
  }
  if (px) {
    AET_CUDA(h, launch_fetch_client(static_cast<const float*>(px), dx, bf16, elems / 4, static_cast<const int32_t*>(py), dy, n, s));
  } else if (!bf16) {
    AET_CUDA(h, cudaMemcpyAsync(dx, x, elems * 4, cudaMemcpyDefault, s));
  } else {
    cudaPointerAttributes attr{};
    cudaError_t pe = cudaPointerGetAttributes(&attr, x);
    if (pe != cudaSuccess) cudaGetLastError();
    const bool on_device = pe == cudaSuccess && (attr.type == cudaMemoryTypeDevice || attr.type == cudaMemoryTypeManaged);
    if (on_device) {
      AET_CUDA(h, launch_to_bf16((const float*)x, dx, elems, s));
    } else {
      float* tmp = nullptr;
      AET_CUDA(h, cudaMalloc((void**)&tmp, elems * 4));
      cudaError_t e = cudaMemcpyAsync(tmp, x, elems * 4, cudaMemcpyHostToDevice, s);
      if (e == cudaSuccess) e = launch_to_bf16(tmp, dx, elems, s);
      if (e == cudaSuccess) e = cudaStreamSynchronize(s);
      cudaFree(tmp);
      if (e != cudaSuccess) return cuda_fail(h, e, "bf16 conversion of client data");
    }
  }
  if (!py) AET_CUDA(h, cudaMemcpyAsync(dy, y, (size_t)n * sizeof(int32_t), cudaMemcpyDefault, s));
  if (debug) {
    if (!bf16) AET_CUDA(h, launch_validate_data((const float*)dx, dy, n, (uint32_t)D, h->cfg.dims[h->cfg.n_layers], h->d_status(), s));
    else AET_CUDA(h, launch_validate_data(nullptr, dy, n, (uint32_t)D, h->cfg.dims[h->cfg.n_layers], h->d_status(), s));
  }
  h->h_clients[client] = ClientData{dx, dy, n, 0};
  h->clients_dirty = true;
  h->last_stream = s;
  return AET_OK;
}

aet_status aet_run_rounds(aet_handle* h, uint32_t n_rounds, void* cuda_stream) {
  if (!h) return AET_ERR_ARG;
  cudaStream_t s = (cudaStream_t)cuda_stream;
  for (uint32_t c = 0; c < h->cfg.n_clients; ++c)
    if (!h->h_clients[c].x) return fail(h, AET_ERR_STATE, "client " + std::to_string(c) + " has no data");
  if (n_rounds == 0) return AET_OK;
  join_prepare(h);
  collect_timings(h);
  h->stats = aet_stats{};
  if (h->cfg.topology == 1) return run_ring_rounds(h, n_rounds, s);

  // ---- a0: integer schedule and launch plan (cached for repeated runs) ----
  auto t0 = std::chrono::steady_clock::now();
  CachedPlan& cp = h->cached;
  if (h->prep_ok && h->prep.valid && h->prep.rounds_before == h->st.rounds_done && h->prep.n_rounds == n_rounds &&
      h->prep.before.clock == h->st.clock && h->prep.before.H == h->st.H) {
    cp = std::move(h->prep);   // prepared by aet_prepare_rounds for exactly this state
    h->delays = std::move(h->prep_delays);
  }
  h->prep_ok = false;
  if (!(cp.valid && cp.rounds_before == h->st.rounds_done && cp.n_rounds == n_rounds &&
        cp.before.clock == h->st.clock && cp.before.H == h->st.H)) {
    cp.valid = false;
    cp.uploaded = false;
    cp.before = h->st;
    cp.rounds_before = h->st.rounds_done;
    cp.n_rounds = n_rounds;
    SchedState st = h->st;
    std::string err;
    if (!simulate(h->cfg, n_rounds, st, h->delays, cp.sched, err)) return fail(h, AET_ERR_CONFIG, err);
    cp.after = st;
    build_plan(h->cfg, h->delays, cp.sched, (h->cfg.flags & AET_FLAG_KEEP_UPDATE_SUMS) != 0, cp.plan);
    cp.valid = true;
  }
  const Plan& plan = cp.plan;
  const size_t E = cp.sched.events.size();
  h->stats.plan_ms = std::chrono::duration<double, std::milli>(std::chrono::steady_clock::now() - t0).count();

  // ---- device buffers ----
  aet_status st_up = upload_clients(h, s);
  if (st_up != AET_OK) return st_up;
  // tasks, sums in flight and updates side by side: one copy
  const size_t off_in = E * sizeof(TaskDesc), off_ap = off_in + plan.inflight.size() * sizeof(InflightRef);
  const size_t plan_bytes = off_ap + E * sizeof(ApplyDesc);
  bool ok = h->snaps.reserve((size_t)plan.n_snap * h->stride) && h->U.reserve((size_t)plan.n_u_rows * h->stride) &&
            h->d_plan.reserve(plan_bytes) &&
            h->d_trig.reserve(E) && h->d_alog.reserve(E);
  if (ok && !h->lr_fast) ok = h->act.reserve((size_t)plan.max_wave_tasks * h->act_floats());
  if (!ok) return fail(h, AET_ERR_NOMEM, "device allocation failed");
  if (!cp.uploaded) {
    std::vector<char>& pack = h->pack;
    pack.resize(plan_bytes);
    memcpy(pack.data(), plan.tasks.data(), off_in);
    if (off_ap > off_in) memcpy(pack.data() + off_in, plan.inflight.data(), off_ap - off_in);
    memcpy(pack.data() + off_ap, plan.applies.data(), plan_bytes - off_ap);
    // (a copy from pageable memory has read its source when it returns: no need to wait)
    AET_CUDA(h, cudaMemcpyAsync(h->d_plan.p, pack.data(), plan_bytes, cudaMemcpyHostToDevice, s));
    cp.uploaded = true;
  }
  // snapshot 0 = the server model as this call begins; no round has been triggered yet
  AET_CUDA(h, launch_copy_and_zero(h->snaps.p, h->w_cur(), h->stride, reinterpret_cast<uint32_t*>(h->d_trig.p), E * sizeof(TriggerRec) / 4, s));

  RoundLaunch r{};
  r.tasks = reinterpret_cast<const TaskDesc*>(h->d_plan.p);
  r.inflight = reinterpret_cast<const InflightRef*>(h->d_plan.p + off_in); r.clients = h->d_clients.p;
  r.sample_keys = h->d_keys.p; r.snaps = h->snaps.p; r.U = h->U.p; r.w_end = nullptr;
  r.trig = h->d_trig.p; r.status = h->d_status(); r.stride = h->stride; r.l2 = h->cfg.l2;
  r.debug_checks = (h->cfg.flags & AET_FLAG_DEBUG_CHECKS) ? 1u : 0u;
  r.step_by_step = (h->cfg.flags & AET_FLAG_STEPWISE_RECURRENCE) ? 1u : 0u;
  r.n_u_rows = plan.n_u_rows; r.n_snap = plan.n_snap;
  ApplyLaunch a{};
  a.applies = reinterpret_cast<const ApplyDesc*>(h->d_plan.p + off_ap); a.U = h->U.p; a.snaps = h->snaps.p; a.w = h->w_cur();
  a.H = h->d_H.p; a.log = h->d_alog.p; a.status = h->d_status(); a.stride = h->stride; a.n_params = h->P;

  // ---- waves: a3/a4 local SGD of independent round-tasks, then a6 aggregation ----
  const uint32_t n_waves = (uint32_t)plan.apply_upto.size();
  uint32_t applied = 0;
  for (uint32_t L = 0; L < n_waves; ++L) {
    r.task_begin = plan.wave_off[L];
    r.n_tasks = plan.wave_off[L + 1] - plan.wave_off[L];
    r.longest = longest_round(plan.tasks.data() + r.task_begin, r.n_tasks);
    aet_status rs = launch_rounds(h, r, s);
    if (rs != AET_OK) return rs;
    if (plan.apply_upto[L] > applied) {
      a.lo = applied; a.hi = plan.apply_upto[L];
      KernelTimer kt(h, s, 1);
      cudaError_t e = launch_apply_updates(a, s);
      if (e != cudaSuccess) return cuda_fail(h, e, "aggregation kernel launch");
      applied = a.hi;
    }
  }
  h->stats.waves = n_waves;

  // ---- host bookkeeping ----
  h->last_H_before = h->st.H;
  h->last_first_event = h->log.size();
  h->last_n_events = E;
  h->last_checked = false;
  h->last_stream = s;
  h->log.insert(h->log.end(), cp.sched.events.begin(), cp.sched.events.end());
  const aet_summary& q = cp.sched.summary;
  h->total.messages_up += q.messages_up; h->total.model_pulls += q.model_pulls;
  h->total.samples_total += q.samples_total; h->total.messages_if_per_sample += q.messages_if_per_sample;
  h->total.messages_if_constant_b += q.messages_if_constant_b; h->total.t_end_ticks = q.t_end_ticks;
  h->st = cp.after;
  return AET_OK;
}

aet_status aet_prepare_rounds(aet_handle* h, uint32_t n_rounds) {
  if (!h) return AET_ERR_ARG;
  join_prepare(h);
  h->prep_ok = false;
  if (n_rounds == 0) return AET_OK;
  h->prep_delays = h->delays;   // the thread works on copies: nothing it touches is shared until it is joined
  if (h->cfg.topology == 1) {
    h->prep_ring = CachedRingPlan{};
    h->prep_ring.before = h->rst;
    h->prep_ring.rounds_before = h->rst.rounds_done;
    h->prep_ring.n_rounds = n_rounds;
  } else {
    h->prep = CachedPlan{};
    h->prep.before = h->st;
    h->prep.rounds_before = h->st.rounds_done;
    h->prep.n_rounds = n_rounds;
  }
  try {
    h->prep_thread = std::thread([h, n_rounds]() {
      std::string err;
      const bool keep = (h->cfg.flags & AET_FLAG_KEEP_UPDATE_SUMS) != 0;
      if (h->cfg.topology == 1) {
        CachedRingPlan& cp = h->prep_ring;
        RingState st = cp.before;
        if (!simulate_ring(h->cfg, n_rounds, st, h->prep_delays, cp.sched, err)) return;   // aet_run_rounds will report it
        cp.after = st;
        build_ring_plan(h->cfg, h->prep_delays, cp.sched, keep, cp.plan);
        cp.valid = true;
      } else {
        CachedPlan& cp = h->prep;
        SchedState st = cp.before;
        if (!simulate(h->cfg, n_rounds, st, h->prep_delays, cp.sched, err)) return;
        cp.after = st;
        build_plan(h->cfg, h->prep_delays, cp.sched, keep, cp.plan);
        cp.valid = true;
      }
      h->prep_ok = true;
    });
  } catch (...) {
    return fail(h, AET_ERR_STATE, "could not start the schedule thread");
  }
  return AET_OK;
}

aet_status aet_get_global_model(aet_handle* h, float* out, size_t n_params, void* cuda_stream) {
  if (!h || !out) return h ? fail(h, AET_ERR_ARG, "null argument") : AET_ERR_ARG;
  if (n_params != h->P) return fail(h, AET_ERR_ARG, "n_params does not match the model");
  if (h->cfg.topology == 1) return fail(h, AET_ERR_STATE, "the peer-to-peer topology has no server model: use aet_get_node_model");
  return read_model(h, h->w_cur(), out, (cudaStream_t)cuda_stream);
}

aet_status aet_get_node_model(aet_handle* h, uint32_t node, float* out, size_t n_params, void* cuda_stream) {
  if (!h || !out) return h ? fail(h, AET_ERR_ARG, "null argument") : AET_ERR_ARG;
  if (n_params != h->P) return fail(h, AET_ERR_ARG, "n_params does not match the model");
  if (node >= h->cfg.n_clients) return fail(h, AET_ERR_ARG, "node index out of range");
  // client-server: at quiescence every client slot equals the server model
  return read_model(h, h->cfg.topology == 1 ? h->node_w.p + (size_t)node * h->stride : h->w_cur(), out, (cudaStream_t)cuda_stream);
}

aet_status aet_get_update_sum(aet_handle* h, uint32_t seq, float* out, size_t n_params, void* cuda_stream) {
  if (!h || !out) return h ? fail(h, AET_ERR_ARG, "null argument") : AET_ERR_ARG;
  if (n_params != h->P) return fail(h, AET_ERR_ARG, "n_params does not match the model");
  if (seq >= h->last_n_events) return fail(h, AET_ERR_ARG, "seq is not an event of the most recent run");
  if (!(h->cfg.flags & AET_FLAG_KEEP_UPDATE_SUMS))
    return fail(h, AET_ERR_STATE, "update sums are recycled during a run unless the handle was created with AET_FLAG_KEEP_UPDATE_SUMS");
  cudaStream_t s = (cudaStream_t)cuda_stream;
  AET_CUDA(h, cudaMemcpyAsync(out, h->U.p + (size_t)seq * h->stride, (size_t)h->P * sizeof(float), cudaMemcpyDefault, s));
  AET_CUDA(h, cudaStreamSynchronize(s));
  return AET_OK;
}

aet_status aet_get_event_log(aet_handle* h, aet_event* out, size_t capacity, size_t* n_events, aet_summary* summary) {
  if (!h || !n_events) return h ? fail(h, AET_ERR_ARG, "null argument") : AET_ERR_ARG;
  if (!h->last_checked && h->last_n_events && h->cfg.topology == 1) {
    // the trigger record every round kernel left behind, against the schedule it was launched from
    const size_t T = h->last_n_events;
    std::vector<TriggerRec> trig(T);
    AET_CUDA(h, cudaStreamSynchronize(h->last_stream));
    AET_CUDA(h, cudaMemcpy(trig.data(), h->d_trig.p, T * sizeof(TriggerRec), cudaMemcpyDeviceToHost));
    if (aet_status ds = check_device_status(h)) return ds;
    for (size_t k = 0; k < T; ++k) {
      const RingTask& t = h->last_ring_tasks[k];
      if (trig[k].flags != 1 || trig[k].client != t.client || trig[k].round != t.round || trig[k].samples_done != t.samples)
        return fail(h, AET_ERR_STATE, "device trigger record " + std::to_string(k) + " does not match the schedule");
    }
    h->last_checked = true;
  }
  if (!h->last_checked && h->last_n_events) {
    // Compare what the kernels recorded (trigger per round-task, apply order and
    // history counts) with the schedule they were launched from.
    const size_t E = h->last_n_events;
    std::vector<TriggerRec> trig(E);
    std::vector<ApplyRec> alog(E);
    AET_CUDA(h, cudaStreamSynchronize(h->last_stream));
    AET_CUDA(h, cudaMemcpy(trig.data(), h->d_trig.p, E * sizeof(TriggerRec), cudaMemcpyDeviceToHost));
    AET_CUDA(h, cudaMemcpy(alog.data(), h->d_alog.p, E * sizeof(ApplyRec), cudaMemcpyDeviceToHost));
    if (aet_status ds = check_device_status(h)) return ds;
    std::vector<uint32_t> H = h->last_H_before, Hdev(h->cfg.n_clients);
    AET_CUDA(h, cudaMemcpy(Hdev.data(), h->d_H.p, Hdev.size() * sizeof(uint32_t), cudaMemcpyDeviceToHost));
    for (size_t k = 0; k < E; ++k) {
      const aet_event& e = h->log[h->last_first_event + k];
      if (trig[k].flags != 1 || trig[k].client != e.client || trig[k].round != e.round || trig[k].samples_done != e.samples)
        return fail(h, AET_ERR_STATE, "device trigger record " + std::to_string(k) + " does not match the schedule");
      H[e.client] += 1;
      // h_after of two updates of one client applied by the same launch may swap
      if (alog[k].seq != k || alog[k].client != e.client || alog[k].round != e.round ||
          alog[k].h_after <= h->last_H_before[e.client] || alog[k].h_after > Hdev[e.client])
        return fail(h, AET_ERR_STATE, "device apply record " + std::to_string(k) + " does not match the schedule");
    }
    if (H != Hdev) return fail(h, AET_ERR_STATE, "device history map H does not match the schedule");
    h->last_checked = true;
  }
  if (out) {
    if (capacity < h->log.size()) return fail(h, AET_ERR_ARG, "capacity is smaller than the log");
    memcpy(out, h->log.data(), h->log.size() * sizeof(aet_event));
  }
  *n_events = h->log.size();
  if (summary) *summary = h->total;
  return AET_OK;
}

static aet_status debug_round(aet_handle* h, uint32_t client, uint32_t round, uint32_t lose, uint32_t max_polls, const float* w_in,
                              float* U_out, float* w_out, void* cuda_stream) {
  if (!h || !w_in) return h ? fail(h, AET_ERR_ARG, "null argument") : AET_ERR_ARG;
  if (client >= h->cfg.n_clients) return fail(h, AET_ERR_ARG, "client index out of range");
  if (round < h->cfg.round_base) return fail(h, AET_ERR_ARG, "round is before round_base");
  if (!h->h_clients[client].x) return fail(h, AET_ERR_STATE, "client has no data");
  join_prepare(h);
  ensure_split(h->cfg, round + 1, h->delays);
  const uint32_t s_i = node_sample_size(h->cfg, h->delays, client, round);
  if (s_i % h->cfg.batch || (s_i == 0 && !h->cfg.split_mode))
    return fail(h, AET_ERR_CONFIG, "batch must divide the round's sample count");
  cudaStream_t s = (cudaStream_t)cuda_stream;
  aet_status up = upload_clients(h, s);
  if (up != AET_OK) return up;
  // private area: [snapshot | U | w_end | task | trigger record]
  const size_t fl = 3 * h->stride + 64;
  if (!h->dbg.reserve(fl)) return fail(h, AET_ERR_NOMEM, "device allocation failed");
  if (!h->lr_fast && !h->act.reserve(h->act_floats())) return fail(h, AET_ERR_NOMEM, "device allocation failed");
  float* snap = h->dbg.p;
  float* U = snap + h->stride;
  float* wend = U + h->stride;
  TaskDesc* dtask = (TaskDesc*)(wend + h->stride);
  TriggerRec* dtrig = (TriggerRec*)((char*)dtask + sizeof(TaskDesc));
  TaskDesc t{};
  t.client = client; t.round = round; t.seq = 0; t.snap_slot = 0;
  t.n_samples = s_i; t.steps = s_i / h->cfg.batch;
  t.inflight_off = 0; t.inflight_cnt = 0;
  t.sample_ctr0 = node_samples_before(h->cfg, h->delays, client, round);
  t.eta = (float)round_step_size(h->cfg, h->delays, client, round);
  AET_CUDA(h, cudaMemcpyAsync(snap, w_in, (size_t)h->P * sizeof(float), cudaMemcpyDefault, s));
  AET_CUDA(h, cudaMemcpyAsync(dtask, &t, sizeof(t), cudaMemcpyHostToDevice, s));
  AET_CUDA(h, cudaStreamSynchronize(s));
  RoundLaunch r{};
  r.tasks = dtask; r.inflight = nullptr; r.clients = h->d_clients.p; r.sample_keys = h->d_keys.p;
  r.snaps = snap; r.U = U; r.w_end = wend; r.trig = dtrig; r.status = h->d_status(); r.stride = h->stride;
  r.task_begin = 0; r.n_tasks = 1; r.l2 = h->cfg.l2;
  r.debug_checks = (h->cfg.flags & AET_FLAG_DEBUG_CHECKS) ? 1u : 0u;
  r.step_by_step = (h->cfg.flags & AET_FLAG_STEPWISE_RECURRENCE) ? 1u : 0u;
  r.n_u_rows = 1; r.n_snap = 1;
  r.lose = lose; r.max_polls = max_polls;
  // (regression) the kernel a wave of this round of all clients runs, so that this parity aid checks it
  r.wave_tasks = h->cfg.n_clients; r.longest = s_i;
  const aet_stats keep = h->stats;
  const bool timing = h->timing;
  h->timing = false;
  aet_status rs = launch_rounds(h, r, s);
  h->timing = timing;
  h->stats = keep;
  if (rs != AET_OK) return rs;
  AET_CUDA(h, cudaStreamSynchronize(s));
  const aet_status ds = check_device_status(h);
  if (ds && !lose) return ds;
  if (U_out) AET_CUDA(h, cudaMemcpyAsync(U_out, U, (size_t)h->P * sizeof(float), cudaMemcpyDefault, s));
  if (w_out) AET_CUDA(h, cudaMemcpyAsync(w_out, wend, (size_t)h->P * sizeof(float), cudaMemcpyDefault, s));
  AET_CUDA(h, cudaStreamSynchronize(s));
  return ds;
}

aet_status aet_debug_run_client_round(aet_handle* h, uint32_t client, uint32_t round, const float* w_in,
                                      float* U_out, float* w_out, void* cuda_stream) {
  return debug_round(h, client, round, 0, 0, w_in, U_out, w_out, cuda_stream);
}

aet_status aet_debug_lost_copies(aet_handle* h, uint32_t client, uint32_t round, uint32_t cta, uint32_t max_polls, const float* w_in,
                                 float* U_out, float* w_out, void* cuda_stream) {
  if (!h) return AET_ERR_ARG;
  if (!h->lr_fast || h->cfg.split_mode || round < h->cfg.round_base) return fail(h, AET_ERR_CONFIG, "lost copies can be played for the regression's rounds only");
  uint32_t at_once[9];
  AET_CUDA(h, clusters_at_once(at_once));
  const LrChoice c = choose_lr_kernel(h->cfg.n_clients, sample_size(h->cfg, round), false, at_once);
  if (c.kernel != LrKernel::kRelay) return fail(h, AET_ERR_CONFIG, "lost copies can be played for few clients only");
  if (cta >= c.cluster || max_polls == 0 || max_polls > (1u << 16)) return fail(h, AET_ERR_ARG, "cta must be below the cluster's width, max_polls in [1, 2^16]");
  return debug_round(h, client, round, cta + 1, max_polls, w_in, U_out, w_out, cuda_stream);
}

aet_status aet_debug_wait_probe(aet_handle* h, uint32_t max_polls, void* cuda_stream) {
  if (!h) return AET_ERR_ARG;
  if (max_polls == 0 || max_polls > (1u << 24)) return fail(h, AET_ERR_ARG, "max_polls must be in [1, 2^24]");
  cudaStream_t s = (cudaStream_t)cuda_stream;
  cudaError_t e = launch_wait_probe(h->d_status(), max_polls, s);
  if (e != cudaSuccess) return cuda_fail(h, e, "wait probe launch");
  AET_CUDA(h, cudaStreamSynchronize(s));
  return check_device_status(h);
}

aet_status aet_set_kernel_timing(aet_handle* h, int enable) {
  if (!h) return AET_ERR_ARG;
  h->timing = enable != 0;
  return AET_OK;
}

aet_status aet_get_stats(aet_handle* h, aet_stats* out) {
  if (!h || !out) return AET_ERR_ARG;
  collect_timings(h);
  *out = h->stats;
  return AET_OK;
}

size_t aet_n_params(const aet_handle* h) { return h ? h->P : 0; }

const char* aet_last_error(const aet_handle* h) { return h ? h->err.c_str() : g_create_error.c_str(); }

aet_status aet_schedule_only(const aet_config* cfg, uint32_t n_rounds, aet_event* out, size_t capacity,
                             size_t* n_events, aet_summary* summary) {
  if (!cfg || !n_events) return fail(nullptr, AET_ERR_ARG, "null argument");
  std::string err;
  if (cfg->struct_size != sizeof(aet_config)) return fail(nullptr, AET_ERR_ARG, "struct_size does not match sizeof(aet_config)");
  if (!validate_config(*cfg, err)) return fail(nullptr, AET_ERR_CONFIG, err);
  DelayCache cache;
  std::vector<aet_event> events;
  aet_summary sum{};
  if (cfg->topology == 1) {
    RingState rst;
    RingResult rres;
    if (!simulate_ring(*cfg, n_rounds, rst, cache, rres, err)) return fail(nullptr, AET_ERR_CONFIG, err);
    events.swap(rres.events);
    sum = rres.summary;
  } else {
    SchedState st;
    SchedResult res;
    if (!simulate(*cfg, n_rounds, st, cache, res, err)) return fail(nullptr, AET_ERR_CONFIG, err);
    events.swap(res.events);
    sum = res.summary;
  }
  if (out) {
    if (capacity < events.size()) return fail(nullptr, AET_ERR_ARG, "capacity is smaller than the log");
    memcpy(out, events.data(), events.size() * sizeof(aet_event));
  }
  *n_events = events.size();
  if (summary) *summary = sum;
  return AET_OK;
}

uint32_t aet_debug_regression_kernel(uint32_t n_tasks, uint32_t longest, uint32_t by_value, const uint32_t* at_once) {
  uint32_t n[9];
  for (int i = 0; i < 9; ++i) n[i] = at_once[i];
  const LrChoice c = choose_lr_kernel(n_tasks, longest, by_value != 0, n);
  return (uint32_t)c.kernel * 16 + c.cluster;
}

uint64_t aet_debug_draw(uint64_t seed, uint32_t stream, uint32_t client, uint64_t counter) {
  return draw(stream_key(seed, stream, client), counter);
}

uint64_t aet_debug_delay_ticks(uint32_t dist, uint64_t r, uint64_t p0, uint64_t p1) {
  return dist == 0 ? exp_ticks(r, p0) : uniform_ticks(r, p0, p1);
}

uint32_t aet_debug_plan_waves(const aet_config* cfg, uint32_t n_rounds) {
  if (!cfg || cfg->struct_size != sizeof(aet_config)) return 0;
  std::string err;
  if (!validate_config(*cfg, err)) return 0;
  SchedState st;
  DelayCache cache;
  SchedResult res;
  if (!simulate(*cfg, n_rounds, st, cache, res, err)) return 0;
  Plan plan;
  build_plan(*cfg, cache, res, (cfg->flags & AET_FLAG_KEEP_UPDATE_SUMS) != 0, plan);
  return (uint32_t)plan.apply_upto.size();
}

aet_status aet_debug_plan_layout(const aet_config* cfg, uint32_t n_rounds, uint32_t* task_seq, uint32_t* task_wave,
                                 uint32_t* task_snap_slot, uint32_t* u_row, int32_t* snap_slot_after,
                                 uint32_t* apply_upto, uint32_t* counts) {
  if (!cfg || !task_seq || !task_wave || !task_snap_slot || !u_row || !snap_slot_after || !apply_upto || !counts)
    return fail(nullptr, AET_ERR_ARG, "null argument");
  if (cfg->struct_size != sizeof(aet_config)) return fail(nullptr, AET_ERR_ARG, "struct_size does not match sizeof(aet_config)");
  std::string err;
  if (!validate_config(*cfg, err)) return fail(nullptr, AET_ERR_CONFIG, err);
  SchedState st;
  DelayCache cache;
  SchedResult res;
  if (!simulate(*cfg, n_rounds, st, cache, res, err)) return fail(nullptr, AET_ERR_CONFIG, err);
  Plan plan;
  build_plan(*cfg, cache, res, (cfg->flags & AET_FLAG_KEEP_UPDATE_SUMS) != 0, plan);
  const uint32_t n_waves = (uint32_t)plan.apply_upto.size();
  for (uint32_t L = 0; L < n_waves; ++L) {
    apply_upto[L] = plan.apply_upto[L];
    for (uint32_t q = plan.wave_off[L]; q < plan.wave_off[L + 1]; ++q) {
      task_seq[q] = plan.tasks[q].seq;
      task_wave[q] = L;
      task_snap_slot[q] = plan.tasks[q].snap_slot;
    }
  }
  for (size_t k = 0; k < res.events.size(); ++k) {
    u_row[k] = plan.applies[k].u_row;
    snap_slot_after[k] = plan.applies[k].snap_slot;
  }
  counts[0] = n_waves; counts[1] = plan.n_u_rows; counts[2] = plan.n_snap;
  return AET_OK;
}

}  // extern "C"
