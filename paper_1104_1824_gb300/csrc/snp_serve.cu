// Serving loop (snp_server_*): explorations submitted at any time are admitted
// while device memory allows and advanced together by the sparse batch form
// (snp_many.cu), a few iterations per tick.  A request that arrives while
// others run joins at the next tick (continuous batching); a finished request
// is copied into its handle, its memory is returned, and its latency (submit
// to result ready) is recorded.
#include <algorithm>
#include <atomic>
#include <chrono>
#include <condition_variable>
#include <cstring>
#include <deque>
#include <map>
#include <mutex>
#include <thread>
#include <vector>

#include "snp_host.h"

using namespace snp;

namespace {

using Clock = std::chrono::steady_clock;

__global__ void k_fill_ranges(unsigned long long* const* ptr, const uint64_t* count, int32_t n, unsigned long long v) {
  for (int32_t r = blockIdx.y; r < n; r += gridDim.y) {
    unsigned long long* p = ptr[r];
    const uint64_t c = count[r];
    for (uint64_t i = (uint64_t)blockIdx.x * blockDim.x + threadIdx.x; i < c; i += (uint64_t)gridDim.x * blockDim.x)
      p[i] = v;
  }
}

// First-fit allocator over [0, size), 256-byte granules.
class RangeAlloc {
 public:
  explicit RangeAlloc(size_t size) { free_[0] = size; }
  bool alloc(size_t bytes, size_t* off) {
    bytes = (bytes + 255) & ~size_t(255);
    for (auto it = free_.begin(); it != free_.end(); ++it) {
      if (it->second >= bytes) {
        *off = it->first;
        const size_t rest = it->second - bytes, at = it->first + bytes;
        free_.erase(it);
        if (rest) free_[at] = rest;
        return true;
      }
    }
    return false;
  }
  void release(size_t off, size_t bytes) {
    bytes = (bytes + 255) & ~size_t(255);
    auto it = free_.emplace(off, bytes).first;
    auto next = std::next(it);
    if (next != free_.end() && it->first + it->second == next->first) {
      it->second += next->second;
      free_.erase(next);
    }
    if (it != free_.begin()) {
      auto prev = std::prev(it);
      if (prev->first + prev->second == it->first) {
        prev->second += it->second;
        free_.erase(it);
      }
    }
  }

 private:
  std::map<size_t, size_t> free_;
};

struct Request {
  uint64_t id = 0;
  snp_system* h = nullptr;
  snp_explore_opts o{};
  Clock::time_point arrival, done;
  size_t bytes = 0;           // pool, table, stats
  size_t off = 0, held = 0;   // range of the server's memory: these, then (unless own) the scratch
  uint32_t qc = 0;            // candidates of a pass
  bool own = false;           // its scratch is its own allocation
  int64_t rows = 0;
  uint64_t nslots = 0;
  int32_t slot = -1;         // place in the device array of systems
  DevBuf scratch;            // own
  int64_t items = 0;         // work items it can have queued
  BatchSys bs{};
  int status = SNP_OK;
};

}  // namespace

struct snp_server {
  int device = 0;
  size_t budget = 0;
  int32_t max_active = 0;
  DevBuf arena, sys_dev, items, ctr, idx_dev, c0_dev, c0_off_dev, fill_ptr, fill_cnt;
  std::vector<Request*> slots;   // requests by their place in sys_dev (null: free)
  std::vector<BatchSys> back;    // sys_dev as read back after a tick
  int64_t item_cap = 0;          // items each queue holds
  int par = 0;                   // parity of the next iteration
  RangeAlloc* alloc = nullptr;
  cudaStream_t st = nullptr;
  std::mutex mu;
  std::condition_variable cv, cv_done;
  std::deque<Request*> pending;
  std::vector<Request*> active;
  std::deque<Request*> finished;
  std::thread loop;
  bool stop = false;
  uint64_t next_id = 1;
  uint64_t submitted = 0, completed = 0;
  int64_t total_new = 0;
  int64_t ticks = 0;
  double busy_ms = 0.0;
  std::vector<double> lat_ms;
  Clock::time_point first_arrival, last_done;
  bool any = false;
  int loop_error = SNP_OK;
  std::string loop_msg;
};

namespace {

constexpr uint32_t kServeQc = 2048;    // claims past the cap a request's table has room for, per depth
// Candidates per work item.  48 requests of 8 to 512 neurons, cap 2^12: 65.8 ms
// with 64, 65.9 with 32, 72.4 with 128, 80.6 with 192; 16 of 8 to 128 neurons,
// cap 2^10: 6.1, 5.6, 7.1, 8.1 ms.
constexpr uint32_t kServeRun = 64;
constexpr int kTickIterations = 8;

size_t request_bytes(const snp_system* h, const snp_explore_opts& o, int64_t* rows, uint64_t* nslots) {
  *rows = 1 + (int64_t)o.depth * o.frontier_cap;
  const uint64_t want = (uint64_t)((long double)(*rows + (int64_t)o.depth * kServeQc) * 4.0L / 3.0L) + kBucket;
  *nslots = std::max<uint64_t>(pow2_at_least(want), kBucket);
  auto r = [](size_t b) { return (b + 255) & ~size_t(255); };
  return r((size_t)*rows * h->m * 4) + r(*nslots * 8) + r(sizeof(BatchDepthStat) * (o.depth + 1));
}

size_t scratch_bytes(const Request* r, uint32_t qc) { return many_scratch_bytes(r->o.frontier_cap, qc, r->h->m); }

// A place in the server's memory for a request's pool, table and statistics,
// and behind them the scratch of its passes: of the size the cap asks for, or,
// where that does not fit beside the requests that run, of 2048 candidates.  A
// request that leaves no room for scratch in the whole of the memory waits
// until no other runs and has the scratch of such passes allocated (r->own).
// false: it has to wait.  (Scratch allocated apart for every request came to
// up to 0.3 GB each beyond what the caller gave the server.)
bool place(snp_server* S, Request* r) {
  const uint32_t full = many_default_qc(r->o.frontier_cap);
  for (const uint32_t qc : {full, std::min(full, kServeQc)}) {
    r->qc = qc;
    r->held = r->bytes + scratch_bytes(r, qc);
    if (S->alloc->alloc(r->held, &r->off)) return true;
  }
  if (!S->active.empty()) return false;
  r->held = r->bytes;
  r->own = true;
  return S->alloc->alloc(r->held, &r->off);
}

ManyQueue queue_of(const snp_server* S) {
  ManyQueue q;
  q.expand[0] = S->items.as<int2>();
  q.expand[1] = q.expand[0] + kMqForms * S->item_cap;
  q.copy = q.expand[1] + kMqForms * S->item_cap;
  q.psi[0] = q.copy + S->item_cap;
  q.psi[1] = q.psi[0] + S->item_cap;
  q.ctr = S->ctr.as<uint32_t>();
  q.cap = S->item_cap;
  return q;
}

// Room in the queues for `items` work items (what is queued is kept).
int ensure_items(snp_server* S, int64_t items) {
  if (!S->ctr.p) {
    TRY(S->ctr.reserve(sizeof(uint32_t) * kMqCounters));
    CK(cudaMemsetAsync(S->ctr.p, 0, sizeof(uint32_t) * kMqCounters, S->st));
  }
  if (items <= S->item_cap) return SNP_OK;
  const int64_t old = S->item_cap, want = std::max<int64_t>(items, 2 * old);
  DevBuf grown;
  TRY(grown.reserve(sizeof(int2) * (2 * kMqForms + 3) * want));
  for (int k = 0; old > 0 && k < 2 * kMqForms + 3; ++k)
    CK(cudaMemcpyAsync(grown.as<int2>() + k * want, S->items.as<int2>() + k * old, sizeof(int2) * old,
                       cudaMemcpyDeviceToDevice, S->st));
  CK(cudaStreamSynchronize(S->st));
  std::swap(S->items.p, grown.p);
  std::swap(S->items.bytes, grown.bytes);
  S->item_cap = want;
  return SNP_OK;
}

// The system of an admitted request as the kernels see it, and its place among them.
void set_up(snp_server* S, Request* r) {
  auto r256 = [](size_t b) { return (b + 255) & ~size_t(255); };
  unsigned char* base = S->arena.as<unsigned char>() + r->off;
  BatchSys& b = r->bs;
  std::memset(&b, 0, sizeof b);
  b.sys = r->h->dev();
  b.pool = reinterpret_cast<int32_t*>(base);
  b.slots = reinterpret_cast<unsigned long long*>(base + r256((size_t)r->rows * r->h->m * 4));
  b.bmask = r->nslots / kBucket - 1;
  b.stats = reinterpret_cast<BatchDepthStat*>(base + r256((size_t)r->rows * r->h->m * 4) + r256(r->nslots * 8));
  b.pool_rows = r->rows;
  b.level_lo = 0;
  b.level_hi = 1;
  b.n_rows = 1;
  b.target_depth = r->o.depth;
  b.max_expand = r->o.max_expand_value;
  b.cap = r->o.frontier_cap;
  b.budget = r->o.candidate_budget > 0 ? r->o.candidate_budget : 0;
  b.overshoot = kServeQc;
  many_carve(b, r->own ? r->scratch.as<unsigned char>() : base + r->bytes, r->qc, kServeRun);
  const ManyPlan mine = many_plan(&r->h->m, 1, 0, 0);
  b.tile = many_tile(mine, r->h->m, 0);
  r->items = many_items(b.cap, r->qc, kServeRun);
  r->slot = 0;
  while (r->slot < (int32_t)S->slots.size() && S->slots[r->slot]) ++r->slot;
  if (r->slot == (int32_t)S->slots.size()) S->slots.push_back(nullptr);
  S->slots[r->slot] = r;
}

// Memory that newly admitted requests need beside their own: before anything of them is on the device.
int room_for(snp_server* S, const std::vector<Request*>& fresh) {
  if (fresh.empty()) return SNP_OK;
  const size_t n = fresh.size();
  size_t counts = 0;
  int64_t items = 0;
  for (const Request* r : S->active) items += r->items;  // the new ones among them
  for (const Request* r : fresh) counts += (size_t)r->h->m;
  TRY(ensure_items(S, items));
  TRY(S->sys_dev.reserve(sizeof(BatchSys) * std::max<size_t>(64, S->slots.size() * 2), S->st, true));
  TRY(S->fill_ptr.reserve(sizeof(void*) * n));
  TRY(S->fill_cnt.reserve(sizeof(uint64_t) * n));
  TRY(S->idx_dev.reserve(sizeof(int32_t) * n));
  TRY(S->c0_dev.reserve(sizeof(int32_t) * counts));
  TRY(S->c0_off_dev.reserve(sizeof(int64_t) * n));
  return SNP_OK;
}

// Device state of newly admitted requests: empty tables, C0 in row 0 and in the table.
int init_requests(snp_server* S, const std::vector<Request*>& fresh) {
  if (fresh.empty()) return SNP_OK;
  const int n = (int)fresh.size();
  std::vector<unsigned long long*> ptr(n);
  std::vector<uint64_t> cnt(n);
  std::vector<int32_t> c0, idx(n);
  std::vector<int64_t> c0_off(n);
  for (int i = 0; i < n; ++i) {
    Request* r = fresh[i];
    ptr[i] = r->bs.slots;
    cnt[i] = r->nslots;
    idx[i] = r->slot;
    c0_off[i] = (int64_t)c0.size();
    c0.insert(c0.end(), r->h->c0.begin(), r->h->c0.end());
  }
  CK(cudaMemcpyAsync(S->fill_ptr.p, ptr.data(), sizeof(void*) * n, cudaMemcpyHostToDevice, S->st));
  CK(cudaMemcpyAsync(S->fill_cnt.p, cnt.data(), sizeof(uint64_t) * n, cudaMemcpyHostToDevice, S->st));
  CK(cudaMemcpyAsync(S->idx_dev.p, idx.data(), sizeof(int32_t) * n, cudaMemcpyHostToDevice, S->st));
  CK(cudaMemcpyAsync(S->c0_dev.p, c0.data(), sizeof(int32_t) * c0.size(), cudaMemcpyHostToDevice, S->st));
  CK(cudaMemcpyAsync(S->c0_off_dev.p, c0_off.data(), sizeof(int64_t) * n, cudaMemcpyHostToDevice, S->st));
  dim3 grid(64, (unsigned)std::min(n, 1024));
  k_fill_ranges<<<grid, 256, 0, S->st>>>(S->fill_ptr.as<unsigned long long*>(), S->fill_cnt.as<uint64_t>(), n, kEmpty);
  CK(cudaGetLastError());
  for (int i = 0; i < n; ++i) {
    Request* r = fresh[i];
    CK(cudaMemsetAsync(r->bs.stats, 0, sizeof(BatchDepthStat) * (r->o.depth + 1), S->st));
    CK(cudaMemcpyAsync(S->sys_dev.as<BatchSys>() + r->slot, &r->bs, sizeof(BatchSys), cudaMemcpyHostToDevice, S->st));
  }
  launch_many_init(S->sys_dev.as<BatchSys>(), S->idx_dev.as<int32_t>(), S->c0_dev.as<int32_t>(),
                   S->c0_off_dev.as<int64_t>(), n, queue_of(S), S->st);
  CK(cudaGetLastError());
  return SNP_OK;
}

// Copies a finished request's configurations and statistics into its handle.
int retire(snp_server* S, Request* r) {
  snp_system* h = r->h;
  const BatchSys& b = r->bs;
  const int depth = r->o.depth;
  std::vector<BatchDepthStat> st(depth + 1);
  CK(cudaMemcpyAsync(st.data(), b.stats, sizeof(BatchDepthStat) * (depth + 1), cudaMemcpyDeviceToHost, S->st));
  const size_t bytes = sizeof(int32_t) * (size_t)b.n_rows * h->m;
  r->scratch.release();  // its passes are done
  if (h->d_pool.reserve(bytes) != SNP_OK) {  // this request fails; the server goes on
    r->status = SNP_E_NOMEM;
    h->explored = false;
    return SNP_OK;
  }
  h->pool_rows = std::max<int64_t>(h->pool_rows, b.n_rows);
  CK(cudaMemcpyAsync(h->d_pool.p, b.pool, bytes, cudaMemcpyDeviceToDevice, S->st));
  CK(cudaStreamSynchronize(S->st));
  h->stats.clear();
  snp_depth_info s0;
  std::memset(&s0, 0, sizeof s0);
  s0.new_configs = 1;
  h->stats.push_back(s0);
  int64_t lo = 0, hi = 1;
  for (int d = 1; d <= std::min(depth, b.cur_depth); ++d) {
    const BatchDepthStat& x = st[d];
    snp_depth_info sd;
    std::memset(&sd, 0, sizeof sd);
    sd.new_configs = x.new_configs;
    sd.parents = hi - lo;
    sd.candidates = x.candidates;
    sd.examined = x.examined;
    sd.truncated = x.truncated;
    sd.chunks = x.chunks;
    h->stats.push_back(sd);
    lo = hi;
    hi += x.new_configs;
  }
  h->n_rows = b.n_rows;
  h->depth_reached = b.depth_reached;
  h->explored = true;
  h->have_parents = false;
  h->batch.reset();
  h->result_pool = h->d_pool.as<int32_t>();
  h->result_perm = nullptr;
  h->result_w = 4;
  h->row_w = 4;
  r->status = (b.error & kErrOverflow) ? SNP_E_OVERFLOW
              : (b.error & kErrTimeout) ? SNP_E_TIMEOUT
              : b.error ? SNP_E_INTERNAL : SNP_OK;
  return SNP_OK;
}

// A few iterations over every active request, then their state read back.
int tick(snp_server* S) {
  if (S->active.empty()) return SNP_OK;
  std::vector<int> ms;
  for (const Request* r : S->active) ms.push_back(r->h->m);
  const ManyPlan mp = many_plan(ms.data(), (int64_t)ms.size(), 0, 0);
  // (a request's tile was chosen for its own rows alone: shared memory for all of them holds it)
  const int n = (int)S->slots.size();
  BatchSys* dsys = S->sys_dev.as<BatchSys>();
  for (int k = 0; k < kTickIterations; ++k) {
    launch_many_iteration(dsys, n, queue_of(S), S->par, mp, S->st, sm_count(S->device));
    S->par ^= 1;
  }
  CK(cudaGetLastError());
  S->back.resize(n);
  CK(cudaMemcpyAsync(S->back.data(), dsys, sizeof(BatchSys) * n, cudaMemcpyDeviceToHost, S->st));
  CK(cudaStreamSynchronize(S->st));
  for (Request* r : S->active) r->bs = S->back[r->slot];
  return SNP_OK;
}

// Requests that have run or failed, from the active ones to the finished ones
// in one step, as snp_server_wait and _stats look at them (S->mu held).
void finish_locked(snp_server* S, const std::vector<Request*>& done) {
  for (Request* r : done) {
    S->active.erase(std::find(S->active.begin(), S->active.end(), r));
    S->alloc->release(r->off, r->held);
    S->completed += 1;
    S->total_new += std::max<int64_t>(r->bs.n_rows - 1, 0);
    S->lat_ms.push_back(std::chrono::duration<double, std::milli>(r->done - r->arrival).count());
    S->last_done = r->done;
    S->finished.push_back(r);
  }
  if (!done.empty()) S->cv_done.notify_all();
}

void finish(snp_server* S, const std::vector<Request*>& done) {
  for (Request* r : done) r->done = Clock::now();
  std::lock_guard<std::mutex> lk(S->mu);
  finish_locked(S, done);
}

void server_loop(snp_server* S) {
  cudaSetDevice(S->device);
  for (;;) {
    std::vector<Request*> fresh;
    {
      std::unique_lock<std::mutex> lk(S->mu);
      if (S->pending.empty() && S->active.empty()) {
        if (S->stop) return;
        S->cv.wait_for(lk, std::chrono::milliseconds(2));
        continue;
      }
      while (!S->pending.empty() && (int32_t)S->active.size() < S->max_active) {
        Request* r = S->pending.front();
        if (!place(S, r)) break;  // admitted when memory frees up
        S->pending.pop_front();
        S->active.push_back(r);
        fresh.push_back(r);
      }
    }
    for (size_t i = 0; i < fresh.size();) {
      Request* r = fresh[i];
      if (r->own && (r->status = r->scratch.reserve(scratch_bytes(r, r->qc))) != SNP_OK) {  // this request fails
        finish(S, {r});
        fresh.erase(fresh.begin() + i);
        continue;
      }
      set_up(S, r);
      ++i;
    }
    const auto t0 = Clock::now();
    int rc = room_for(S, fresh);
    if (rc == SNP_E_NOMEM) {  // the new requests fail; those that run go on
      for (Request* r : fresh) {
        r->status = rc;
        r->scratch.release();
        S->slots[r->slot] = nullptr;
      }
      finish(S, fresh);
      fresh.clear();
      rc = SNP_OK;
    }
    if (rc == SNP_OK) rc = init_requests(S, fresh);
    const int ticked = rc == SNP_OK && !S->active.empty() ? 1 : 0;
    if (rc == SNP_OK) rc = tick(S);
    std::vector<Request*> done;
    for (Request* r : S->active) {
      if (rc != SNP_OK) break;
      if (!(r->bs.done || r->bs.cur_depth >= r->bs.target_depth || r->bs.error)) continue;
      rc = retire(S, r);
      if (rc != SNP_OK) break;
      r->done = Clock::now();
      S->slots[r->slot] = nullptr;
      done.push_back(r);
    }
    const double busy = std::chrono::duration<double, std::milli>(Clock::now() - t0).count();
    std::lock_guard<std::mutex> lk(S->mu);
    S->busy_ms += busy;
    S->ticks += ticked;
    if (rc != SNP_OK && S->loop_error == SNP_OK) {
      S->loop_error = rc;
      S->loop_msg = g_err;
    }
    finish_locked(S, done);
    if (rc != SNP_OK) {  // a device error ends the loop; waiting callers are released
      for (Request* r : S->active) {
        r->status = rc;
        S->finished.push_back(r);
      }
      S->active.clear();
      for (Request* r : S->pending) {
        r->status = rc;
        S->finished.push_back(r);
      }
      S->pending.clear();
      S->cv_done.notify_all();
      return;
    }
  }
}

double percentile(std::vector<double> v, double q) {
  if (v.empty()) return 0.0;
  std::sort(v.begin(), v.end());
  const double pos = q * (v.size() - 1);
  const size_t i = (size_t)pos;
  const double f = pos - i;
  return i + 1 < v.size() ? v[i] * (1 - f) + v[i + 1] * f : v[i];
}

}  // namespace

extern "C" {

int snp_server_create(size_t hbm_budget, int32_t max_active, void** out) {
  g_err.clear();
  if (!out || hbm_budget < (1u << 20) || max_active < 1) return fail(SNP_E_INVALID, "bad arguments");
  *out = nullptr;
  auto* S = new (std::nothrow) snp_server;
  if (!S) return fail(SNP_E_NOMEM, "host allocation failed");
  CK(cudaGetDevice(&S->device));
  S->budget = hbm_budget;
  S->max_active = max_active;
  int rc = S->arena.reserve(hbm_budget);
  if (rc != SNP_OK) {
    delete S;
    return rc;
  }
  S->alloc = new RangeAlloc(hbm_budget);
  CK(cudaStreamCreateWithFlags(&S->st, cudaStreamNonBlocking));
  S->loop = std::thread(server_loop, S);
  *out = S;
  return SNP_OK;
}

int snp_server_submit(void* srv, snp_handle h, const snp_explore_opts* o, uint64_t* req_id) {
  g_err.clear();
  auto* S = static_cast<snp_server*>(srv);
  if (!S || !h || !o || !req_id) return fail(SNP_E_INVALID, "bad arguments");
  if (h->device != S->device) return fail(SNP_E_INVALID, "handle on device %d, server on %d", h->device, S->device);
  if (o->depth < 1) return fail(SNP_E_INVALID, "depth = %d < 1", o->depth);
  if (o->transition != SNP_T_SPARSE_I32 || o->record_parents)
    return fail(SNP_E_INVALID, "the server runs the sparse transition without parent records");
  if (o->frontier_cap < 1 || o->frontier_cap > (1 << 20))
    return fail(SNP_E_INVALID, "the server needs 1 <= frontier_cap <= 2^20");
  auto* r = new (std::nothrow) Request;
  if (!r) return fail(SNP_E_NOMEM, "host allocation failed");
  r->h = h;
  r->o = *o;
  r->bytes = request_bytes(h, *o, &r->rows, &r->nslots);
  if (r->bytes > S->budget) {
    delete r;
    return fail(SNP_E_NOMEM, "request needs %zu bytes, the server holds %zu", r->bytes, S->budget);
  }
  h->explored = false;
  h->batch.reset();
  h->result_pool = nullptr;
  h->result_perm = nullptr;
  {
    std::lock_guard<std::mutex> lk(S->mu);
    if (S->loop_error != SNP_OK) {
      delete r;
      return fail(S->loop_error, "server stopped: %s", S->loop_msg.c_str());
    }
    r->id = S->next_id++;
    r->arrival = Clock::now();
    if (!S->any) {
      S->first_arrival = r->arrival;
      S->any = true;
    }
    S->pending.push_back(r);
    S->submitted += 1;
    *req_id = r->id;
  }
  S->cv.notify_one();
  return SNP_OK;
}

int snp_server_poll(void* srv, uint64_t* ids, double* latency_ms, int32_t* statuses, int32_t max, int32_t* n) {
  g_err.clear();
  auto* S = static_cast<snp_server*>(srv);
  if (!S || !n || max < 0) return fail(SNP_E_INVALID, "bad arguments");
  std::lock_guard<std::mutex> lk(S->mu);
  int32_t k = 0;
  while (k < max && !S->finished.empty()) {
    Request* r = S->finished.front();
    S->finished.pop_front();
    if (ids) ids[k] = r->id;
    if (latency_ms) latency_ms[k] = std::chrono::duration<double, std::milli>(r->done - r->arrival).count();
    if (statuses) statuses[k] = r->status;
    delete r;
    ++k;
  }
  *n = k;
  return SNP_OK;
}

int snp_server_wait(void* srv) {
  g_err.clear();
  auto* S = static_cast<snp_server*>(srv);
  if (!S) return fail(SNP_E_INVALID, "bad arguments");
  std::unique_lock<std::mutex> lk(S->mu);
  S->cv_done.wait(lk, [&] { return (S->pending.empty() && S->active.empty()) || S->loop_error != SNP_OK; });
  if (S->loop_error != SNP_OK) return fail(S->loop_error, "server stopped: %s", S->loop_msg.c_str());
  return SNP_OK;
}

int snp_server_stats(void* srv, snp_server_info* out) {
  g_err.clear();
  auto* S = static_cast<snp_server*>(srv);
  if (!S || !out) return fail(SNP_E_INVALID, "bad arguments");
  std::lock_guard<std::mutex> lk(S->mu);
  std::memset(out, 0, sizeof *out);
  out->submitted = (int64_t)S->submitted;
  out->completed = (int64_t)S->completed;
  out->active = (int64_t)S->active.size();
  out->pending = (int64_t)S->pending.size();
  out->new_configs = S->total_new;
  out->ticks = S->ticks;
  out->busy_ms = S->busy_ms;
  out->span_ms = S->any && S->completed ? std::chrono::duration<double, std::milli>(S->last_done - S->first_arrival).count()
                                        : 0.0;
  out->p50_ms = percentile(S->lat_ms, 0.50);
  out->p99_ms = percentile(S->lat_ms, 0.99);
  out->max_ms = percentile(S->lat_ms, 1.0);
  return SNP_OK;
}

int snp_server_destroy(void* srv) {
  auto* S = static_cast<snp_server*>(srv);
  if (!S) return SNP_OK;
  {
    std::lock_guard<std::mutex> lk(S->mu);
    S->stop = true;
  }
  S->cv.notify_all();
  if (S->loop.joinable()) S->loop.join();
  for (Request* r : S->finished) delete r;
  for (Request* r : S->pending) delete r;
  for (Request* r : S->active) delete r;
  if (S->st) cudaStreamDestroy(S->st);
  delete S->alloc;
  delete S;
  return SNP_OK;
}

}  // extern "C"
