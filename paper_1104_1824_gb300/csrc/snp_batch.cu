// Batch engine, host side (snp_explore_batch, snp_batch_autotune): packs many
// loaded systems into one device arena and advances them together.  Sparse
// form: iterations of snp_many.cu until no system is left, the next one
// enqueued before the last one's count is read back.  Tensor-core form: one
// depth per launch of k_batch_depth_tc, captured in one CUDA graph.
#include <algorithm>
#include <chrono>
#include <cstring>
#include <vector>

#include "snp_host.h"

using namespace snp;

namespace snp {

// Device memory of one batch; shared by its handles until they move on.
struct BatchArena {
  DevBuf sys, stats, pools, slots, scratch, queue, items, c0, c0_off;
  int32_t n = 0, depth = 0;
  // shape the buffers and the captured graph were made for
  std::vector<snp_system*> handles;
  int64_t cap = 0, budget = 0;
  int32_t max_expand = 0, blocks = 0, tc = 0;
  uint32_t qc = 0;
  uint64_t nslots = 0;
  size_t scratch_stride = 0, pool_bytes = 0;
  cudaGraphExec_t exec = nullptr;
  ~BatchArena() {
    if (exec) cudaGraphExecDestroy(exec);
  }
};

}  // namespace snp

namespace {

struct BatchPlan {
  uint32_t qc = 0;         // candidates per pass (0: chosen by the cap)
  int tile = 0, warps = 0;  // rows of an expand tile, warps per CTA (0: automatic)
};

// Scratch the systems of one group share the device with.
constexpr size_t kGroupScratch = (size_t)12 << 30;
// Scratch that stays with the results for the next batch of the same handles;
// more is given back when the call returns.  (Giving back all of it: 512
// systems with 2.9 GB of scratch, 48.4 -> 51.1 ms.)
constexpr size_t kKeptScratch = (size_t)4 << 30;

// Device time of the parts of a batch that count: what lies between start()
// and stop(), allocations and graph capture left out.
struct BatchTimer {
  cudaEvent_t e0 = nullptr, e1 = nullptr;
  float ms = 0.f;
  ~BatchTimer() {
    if (e0) cudaEventDestroy(e0);
    if (e1) cudaEventDestroy(e1);
  }
  int start(cudaStream_t st) {
    if (!e0) CK(cudaEventCreate(&e0));
    if (!e1) CK(cudaEventCreate(&e1));
    CK(cudaEventRecord(e0, st));
    return SNP_OK;
  }
  int stop(cudaStream_t st) {
    CK(cudaEventRecord(e1, st));
    CK(cudaEventSynchronize(e1));
    float part = 0.f;
    CK(cudaEventElapsedTime(&part, e0, e1));
    ms += part;
    return SNP_OK;
  }
};

// Runs systems [lo, hi) of the arena (sparse form) to their end on st.
int many_group(BatchArena* arena, std::vector<BatchSys>& sys, const int64_t* c0_off, int32_t lo, int32_t hi,
               const BatchPlan& plan, uint32_t qc, PinnedState& pin, cudaEvent_t* evs, BatchTimer* timer,
               int64_t* launches, cudaStream_t st, int nsm) {
  const int32_t n = hi - lo;
  std::vector<int> ms(n);
  for (int32_t i = 0; i < n; ++i) ms[i] = sys[lo + i].sys.m;
  const ManyPlan mp = many_plan(ms.data(), n, plan.tile, plan.warps);
  // runs of about a quarter of a warp's share of a full pass, 64 to 128
  // candidates (512 systems: 57.7 ms with 352, 50.2 with 128, 56.2 with 64)
  const uint64_t warps = (uint64_t)nsm * mp.ctas_per_sm * mp.warps;
  const uint32_t run = (uint32_t)std::min<uint64_t>(128, std::max<uint64_t>(64, ((uint64_t)n * qc / (4 * warps) + 31) / 32 * 32));
  size_t at = 0;
  int64_t items = 0;
  for (int32_t i = lo; i < hi; ++i) {
    BatchSys& b = sys[i];
    many_carve(b, arena->scratch.as<unsigned char>() + at, qc, run);
    at += many_scratch_bytes(b.cap, qc, b.sys.m);
    b.tile = many_tile(mp, b.sys.m, plan.tile);
    b.fixed_q = plan.qc > 0 ? 1 : 0;
    items += many_items(b.cap, qc, run);
  }
  TRY(arena->items.reserve(sizeof(int2) * (2 * kMqForms + 3) * items));
  TRY(arena->queue.reserve(sizeof(uint32_t) * kMqCounters));
  ManyQueue q;
  q.expand[0] = arena->items.as<int2>();
  q.expand[1] = q.expand[0] + kMqForms * items;
  q.copy = q.expand[1] + kMqForms * items;
  q.psi[0] = q.copy + items;
  q.psi[1] = q.psi[0] + items;
  q.ctr = arena->queue.as<uint32_t>();
  q.cap = items;
  if (timer) TRY(timer->start(st));
  BatchSys* dsys = arena->sys.as<BatchSys>() + lo;
  CK(cudaMemcpyAsync(dsys, sys.data() + lo, sizeof(BatchSys) * n, cudaMemcpyHostToDevice, st));
  CK(cudaMemsetAsync(q.ctr, 0, sizeof(uint32_t) * kMqCounters, st));
  launch_many_init(dsys, nullptr, arena->c0.as<int32_t>(), arena->c0_off.as<int64_t>() + lo, n, q, st);
  CK(cudaGetLastError());
  *launches += 1;
  // two iterations in flight: the count read back is the one before last
  uint32_t* active[2] = {reinterpret_cast<uint32_t*>(pin.slot[0]), reinterpret_cast<uint32_t*>(pin.slot[1])};
  for (int it = 0;; ++it) {
    if (it >= 2) {
      CK(cudaEventSynchronize(evs[it & 1]));
      if (*active[it & 1] == 0) break;
    }
    *launches += launch_many_iteration(dsys, n, q, it & 1, mp, st, nsm);
    CK(cudaGetLastError());
    CK(cudaMemcpyAsync(active[it & 1], q.ctr + kMqActive, sizeof(uint32_t), cudaMemcpyDeviceToHost, st));
    CK(cudaEventRecord(evs[it & 1], st));
  }
  if (timer) TRY(timer->stop(st));
  CK(cudaStreamSynchronize(st));
  return SNP_OK;
}

int batch_setup(snp_handle* hs, int32_t n, const snp_explore_opts* o) {
  if (!hs || n < 1 || !o) return fail(SNP_E_INVALID, "bad arguments");
  if (o->depth < 0) return fail(SNP_E_INVALID, "depth = %d < 0", o->depth);
  if (o->transition == SNP_T_TC_I8)
    return fail(SNP_E_INVALID, "the batch engine's tensor-core form is SNP_T_TC_F8 (tcgen05 has no int8 kind on this GPU)");
  if (o->transition != SNP_T_SPARSE_I32 && o->transition != SNP_T_TC_F8)
    return fail(SNP_E_INVALID, "unknown transition %d", o->transition);
  if (o->record_parents) return fail(SNP_E_INVALID, "the batch engine keeps no parent records");
  if (o->frontier_cap < 1 || o->frontier_cap > (1 << 20))
    return fail(SNP_E_INVALID, "the batch engine needs 1 <= frontier_cap <= 2^20 (got %lld)", (long long)o->frontier_cap);
  int dev = 0;
  CK(cudaGetDevice(&dev));
  for (int32_t i = 0; i < n; ++i) {
    if (!hs[i]) return fail(SNP_E_INVALID, "handle %d is NULL", i);
    if (hs[i]->device != dev) return fail(SNP_E_INVALID, "handle %d lives on device %d, not %d", i, hs[i]->device, dev);
    if (o->transition == SNP_T_TC_F8) {
      if (hs[i]->max_abs_m > 16)
        return fail(SNP_E_RANGE, "fp8 transition refused: |M_Pi| of system %d reaches %d > 16", i, hs[i]->max_abs_m);
      if ((hs[i]->R + 31) / 32 > 1024) return fail(SNP_E_INVALID, "system %d has more than 32768 rules", i);
      TRY(tc5_prepare(hs[i], 0));
    }
  }
  return SNP_OK;
}

// Tensor-core form: depth launches, captured once per arena and replayed as one graph.
int run_tc_depths(BatchArena* arena, const std::vector<BatchSys>& sys, const BatchArgs& args, int blocks, int depth,
                  bool fresh, size_t scratch_stride, BatchTimer* timer, cudaStream_t st, int nsm) {
  const int32_t n = (int32_t)sys.size();
  CK(cudaMemcpyAsync(arena->sys.p, sys.data(), sizeof(BatchSys) * n, cudaMemcpyHostToDevice, st));
  CK(cudaMemsetAsync(arena->queue.p, 0, sizeof(unsigned int) * (depth + 1), st));
  if (fresh) CK(cudaMemsetAsync(arena->scratch.p, 0, scratch_stride * blocks, st));  // bitmaps start (and stay) clear
  k_batch_init<<<grid_for(n, 8, nsm * 16), 256, 0, st>>>(arena->sys.as<BatchSys>(), arena->c0.as<int32_t>(),
                                                          arena->c0_off.as<int64_t>(), n);
  CK(cudaGetLastError());
  if (!arena->exec) {
    BatchArgs a = args;
    cudaStream_t cap_st = nullptr;
    CK(cudaStreamCreateWithFlags(&cap_st, cudaStreamNonBlocking));
    cudaGraph_t graph = nullptr;
    CK(cudaStreamBeginCapture(cap_st, cudaStreamCaptureModeThreadLocal));
    for (int d = 1; d <= depth; ++d) {
      a.launch = d;
      launch_batch_depth_tc(a, blocks, cap_st);
    }
    cudaError_t ce = cudaStreamEndCapture(cap_st, &graph);
    if (ce == cudaSuccess) ce = cudaGraphInstantiate(&arena->exec, graph, 0);
    if (graph) cudaGraphDestroy(graph);
    cudaStreamDestroy(cap_st);
    if (ce != cudaSuccess) {
      arena->exec = nullptr;
      return fail(SNP_E_CUDA, "batch graph: %s", cudaGetErrorString(ce));
    }
  }
  if (timer) TRY(timer->start(st));
  cudaError_t ce = cudaGraphLaunch(arena->exec, st);
  if (timer && ce == cudaSuccess) TRY(timer->stop(st));
  if (ce == cudaSuccess) ce = cudaStreamSynchronize(st);
  if (ce != cudaSuccess) return fail(SNP_E_CUDA, "batch run: %s", cudaGetErrorString(ce));
  return SNP_OK;
}

// Runs depths 1..depth of the batch (all handles) with the given plan; fills
// the handles' results.  timer (optional) receives the device time of the depths.
int batch_run(snp_handle* hs, int32_t n, const snp_explore_opts* o, const BatchPlan& plan, int32_t* statuses,
              BatchTimer* timer) {
  const int dev = hs[0]->device;
  CK(cudaSetDevice(dev));
  cudaStream_t st = static_cast<cudaStream_t>(o->stream);
  const int nsm = sm_count(dev);
  const int64_t cap = o->frontier_cap;
  const int depth = o->depth;
  const bool tc = o->transition == SNP_T_TC_F8;
  int m_max = 1;
  for (int32_t i = 0; i < n; ++i) m_max = std::max(m_max, hs[i]->m);
  const int64_t rows_per = 1 + (int64_t)depth * cap;
  // passes: the caller's size, else up to 2048 in the tensor-core form and by the cap in the sparse form
  const uint32_t qs = plan.qc > 0 ? plan.qc : 2048;  // claims past the cap the table has room for, per depth
  const uint32_t qc = plan.qc > 0 ? plan.qc : tc ? 2048 : many_default_qc(cap);
  const uint64_t want_slots = (uint64_t)((long double)(rows_per + (int64_t)depth * qs) * 4.0L / 3.0L) + kBucket;
  const uint64_t nslots = std::max<uint64_t>(pow2_at_least(want_slots), kBucket);
  // tensor-core form: two CTAs of 128 TMEM columns per SM
  const int blocks = std::max(1, std::min<int>(nsm * 2, n));
  const size_t scratch_stride = tc ? (batch_scratch_bytes(cap, qc, m_max) + 255) & ~size_t(255) : 0;

  size_t pool_bytes = 0;
  std::vector<size_t> pool_off(n);
  for (int32_t i = 0; i < n; ++i) {
    pool_off[i] = pool_bytes;
    pool_bytes += ((size_t)rows_per * hs[i]->m * sizeof(int32_t) + 255) & ~size_t(255);
  }
  // Reuse the arena (and its graph) of the previous batch over the same handles and shape.
  std::shared_ptr<BatchArena> arena = hs[0]->batch;
  bool same = arena && arena->n == n && arena->depth == depth && arena->cap == cap &&
              arena->budget == (o->candidate_budget > 0 ? o->candidate_budget : 0) &&
              arena->max_expand == o->max_expand_value && arena->blocks == blocks && arena->qc == qc &&
              arena->nslots == nslots && arena->pool_bytes == pool_bytes &&
              arena->scratch_stride == scratch_stride && arena->tc == (tc ? 1 : 0);
  for (int32_t i = 0; same && i < n; ++i) same = arena->handles[i] == hs[i] && hs[i]->batch == arena;
  if (!same) {
    arena = std::make_shared<BatchArena>();
    arena->n = n;
    arena->depth = depth;
    arena->handles.assign(hs, hs + n);
    arena->cap = cap;
    arena->budget = o->candidate_budget > 0 ? o->candidate_budget : 0;
    arena->max_expand = o->max_expand_value;
    arena->blocks = blocks;
    arena->qc = qc;
    arena->nslots = nslots;
    arena->pool_bytes = pool_bytes;
    arena->scratch_stride = scratch_stride;
    arena->tc = tc ? 1 : 0;
    for (int32_t i = 0; i < n; ++i) {  // release older arenas before allocating
      hs[i]->batch.reset();
      hs[i]->result_pool = nullptr;
      hs[i]->result_perm = nullptr;
      hs[i]->explored = false;
    }
  }
  TRY(arena->sys.reserve(sizeof(BatchSys) * n));
  TRY(arena->stats.reserve(sizeof(BatchDepthStat) * n * (depth + 1)));
  TRY(arena->pools.reserve(pool_bytes));
  TRY(arena->slots.reserve(sizeof(unsigned long long) * nslots * n));
  if (tc) {
    TRY(arena->scratch.reserve(scratch_stride * blocks));
    TRY(arena->queue.reserve(sizeof(unsigned int) * (depth + 1)));
  }
  std::vector<int32_t> c0;
  std::vector<int64_t> c0_off(n);
  std::vector<BatchSys> sys(n);
  for (int32_t i = 0; i < n; ++i) {
    snp_system* h = hs[i];
    c0_off[i] = (int64_t)c0.size();
    c0.insert(c0.end(), h->c0.begin(), h->c0.end());
    BatchSys& b = sys[i];
    std::memset(&b, 0, sizeof b);
    b.sys = h->dev();
    b.pool = reinterpret_cast<int32_t*>(arena->pools.as<char>() + pool_off[i]);
    b.slots = arena->slots.as<unsigned long long>() + (size_t)i * nslots;
    b.bmask = nslots / kBucket - 1;
    b.pool_rows = rows_per;
    b.level_lo = 0;
    b.level_hi = 1;
    b.n_rows = 1;
    b.cur_depth = 0;
    b.target_depth = depth;
    b.max_expand = o->max_expand_value;
    b.cap = cap;
    b.budget = o->candidate_budget > 0 ? o->candidate_budget : 0;
    b.stats = arena->stats.as<BatchDepthStat>() + (size_t)i * (depth + 1);
    b.MB = tc ? h->d_MB.as<uint8_t>() : nullptr;
    b.np = h->t5_np;
    b.nblocks = h->t5_nblocks;
    b.overshoot = qs;
  }
  TRY(arena->c0.reserve(sizeof(int32_t) * c0.size()));
  TRY(arena->c0_off.reserve(sizeof(int64_t) * n));
  CK(cudaMemcpyAsync(arena->c0.p, c0.data(), sizeof(int32_t) * c0.size(), cudaMemcpyHostToDevice, st));
  CK(cudaMemcpyAsync(arena->c0_off.p, c0_off.data(), sizeof(int64_t) * n, cudaMemcpyHostToDevice, st));
  CK(cudaMemsetAsync(arena->stats.p, 0, sizeof(BatchDepthStat) * n * (depth + 1), st));
  k_fill_u64<<<grid_for((int64_t)(nslots * n), 256, nsm * 32), 256, 0, st>>>(arena->slots.as<unsigned long long>(),
                                                                             nslots * n, kEmpty);
  CK(cudaGetLastError());
  BatchArgs a;  // tensor-core form
  std::memset(&a, 0, sizeof a);
  a.sys = arena->sys.as<BatchSys>();
  a.n = n;
  a.qc = qc;
  a.queue = arena->queue.as<unsigned int>();
  a.scratch = arena->scratch.as<unsigned char>();
  a.scratch_stride = scratch_stride;
  a.pmax = cap;
  a.m_max = m_max;
  int rc = SNP_OK;
  int64_t launches = 1;  // the tables' fill above
  if (tc) {
    launches += 1 + depth;
    rc = run_tc_depths(arena.get(), sys, a, blocks, depth, !same, scratch_stride, timer, st, nsm);
  } else {
    // groups of systems whose scratch fits kGroupScratch; with little memory
    // left, smaller groups (down to one system) and passes of 2048
    size_t limit = kGroupScratch;
    uint32_t q = qc;
    for (int32_t lo = 0; lo < n && rc == SNP_OK;) {
      int32_t hi = lo;
      size_t need = 0;
      while (hi < n) {
        const size_t one = many_scratch_bytes(cap, q, hs[hi]->m);
        if (hi > lo && need + one > limit) break;
        need += one;
        ++hi;
      }
      rc = arena->scratch.reserve(need);
      if (rc == SNP_E_NOMEM && (hi > lo + 1 || q > qs)) {
        limit = std::min(limit, need) / 4;
        q = std::min(q, std::max<uint32_t>(qs, 1));
        rc = SNP_OK;
        g_err.clear();  // not a failure of the call
        continue;
      }
      if (rc == SNP_OK)
        rc = many_group(arena.get(), sys, c0_off.data(), lo, hi, plan, q, hs[0]->pin, hs[0]->evs, timer, &launches, st,
                        nsm);
      lo = hi;
    }
  }
  if (rc != SNP_OK) return rc;
  if (arena->scratch.bytes > kKeptScratch) arena->scratch.release();
  // results
  std::vector<BatchDepthStat> stats((size_t)n * (depth + 1));
  CK(cudaMemcpy(sys.data(), arena->sys.p, sizeof(BatchSys) * n, cudaMemcpyDeviceToHost));
  CK(cudaMemcpy(stats.data(), arena->stats.p, sizeof(BatchDepthStat) * stats.size(), cudaMemcpyDeviceToHost));
  for (int32_t i = 0; i < n; ++i) {
    snp_system* h = hs[i];
    const BatchSys& b = sys[i];
    h->stats.clear();
    snp_depth_info s0;
    std::memset(&s0, 0, sizeof s0);
    s0.new_configs = 1;
    s0.launches = launches;
    h->stats.push_back(s0);
    int64_t lo = 0, hi = 1;
    for (int d = 1; d <= depth; ++d) {
      const BatchDepthStat& x = stats[(size_t)i * (depth + 1) + d];
      if (d > 1 && h->stats.back().new_configs == 0) break;
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
    h->batch = arena;
    h->result_pool = b.pool;
    h->result_perm = nullptr;
    h->result_w = 4;
    int code = SNP_OK;
    if (b.error & kErrOverflow) code = SNP_E_OVERFLOW;
    else if (b.error & kErrTimeout) code = SNP_E_TIMEOUT;
    else if (b.error) code = SNP_E_INTERNAL;
    if (statuses) statuses[i] = code;
  }
  return SNP_OK;
}

}  // namespace

extern "C" int snp_explore_batch(snp_handle* hs, int32_t n, const snp_explore_opts* o, int32_t* statuses) {
  g_err.clear();
  TRY(batch_setup(hs, n, o));
  BatchPlan plan;
  if (o->chunk > 0) plan.qc = (uint32_t)std::min<int64_t>(o->chunk, 1 << 16);
  if (o->tile > 0) plan.tile = std::min(o->tile, 32);
  if (o->warps > 0) plan.warps = o->warps;
  return batch_run(hs, n, o, plan, statuses, nullptr);
}

extern "C" int snp_batch_autotune(snp_handle* hs, int32_t n, const snp_explore_opts* o, int32_t* chunk, int32_t* tile,
                                  int32_t* warps) {
  g_err.clear();
  TRY(batch_setup(hs, n, o));
  if (!chunk || !tile || !warps) return fail(SNP_E_INVALID, "bad arguments");
  snp_explore_opts t = *o;
  t.depth = std::min(o->depth, 2);
  std::vector<uint32_t> qcs = {1024, 2048, 4096};
  // what the sparse form takes by itself for a large cap (64 systems, cap 2^14: 24 ms, 60 ms with passes of 4096)
  if (o->transition == SNP_T_SPARSE_I32 && many_default_qc(o->frontier_cap) > qcs.back())
    qcs.push_back(many_default_qc(o->frontier_cap));
  const int tiles[] = {8, 16, 32};
  const int ws[] = {4, 8};
  const bool tc = o->transition == SNP_T_TC_F8;  // the tensor-core form: tile and warps are fixed
  float best = 1e30f;
  BatchPlan bestp;
  for (uint32_t qc : qcs)
    for (int tl : tiles)
      for (int w : ws) {
        if (tc && (tl != tiles[0] || w != ws[0])) continue;
        BatchPlan p;
        p.qc = qc;
        p.tile = tl;
        p.warps = w;
        BatchTimer timer;
        TRY(batch_run(hs, n, &t, p, nullptr, &timer));
        if (timer.ms < best) {
          best = timer.ms;
          bestp = p;
        }
      }
  *chunk = (int32_t)bestp.qc;
  *tile = bestp.tile;
  *warps = bestp.warps;
  for (int32_t i = 0; i < n; ++i) {
    hs[i]->batch.reset();
    hs[i]->result_pool = nullptr;
    hs[i]->result_perm = nullptr;
    hs[i]->explored = false;
  }
  return SNP_OK;
}
