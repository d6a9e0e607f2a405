// Sparse form of the batch engine and the serving loop: many independent
// systems advance together through work shared by the whole grid.
//
// An iteration is six launches over all systems:
//   k_many_psi      step (a) of new frontiers: Psi, a warp per 32 rows (two
//                   launches: without and with the parents' records);
//   k_many_scan     a CTA per system with a new frontier: the saturating scan
//                   of Psi, the depth's candidates, its first pass;
//   k_many_expand   steps (b)-(d) of every system's pass: warps take runs of
//                   candidates, whatever system they belong to, from one
//                   queue (device code of snp_expand.cuh; rows of more than
//                   kWideM neurons in the wide mode);
//   k_many_control  a CTA per system with a pass: first-occurrence marks,
//                   ranks, what the cap accepts, the next pass or frontier;
//   k_many_copy     accepted rows to their pool rows, table slots pointed at
//                   them, a warp per 8 first occurrences.
// Systems do not wait for one another: each is in its own depth and pass.
//
// Why a shared queue: with a CTA per system and depth, a depth lasted as long
// as its slowest system on one SM (a burst of 48 systems of up to 512 neurons
// left 104 SMs idle), and the tile of every system was as small as the widest
// one's.  48 requests of 8 to 512 neurons (depths 4 to 32, cap 2^12, budget
// 2^16): 618 ms -> 67 ms; 512 systems of 16 to 256 neurons to depth 6: 101 ms
// -> 49 ms.
#include <algorithm>

#include "snp_expand.cuh"

namespace snp {

namespace {

constexpr int kManyThreads = 256;           // psi, expand, copy
constexpr int kControlThreads = 1024;       // scan, control
constexpr uint32_t kManyMaxQ = 1u << 16;    // candidates of one pass of one system
constexpr uint32_t kCopyRows = 8;           // first occurrences per copy item: many short items keep more loads in flight
constexpr size_t kArgsBytes = 512;          // a warp's copy of its system's pass arguments
static_assert(sizeof(ClaimArgs) <= kArgsBytes && sizeof(ClaimArgs) % 8 == 0, "pass arguments");

// count elements of a system into a queue, `per` per item, by the whole CTA.
__device__ __forceinline__ void push_items(int2* items, uint32_t* ctr, int32_t si, uint64_t count, uint32_t per,
                                           uint32_t* s_base) {
  const uint32_t k = (uint32_t)((count + per - 1) / per);
  __syncthreads();
  if (threadIdx.x == 0) *s_base = k ? atomicAdd(ctr, k) : 0u;
  __syncthreads();
  const uint32_t base = *s_base;
  for (uint32_t i = threadIdx.x; i < k; i += blockDim.x) items[base + i] = make_int2(si, (int)(i * per));
}

// The expand form of rows of m neurons: wide ones first, their items take longest.
__device__ __forceinline__ int form_of(int m) { return (m > kWideM ? 0 : 2) + ((m & 3) == 0 ? 0 : 1); }

// Q candidates of a system's next pass into the queue of parity par.
__device__ __forceinline__ void push_pass(const ManyQueue& q, int par, const BatchSys& b, uint64_t Q,
                                          uint32_t* s_base) {
  const int form = form_of(b.sys.m);
  push_items(q.expand[par] + form * q.cap, q.ctr + kMqExpand + par * kMqForms + form, (int32_t)blockIdx.x, Q, b.a.run,
             s_base);
}

// Size of the next pass (one thread): what is left, what the scratch holds
// and, when the caller set no pass size, what the cap is expected to take.
// Claims past the cap become tombstones, so a pass never has more candidates
// than the cap still takes plus the table's room for this depth.
__device__ __forceinline__ void begin_pass(BatchSys& b) {
  uint64_t q = min(b.T - b.a.g0, (uint64_t)b.qc);
  if (!b.fixed_q) {
    const uint64_t room = (b.bmask + 1) * kBucket / 4 * 3;
    const int64_t left = b.target_depth - b.cur_depth;  // depths to finish, this one included
    const uint64_t used = (uint64_t)b.n_rows + b.tombs + b.remaining + (uint64_t)(left - 1) * (uint64_t)b.cap;
    const uint64_t over = max((uint64_t)b.overshoot, room > used ? (room - used) / (uint64_t)left : (uint64_t)0);
    q = min(q, b.remaining + over);
    const float want = (float)b.remaining / fmaxf(b.rate, 1.f / 1024.f) * 1.25f + 512.f;
    if (want < (float)q) q = (uint64_t)want;
  }
  b.a.Q = (uint32_t)q;
  b.phase = kPhaseExpand;
}

// The depth's record and the next frontier (one thread); returns its rows, 0
// when the system is finished.
__device__ __forceinline__ int64_t finish_depth(BatchSys& b, uint32_t* active) {
  const int32_t d = b.cur_depth + 1;
  BatchDepthStat* stat = b.stats + d;
  stat->new_configs = b.nnew;
  stat->examined = (int64_t)b.examined;
  stat->candidates = b.total;
  stat->truncated = b.examined < b.total ? 1 : 0;
  stat->chunks = b.chunks;
  b.cur_depth = d;
  if (b.nnew == 0) {
    b.done = 1;
  } else {
    b.depth_reached = d;
    b.level_lo = b.level_hi;
    b.level_hi = b.n_rows;
  }
  if (b.done || b.error || d >= b.target_depth) {
    b.phase = kPhaseIdle;
    atomicSub(active, 1u);
    return 0;
  }
  b.phase = kPhasePsi;
  b.a.parents = b.pool + (size_t)b.level_lo * b.sys.m;
  b.a.P = b.nnew;
  b.a.prec = b.few ? b.rec : nullptr;
  return b.nnew;
}

// expand_task out of line: its four forms in one kernel keep their registers
// to themselves (inlined together they spilled 1.4 KB).
template <class RF, int KIND>
__device__ __noinline__ void expand_item(const ClaimArgs& a, unsigned char* smem, int B, uint64_t la, uint64_t lb,
                                         WarpTask& k) {
  const int lane = threadIdx.x & 31, m = a.sys.m, ts = round4(m) + 4;
  ExpandSmem w = KIND == kWide ? expand_smem_wide(smem, m) : expand_smem(smem, m, B, ts);
  expand_task<RF, KIND>(a, a.P, a.Q, B, ts, w, la, lb, k, lane);
}

}  // namespace

__global__ void __launch_bounds__(kManyThreads) k_many_init(BatchSys* sys, const int32_t* idx, const int32_t* c0,
                                                            const int64_t* c0_off, int32_t n, ManyQueue q) {
  const int lane = threadIdx.x & 31;
  const int64_t nw = (int64_t)gridDim.x * (blockDim.x >> 5);
  for (int64_t i = (int64_t)blockIdx.x * (blockDim.x >> 5) + (threadIdx.x >> 5); i < n; i += nw) {
    const int32_t si = idx ? idx[i] : (int32_t)i;
    BatchSys& b = sys[si];
    const int m = b.sys.m;
    const int32_t* src = c0 + c0_off[i];
    for (int j = lane; j < m; j += 32) b.pool[j] = src[j];
    for (uint32_t w = lane; w < b.qc / 32 + 1; w += 32) b.a.ownbits[w] = 0u;
    __syncwarp();
    const uint64_t h = fingerprint(b.sys, b.pool, lane);
    if (lane == 0) {
      b.slots[(h & b.bmask) * kBucket] = (unsigned long long)fp32_of(h) << 32;  // row 0, in an empty table
      ChunkState z = {};
      *b.a.st = z;
      b.rate = 1.f;
      if (b.target_depth >= 1) {
        b.phase = kPhasePsi;
        b.a.parents = b.pool;
        b.a.P = 1;
        b.few = 1;
        b.a.prec = b.rec;
        q.psi[1][atomicAdd(q.ctr + kMqPsi + 1, 1u)] = make_int2(si, 0);
        atomicAdd(q.ctr + kMqActive, 1u);
      } else {
        b.phase = kPhaseIdle;
      }
    }
  }
}

// Step (a): a warp takes 32 frontier rows and moves them through shared
// memory 32 columns at a time (a row's slab is one coalesced 128-byte load,
// the 32 rows' loads in flight together); lane r then visits row r's slab at
// a stride of 33 words.  With fewer items than warps, two or four warps share
// an item's rows and two or four lanes a row's columns: a row of 512 neurons
// is 64 batches of lookups for one lane, the length of the launch.
// REC: the rows' parent records too, in neuron order (systems whose last depth
// had few candidates per parent; the others' rows take fewer registers and
// lookups).
template <bool REC>
__global__ void __launch_bounds__(kManyThreads, REC ? 2 : 3) k_many_psi(BatchSys* sys, ManyQueue q) {
  __shared__ int32_t slabs[kManyThreads / 32][32][33];
  const int lane = threadIdx.x & 31, wib = threadIdx.x >> 5;
  int32_t(*slab)[33] = slabs[wib];
  const uint32_t count = __ldcg(q.ctr + kMqPsi + (REC ? 1 : 0));
  const uint32_t nw = gridDim.x * (blockDim.x >> 5);
  // log2 of the lanes per row
  const int sl = REC || count > nw / 2 ? 0 : count > nw / 4 ? 1 : 2;
  const int rows_per = 32 >> sl;                      // rows of a warp's share = columns of a lane's
  const int r = lane & (rows_per - 1), part = lane >> (5 - sl);
  for (uint32_t it = blockIdx.x * (blockDim.x >> 5) + wib; it < count << sl; it += nw) {
    const int2 item = __ldcg(q.psi[REC ? 1 : 0] + (it >> sl));
    BatchSys& b = sys[item.x];
    const DevSys s = b.sys;
    const int m = s.m;
    const int64_t p0 = (int64_t)item.y + (int64_t)(it & ((1u << sl) - 1u)) * rows_per;
    const int nr = (int)max((int64_t)0, min((int64_t)rows_per, b.a.P - p0));
    const int32_t* rows = b.a.parents + (size_t)p0 * m;
    ParentRec* rec = REC ? b.rec + p0 + r : nullptr;
    const int32_t max_expand = b.max_expand;
    PsiAcc acc;
    for (int n0 = 0; n0 < m && nr > 0; n0 += 32) {
      const int w = min(32, m - n0);
      __syncwarp();
      if (lane < w) {
        for (int r0 = 0; r0 < nr; r0 += 8) {
          int32_t v[8];
#pragma unroll
          for (int u = 0; u < 8; ++u)
            if (r0 + u < nr) v[u] = __ldcg(rows + (size_t)(r0 + u) * m + n0 + lane);
#pragma unroll
          for (int u = 0; u < 8; ++u)
            if (r0 + u < nr) slab[r0 + u][lane] = v[u];
        }
      }
      __syncwarp();
      const int c0 = part * rows_per, cw = min(rows_per, w - c0);
      if (r < nr && cw > 0) acc.visit_run<REC>(s, n0 + c0, slab[r] + c0, cw, max_expand, rec);
    }
    uint64_t prod = acc.prod;
    bool skip = acc.skip, ov = acc.ov;
    for (int o = rows_per; o < 32; o <<= 1) {  // a row's lanes together
      prod = sat_mul(prod, __shfl_xor_sync(0xffffffffu, prod, o));
      skip |= __shfl_xor_sync(0xffffffffu, skip ? 1 : 0, o) != 0;
      ov |= __shfl_xor_sync(0xffffffffu, ov ? 1 : 0, o) != 0;
    }
    if (part == 0 && r < nr) {
      b.off[p0 + r] = skip ? 0ull : prod;
      if (REC) {
        rec->hbase = acc.hb;
        rec->nnt = acc.nnt;
      }
    }
    if (__any_sync(0xffffffffu, r < nr && ov && !skip) && lane == 0) atomicOr(&b.error, kErrOverflow);
  }
}

__global__ void __launch_bounds__(kControlThreads) k_many_scan(BatchSys* sys, ManyQueue q, int par) {
  __shared__ uint64_t wsum[kControlThreads / 32];
  __shared__ uint32_t s_base;
  __shared__ uint64_t s_q;
  if (blockIdx.x == 0 && threadIdx.x == 0) {  // consumed: the psi items of this iteration, the copy items of the last
    q.ctr[kMqPsi] = 0;
    q.ctr[kMqPsi + 1] = 0;
    q.ctr[kMqCopy] = 0;
  }
  BatchSys& b = sys[blockIdx.x];
  if (b.phase != kPhasePsi) return;
  const int64_t P = b.a.P;
  if (threadIdx.x == 0) b.off[P] = 0;
  __syncthreads();
  block_scan_sat(b.off, P + 1, wsum);
  __syncthreads();
  if (threadIdx.x == 0) {
    const uint64_t total = b.off[P];
    b.total = total;
    b.few = total <= 256ull * (uint64_t)P ? 1 : 0;
    b.T = b.budget > 0 ? min(total, (uint64_t)b.budget) : total;
    b.remaining = (uint64_t)b.cap;
    b.a.g0 = 0;
    b.nnew = 0;
    b.examined = 0;
    b.chunks = 0;
    s_q = 0;
    if (b.T == 0 || b.error) {
      finish_depth(b, q.ctr + kMqActive);
    } else {
      begin_pass(b);
      s_q = b.a.Q;
    }
  }
  __syncthreads();
  push_pass(q, par, b, s_q, &s_base);
}

// Steps (b)-(d): a warp takes runs of candidates from the queue and works on
// them with a copy of their system's pass arguments in shared memory.
// Registers bound it to 16 warps per SM (128 each), as k_expand.
__global__ void __launch_bounds__(kManyThreads, 2) k_many_expand(BatchSys* sys, ManyQueue q, int par,
                                                                 uint32_t warp_bytes) {
  extern __shared__ __align__(16) unsigned char smem_raw[];
  const int lane = threadIdx.x & 31, wib = threadIdx.x >> 5;
  unsigned char* base = smem_raw + (size_t)wib * (warp_bytes + kArgsBytes);
  ClaimArgs& a = *reinterpret_cast<ClaimArgs*>(base);
  unsigned char* smem = base + kArgsBytes;
  int32_t cur = -1;
  int B = 0;
  WarpTask k;
  // one form after the other: the code of one fits the instruction caches, and
  // warps in four forms at once mostly waited for instructions
  for (int form = 0; form < kMqForms; ++form) {
    const uint32_t count = __ldcg(q.ctr + kMqExpand + par * kMqForms + form);
    const int2* items = q.expand[par] + form * q.cap;
    while (count) {
      uint32_t it = 0;
      if (lane == 0) it = atomicAdd(q.ctr + kMqHead + par * kMqForms + form, 1u);
      it = __shfl_sync(0xffffffffu, it, 0);
      if (it >= count) break;
      const int2 item = __ldcg(items + it);
      if (item.x != cur) {
        cur = item.x;
        const BatchSys& b = sys[cur];
        __syncwarp();
        const unsigned long long* src = reinterpret_cast<const unsigned long long*>(&b.a);
        for (int i = lane; i < (int)(sizeof(ClaimArgs) / 8); i += 32)
          reinterpret_cast<unsigned long long*>(base)[i] = __ldcg(src + i);
        B = __ldcg(&b.tile);
        __syncwarp();
        k = WarpTask();
      }
      const uint64_t la = (uint32_t)item.y, lb = min(la + a.run, (uint64_t)a.Q);
      if (form == 0)
        expand_item<RowI32V, kWide>(a, smem, kWideB, la, lb, k);
      else if (form == 1)
        expand_item<RowI32, kWide>(a, smem, kWideB, la, lb, k);
      else if (form == 2)
        expand_item<RowI32V, 0>(a, smem, B, la, lb, k);
      else
        expand_item<RowI32, 0>(a, smem, B, la, lb, k);
    }
  }
}

__global__ void __launch_bounds__(kControlThreads) k_many_control(BatchSys* sys, ManyQueue q, int par) {
  __shared__ uint32_t bits[kManyMaxQ / 32], pre[kManyMaxQ / 32];
  __shared__ uint32_t wsum[kControlThreads / 32];
  __shared__ uint32_t s_base, s_last;
  __shared__ int64_t s_parents;
  __shared__ uint64_t s_q;
  BatchSys& b = sys[blockIdx.x];
  if (b.phase != kPhaseExpand) return;
  const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5, nwarps = kControlThreads / 32;
  const uint32_t Q = b.a.Q, nwords = (Q + 31) / 32;
  uint32_t* own = b.a.ownbits;
  const uint32_t* gmin = b.a.gmin;
  for (uint32_t w = tid; w < nwords; w += kControlThreads) bits[w] = 0u;
  if (tid == 0) s_last = 0;
  __syncthreads();
  // first occurrences: every owner names its key's first candidate
  for (uint32_t w = warp; w < nwords; w += nwarps) {
    const uint32_t word = own[w];
    __syncwarp();
    if (!word) continue;
    if (lane == 0) own[w] = 0u;
    if ((word >> lane) & 1u) {
      const uint32_t o = w * 32u + (uint32_t)lane;
      const uint32_t f = o < Q ? gmin[o] : 0xFFFFFFFFu;
      if (f >= Q) {  // not a claim of this pass: record and skip
        atomicOr(&b.a.st->error, kErrInternal);
      } else {
        atomicOr(bits + (f >> 5), 1u << (f & 31));
        b.srow[f] = o;
      }
    }
  }
  __syncthreads();
  // ranks: exclusive scan of the words' popcounts, two words per thread
  const uint32_t w0 = 2u * tid;
  const uint32_t c0 = w0 < nwords ? __popc(bits[w0]) : 0u, c1 = w0 + 1 < nwords ? __popc(bits[w0 + 1]) : 0u;
  uint32_t inc = c0 + c1;
#pragma unroll
  for (int o = 1; o < 32; o <<= 1) {
    const uint32_t y = __shfl_up_sync(0xffffffffu, inc, o);
    if (lane >= o) inc += y;
  }
  if (lane == 31) wsum[warp] = inc;
  __syncthreads();
  if (warp == 0) {
    uint32_t v = wsum[lane];
#pragma unroll
    for (int o = 1; o < 32; o <<= 1) {
      const uint32_t y = __shfl_up_sync(0xffffffffu, v, o);
      if (lane >= o) v += y;
    }
    wsum[lane] = v;
  }
  __syncthreads();
  const uint32_t before = (warp > 0 ? wsum[warp - 1] : 0u) + inc - c0 - c1;
  if (w0 < nwords) pre[w0] = before;
  if (w0 + 1 < nwords) pre[w0 + 1] = before + c0;
  const uint32_t found = wsum[nwarps - 1];
  const uint64_t accept = b.remaining;
  __syncthreads();
  for (uint32_t w = warp; w < nwords; w += nwarps) {
    const uint32_t word = bits[w];
    if (!((word >> lane) & 1u)) continue;
    const uint32_t f = w * 32u + (uint32_t)lane;
    const uint32_t rank = pre[w] + __popc(word & ((1u << lane) - 1u));
    b.order[rank] = b.srow[f];
    if ((uint64_t)rank + 1 == accept) s_last = f;
  }
  __syncthreads();
  if (tid == 0) {
    const uint64_t acc = min((uint64_t)found, accept);
    const bool capped = (uint64_t)found >= accept;
    b.copy_row0 = b.n_rows;
    b.copy_n = found;
    b.copy_acc = (uint32_t)acc;
    b.examined = capped ? b.a.g0 + s_last + 1 : b.a.g0 + Q;
    b.n_rows += (int64_t)acc;
    b.nnew += (int64_t)acc;
    b.remaining -= acc;
    b.tombs += found - acc;
    b.rate = (float)found / (float)Q;
    b.a.g0 += Q;
    b.chunks += 1;
    if (b.a.st->error) atomicOr(&b.error, b.a.st->error);
    s_q = 0;
    s_parents = 0;
    if (capped || b.a.g0 >= b.T || b.error) {
      s_parents = finish_depth(b, q.ctr + kMqActive);
    } else {
      begin_pass(b);
      s_q = b.a.Q;
    }
  }
  __syncthreads();
  push_items(q.copy, q.ctr + kMqCopy, (int32_t)blockIdx.x, found, kCopyRows, &s_base);
  push_items(q.psi[b.few], q.ctr + kMqPsi + b.few, (int32_t)blockIdx.x, (uint64_t)s_parents, 32u, &s_base);
  push_pass(q, par ^ 1, b, s_q, &s_base);
}

// Accepted first occurrences: the staged row to its pool row, the table slot
// pointed at it; the others' slots become tombstones.
__global__ void __launch_bounds__(kManyThreads) k_many_copy(BatchSys* sys, ManyQueue q, int par) {
  const int lane = threadIdx.x & 31, wib = threadIdx.x >> 5;
  if (blockIdx.x == 0 && threadIdx.x == 0) {  // this iteration's expand items are consumed
    for (int f = 0; f < kMqForms; ++f) {
      q.ctr[kMqExpand + par * kMqForms + f] = 0;
      q.ctr[kMqHead + par * kMqForms + f] = 0;
    }
  }
  const uint32_t count = __ldcg(q.ctr + kMqCopy);
  const uint32_t nw = gridDim.x * (blockDim.x >> 5);
  for (uint32_t it = blockIdx.x * (blockDim.x >> 5) + wib; it < count; it += nw) {
    const int2 item = __ldcg(q.copy + it);
    const BatchSys& b = sys[item.x];
    const int m = b.sys.m;
    const uint32_t r0 = (uint32_t)item.y, n = b.copy_n, acc = b.copy_acc;
    const uint32_t rank = r0 + (uint32_t)lane;
    if (lane < (int)kCopyRows && rank < n) {
      unsigned long long* slot = b.slots + b.a.slot_of[b.order[rank]];
      const unsigned long long hi = *slot & 0xFFFFFFFF00000000ull;
      *slot = hi | (rank < acc ? (uint32_t)(b.copy_row0 + rank) : kRowTomb);
    }
    if (r0 >= acc) continue;
    const uint32_t rows = min(kCopyRows, acc - r0);
    const uint32_t* order = b.order + r0;
    int32_t* dst = b.pool + (size_t)(b.copy_row0 + r0) * m;
    const int32_t* staging = b.a.staging;
    if ((m & 3) == 0) {
      const uint32_t per = (uint32_t)m >> 2, total = rows * per;
      const int4* s4 = reinterpret_cast<const int4*>(staging);
      int4* d4 = reinterpret_cast<int4*>(dst);
      for (uint32_t i0 = lane; i0 < total; i0 += 32 * 8) {  // eight loads in flight
        int4 v[8];
#pragma unroll
        for (int u = 0; u < 8; ++u) {
          const uint32_t i = i0 + 32u * u, r = i / per;
          if (i < total) v[u] = __ldcs(s4 + (size_t)order[r] * per + (i - r * per));
        }
#pragma unroll
        for (int u = 0; u < 8; ++u)
          if (i0 + 32u * u < total) d4[i0 + 32u * u] = v[u];
      }
    } else {
      const uint32_t per = (uint32_t)m, total = rows * per;
      for (uint32_t i0 = lane; i0 < total; i0 += 32 * 16) {
        int32_t v[16];
#pragma unroll
        for (int u = 0; u < 16; ++u) {
          const uint32_t i = i0 + 32u * u, r = i / per;
          if (i < total) v[u] = __ldcs(staging + (size_t)order[r] * per + (i - r * per));
        }
#pragma unroll
        for (int u = 0; u < 16; ++u)
          if (i0 + 32u * u < total) dst[i0 + 32u * u] = v[u];
      }
    }
  }
}

namespace {

size_t up256(size_t b) { return (b + 255) & ~size_t(255); }

// Shared memory per warp that leaves 16 warps on an SM (two CTAs of eight).
constexpr size_t kManyWarpBytes = 13312;

}  // namespace

uint32_t many_default_qc(int64_t cap) { return (uint32_t)std::min<int64_t>(kManyMaxQ, 2 * cap + 2048); }

size_t many_scratch_bytes(int64_t cap, uint32_t qc, int m) {
  return up256(sizeof(ChunkState)) + up256((size_t)(qc / 32 + 1) * 4) + up256((size_t)(cap + 1) * 8) +
         up256((size_t)cap * sizeof(ParentRec)) + up256((size_t)qc * m * 4) + 4 * up256((size_t)qc * 4);
}

void many_carve(BatchSys& b, unsigned char* base, uint32_t qc, uint32_t run) {
  size_t at = 0;
  auto take = [&](size_t bytes) {
    unsigned char* p = base + at;
    at += up256(bytes);
    return p;
  };
  ClaimArgs a;
  a.st = reinterpret_cast<ChunkState*>(take(sizeof(ChunkState)));
  a.ownbits = reinterpret_cast<uint32_t*>(take((size_t)(qc / 32 + 1) * 4));
  b.off = reinterpret_cast<uint64_t*>(take((size_t)(b.cap + 1) * 8));
  b.rec = reinterpret_cast<ParentRec*>(take((size_t)b.cap * sizeof(ParentRec)));
  a.staging = reinterpret_cast<int32_t*>(take((size_t)qc * b.sys.m * 4));
  a.gmin = reinterpret_cast<uint32_t*>(take((size_t)qc * 4));
  a.slot_of = reinterpret_cast<uint32_t*>(take((size_t)qc * 4));
  b.srow = reinterpret_cast<uint32_t*>(take((size_t)qc * 4));
  b.order = reinterpret_cast<uint32_t*>(take((size_t)qc * 4));
  a.sys = b.sys;
  a.parents = b.pool;
  a.pperm = nullptr;
  a.off = b.off;
  a.P = 0;
  a.g0 = 0;
  a.Q = 0;
  a.run = run;
  a.table = DevTable{b.slots, b.bmask};
  a.pool = b.pool;
  a.store_ctr = nullptr;
  a.sidx_of = nullptr;
  a.store_cap = 0;
  a.prec = b.rec;
  a.ctr = nullptr;
  b.a = a;
  b.qc = qc;
}

int64_t many_items(int64_t cap, uint32_t qc, uint32_t run) {
  return std::max<int64_t>({cap / 32 + 1, (int64_t)qc / run + 1, (int64_t)qc / kCopyRows + 1});
}

int many_tile(const ManyPlan& p, int m, int tile) {
  if (m > kWideM) return kWideB;
  const int ts = round4(m) + 4;
  int B = tile > 0 ? std::min(tile, 32) : 32;
  while (B > 1 && expand_warp_bytes(m, B, ts) > p.warp_bytes) --B;
  // a tile of 16 rows beats 17 to 31: blocks are products of choice counts, mostly 16
  return tile <= 0 && B > 16 && B < 32 ? 16 : B;
}

ManyPlan many_plan(const int32_t* ms, int64_t n, int tile, int warps) {
  ManyPlan p;
  size_t need = 0;  // the least shared memory a warp can do with
  size_t like = 0;  // with full tiles
  for (int64_t i = 0; i < n; ++i) {
    const int m = ms[i];
    const size_t least = m > kWideM ? expand_wide_bytes(m) : expand_warp_bytes(m, 1, round4(m) + 4);
    need = std::max(need, least);
    like = std::max(like, m > kWideM ? least : expand_warp_bytes(m, tile > 0 ? std::min(tile, 32) : 32, round4(m) + 4));
  }
  p.warp_bytes = (std::max(need, std::min(like, kManyWarpBytes)) + 15) & ~size_t(15);
  const size_t warp = p.warp_bytes + kArgsBytes;
  p.warps = warps == 4 || (warps != 8 && p.warp_bytes > kManyWarpBytes) ? 4 : 8;
  while (p.warps > 1 && warp * p.warps > (226u << 10)) p.warps /= 2;
  p.ctas_per_sm = (int)std::max<size_t>(1, std::min<size_t>(16 / p.warps, (227u << 10) / (warp * p.warps + 1024)));
  return p;
}

void launch_many_init(BatchSys* sys, const int32_t* idx, const int32_t* c0, const int64_t* c0_off, int32_t n,
                      const ManyQueue& q, cudaStream_t st) {
  const int per = kManyThreads / 32;
  k_many_init<<<std::min((n + per - 1) / per, 152 * 16), kManyThreads, 0, st>>>(sys, idx, c0, c0_off, n, q);
}

int launch_many_iteration(BatchSys* sys, int32_t n, const ManyQueue& q, int par, const ManyPlan& p, cudaStream_t st,
                           int nsm) {
  const size_t smem = (p.warp_bytes + kArgsBytes) * p.warps;
  allow_smem(k_many_expand);
  k_many_psi<false><<<nsm * 3, kManyThreads, 0, st>>>(sys, q);
  k_many_psi<true><<<nsm * 2, kManyThreads, 0, st>>>(sys, q);
  k_many_scan<<<n, kControlThreads, 0, st>>>(sys, q, par);
  k_many_expand<<<nsm * p.ctas_per_sm, p.warps * 32, smem, st>>>(sys, q, par, (uint32_t)p.warp_bytes);
  k_many_control<<<n, kControlThreads, 0, st>>>(sys, q, par);
  k_many_copy<<<nsm * 8, kManyThreads, 0, st>>>(sys, q, par);
  return 6;
}

}  // namespace snp
