// The batch engine's tensor-core form (the sparse form: snp_many.cu).
#include <algorithm>

#include "snp_expand.cuh"
#include "snp_tcgen05.cuh"

// One launch runs depth d of every system of a batch.  A CTA takes systems
// from a work queue; for each it runs the whole depth with block barriers in
// place of the host: Psi of its frontier (Eq. psi), the saturating scan, then
// passes of up to qc candidates -- rows by tensor core, resolve,
// first-occurrence marks, ranks, commit -- until the frontier cap, the
// candidate budget or the candidates run out.

namespace snp {

namespace {

struct BatchScratch {
  uint64_t* psi;   // [pmax + 1]
  uint64_t* off;   // [pmax + 1]
  int32_t* staging;
  uint32_t *gmin, *slot_of, *srow, *own, *bits, *wbase;
  ChunkState* st;
  unsigned long long* hash;  // [qc] tensor-core form: linear hash of each candidate's row
  uint8_t* red;              // [qc] tensor-core form: the candidate repeats an earlier one
};

__device__ __forceinline__ BatchScratch batch_scratch(unsigned char* base, int64_t pmax, uint32_t qc, int m_max) {
  size_t at = 0;
  auto take = [&](size_t bytes) {
    unsigned char* p = base + at;
    at += (bytes + 255) & ~size_t(255);
    return p;
  };
  BatchScratch b;
  const int64_t npsi = (pmax + 1) > (int64_t)(qc / 32 + 1) ? (pmax + 1) : (int64_t)(qc / 32 + 1);
  b.psi = reinterpret_cast<uint64_t*>(take((size_t)npsi * 8));
  b.off = reinterpret_cast<uint64_t*>(take((pmax + 1) * 8));
  b.staging = reinterpret_cast<int32_t*>(take((size_t)qc * m_max * 4));
  b.gmin = reinterpret_cast<uint32_t*>(take(qc * 4));
  b.slot_of = reinterpret_cast<uint32_t*>(take(qc * 4));
  b.srow = reinterpret_cast<uint32_t*>(take(qc * 4));
  b.own = reinterpret_cast<uint32_t*>(take((qc / 32 + 1) * 4));
  b.bits = reinterpret_cast<uint32_t*>(take((qc / 32 + 1) * 4));
  b.wbase = reinterpret_cast<uint32_t*>(take((qc / 32 + 1) * 4));
  b.st = reinterpret_cast<ChunkState*>(take(sizeof(ChunkState)));
  b.hash = reinterpret_cast<unsigned long long*>(take((size_t)qc * 8));
  b.red = reinterpret_cast<uint8_t*>(take(qc));
  return b;
}

// ---------------------------------------------------------------------------
// Tensor-core form of a batch pass (SNP_T_TC_F8): the rows of candidates
// g0 .. g0 + Q - 1 of the CTA's current system, C' = C_p + S . M_Pi
// (Eq. next-config) with the 0/1 spiking vector S of every firing neuron, by
// tcgen05.mma kind::f8f6f4 over tiles of 128 candidates (one thread and one
// TMEM lane per candidate), into the CTA's staging rows, with their linear
// hashes and repeat flags; the pass then resolves them like the sparse form.
// The MMA waits synchronously (the batch's CTAs overlap one another).

constexpr int kBtcSlots = 8;  // rule blocks of the left operand held at once

struct BatchTcSmem {
  uint8_t* A;          // [kBtcSlots][4096] left operand
  uint8_t* B;          // [kBtcSlots][128 * 32] M_Pi^T blocks of one 128-column chunk
  uint32_t* bitmap;    // [32] active rule blocks (at most 1024 blocks)
  uint16_t* slot_of;   // [1024]
  uint16_t* act;       // [1024]
  int* nact;
  unsigned long long* bars;  // operand arrival, MMA completion
  uint32_t* tmem_slot;
};

__host__ __device__ inline size_t batch_tc_smem_bytes() {
  return (size_t)kBtcSlots * t5::kT5ABytes * 2 + 32 * 4 + 1024 * 2 * 2 + 16 + 16 + 16 + 256;
}

__device__ __forceinline__ BatchTcSmem batch_tc_smem(unsigned char* raw) {
  unsigned char* p = reinterpret_cast<unsigned char*>(((uintptr_t)raw + 1023) & ~(uintptr_t)1023);
  BatchTcSmem w;
  w.A = p;
  p += (size_t)kBtcSlots * t5::kT5ABytes;
  w.B = p;
  p += (size_t)kBtcSlots * t5::kT5ABytes;
  w.bitmap = reinterpret_cast<uint32_t*>(p);
  p += 32 * 4;
  w.slot_of = reinterpret_cast<uint16_t*>(p);
  p += 1024 * 2;
  w.act = reinterpret_cast<uint16_t*>(p);
  p += 1024 * 2;
  w.nact = reinterpret_cast<int*>(p);
  p += 16;
  w.bars = reinterpret_cast<unsigned long long*>(p);
  p += 16;
  w.tmem_slot = reinterpret_cast<uint32_t*>(p);
  return w;
}

// Chosen rule of every neuron of parent row prow for candidate t (last
// neuron least significant): f(rule or -1, mask, spikes, neuron).  Returns
// false if t is not a valid index.
template <typename F>
__device__ __forceinline__ bool batch_walk(const DevSys& s, const int32_t* prow, uint64_t t, F&& f) {
  uint64_t q = t;
  for (int n = s.m - 1; n >= 0; --n) {
    const int32_t x = prow[n];
    const uint32_t mask = (uint32_t)appl(s, n, x);
    if (!mask) {
      f(-1, 0u, x, n);
      continue;
    }
    const uint32_t radix = (uint32_t)__popc(mask);
    uint32_t d = 0;
    if (radix > 1) {
      d = (uint32_t)(q % radix);
      q /= radix;
    }
    f(__ldg(s.first_rule + n) + nth_set_bit(mask, (int)d), mask, x, n);
  }
  return q == 0;
}

// Rows of the pass by tensor core; returns false when an mbarrier wait ran
// out (the CTA then stops: products may still be in flight).
__device__ bool batch_tc_rows(const ClaimArgs& a, const BatchSys* bs, const BatchTcSmem& w, uint32_t tmem,
                              unsigned long long* hash, uint8_t* red_out, uint32_t& ph_b, uint32_t& ph_m) {
  using namespace t5;
  const DevSys& s = a.sys;
  const int m = s.m, tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
  const int np = bs->np, nblocks = bs->nblocks;
  const int nbw = (nblocks + 31) / 32, nchunks = (np + kT5NC - 1) / kT5NC;
  const uint32_t bar_b = saddr(w.bars), bar_m = saddr(w.bars + 1);
  const uint32_t ntiles = (a.Q + kT5M - 1) / kT5M;
  for (uint32_t tile = 0; tile < ntiles; ++tile) {
    const uint32_t lid = tile * kT5M + tid;
    const bool valid = lid < a.Q;
    const uint64_t g = a.g0 + (valid ? lid : tile * kT5M);
    // parent: largest p with off[p] <= g
    int64_t lo = 0, hi = a.P;
    while (hi - lo > 1) {
      const int64_t mid = lo + (hi - lo) / 2;
      if (__ldcg(a.off + mid) <= g) lo = mid;
      else hi = mid;
    }
    const int32_t* prow = a.parents + (size_t)lo * m;
    const uint64_t t = g - __ldcg(a.off + lo);
    for (int i = tid; i < nbw; i += kT5M) w.bitmap[i] = 0u;
    __syncthreads();
    uint64_t h = 0;
    bool red = false;
    if (valid) {
      const bool ok = batch_walk(s, prow, t, [&](int r, uint32_t mask, int32_t x, int n) {
        h += col_hash(s, n, x);
        if (r < 0) return;
        atomicOr(w.bitmap + (r >> 10), 1u << ((r >> 5) & 31));
        h += __ldg(s.rowkey + r);
        red |= redundant_choice(s, mask, r);
      });
      if (!ok) atomicOr(&a.st->error, kErrInternal);
      hash[lid] = h;
      red_out[lid] = red ? 1 : 0;
    }
    __syncthreads();
    if (warp == 0) {
      int cnt = 0;
      for (int b0 = 0; b0 < nblocks; b0 += 32) {
        const int bk = b0 + lane;
        const bool on = bk < nblocks && ((w.bitmap[bk >> 5] >> (bk & 31)) & 1u);
        const uint32_t bb = __ballot_sync(0xffffffffu, on);
        if (on) {
          const int pos = cnt + __popc(bb & ((1u << lane) - 1u));
          w.act[pos] = (uint16_t)bk;
          w.slot_of[bk] = (uint16_t)pos;
        }
        cnt += __popc(bb);
      }
      if (lane == 0) *w.nact = cnt;
    }
    __syncthreads();
    const int nact = *w.nact;
    const int ngroups = (nact + kBtcSlots - 1) / kBtcSlots;
    for (int nc = 0; nc < nchunks; ++nc) {
      const int c0 = nc * kT5NC, nc_cols = min(kT5NC, np - c0);
      for (int gi = 0; gi < ngroups; ++gi) {
        const int ga = gi * kBtcSlots, gb = min(nact, ga + kBtcSlots), gn = gb - ga;
        if (nc == 0 || ngroups > 1) {  // left operand of this group of blocks
          uint4* A4 = reinterpret_cast<uint4*>(w.A);
          for (int i = tid; i < gn * (kT5ABytes / 16); i += kT5M) A4[i] = make_uint4(0, 0, 0, 0);
          __syncthreads();
          if (valid)
            batch_walk(s, prow, t, [&](int r, uint32_t, int32_t, int) {
              if (r < 0) return;
              const int pos = w.slot_of[r >> 5];
              if (pos >= ga && pos < gb) w.A[(size_t)(pos - ga) * kT5ABytes + a_off(tid, r & 31)] = kF8PlusOne;
            });
          fence_async_smem();
          __syncthreads();
        }
        bool ok = true;
        if (tid == 0) {
          const uint32_t bytes = (uint32_t)nc_cols * kT5K;
          bar_expect_tx(bar_b, bytes * (uint32_t)gn);
          for (int k = 0; k < gn; ++k)
            bulk_g2s(saddr(w.B + (size_t)k * kT5ABytes), bs->MB + ((size_t)w.act[ga + k] * np + c0) * kT5K, bytes,
                     bar_b);
          ok = bar_wait(bar_b, ph_b);
          ph_b ^= 1u;
          fence_after_sync();
          const uint32_t id = idesc_f8(kT5M, nc_cols);
          for (int k = 0; k < gn; ++k)
            mma_f8(tmem, smem_desc(saddr(w.A + (size_t)k * kT5ABytes), 128, 256),
                   smem_desc(saddr(w.B + (size_t)k * kT5ABytes), 128, 256), id, (gi > 0 || k > 0) ? 1u : 0u);
          mma_commit(bar_m);
        }
        ok = bar_wait(bar_m, ph_m) && ok;
        ph_m ^= 1u;
        fence_after_sync();
        if (__syncthreads_or(!ok)) {
          if (tid == 0) atomicOr(&a.st->error, kErrTimeout);
          return false;
        }
      }
      // C' = C_p + D for this chunk's columns, to staging row lid
      const uint32_t acc = tmem + ((uint32_t)(warp * 32) << 16);
      for (int c = 0; c < nc_cols; c += 32) {
        uint32_t r[32];
        const bool two = c + 32 <= nc_cols;
        if (nact == 0) {
#pragma unroll
          for (int i = 0; i < 32; ++i) r[i] = 0u;
        } else {
          if (two) tmem_ld32(acc + (uint32_t)c, r);
          else tmem_ld16(acc + (uint32_t)c, r);
          tmem_wait_ld();
        }
        const int j0 = c0 + c, cnt = min(two ? 32 : 16, m - j0);
        if (valid && !red) {
          int32_t* dst = a.staging + (size_t)lid * m + j0;
#pragma unroll
          for (int i = 0; i < 32; ++i)
            if (i < cnt) __stcg(dst + i, prow[j0 + i] + __float2int_rn(__uint_as_float(r[i])));
        }
      }
      fence_before_sync();
      __syncthreads();
      fence_after_sync();
    }
  }
  return true;
}

}  // namespace

__global__ void k_batch_init(BatchSys* sys, const int32_t* c0, const int64_t* c0_off, int32_t n) {
  const int lane = threadIdx.x & 31;
  const int64_t nw = (int64_t)gridDim.x * (blockDim.x >> 5);
  for (int64_t i = (int64_t)blockIdx.x * (blockDim.x >> 5) + (threadIdx.x >> 5); i < n; i += nw) {
    BatchSys& b = sys[i];
    const int m = b.sys.m;
    const int32_t* src = c0 + c0_off[i];
    for (int j = lane; j < m; j += 32) b.pool[j] = src[j];
    __syncwarp();
    const uint64_t h = fingerprint(b.sys, b.pool, lane);
    if (lane == 0) {
      const unsigned long long val = ((unsigned long long)fp32_of(h) << 32) | 0u;
      b.slots[(h & b.bmask) * kBucket] = val;  // the table is empty: first slot of its bucket
    }
  }
}

// Tensor-core form: one depth of every system, a system's whole depth by one
// CTA of four warps (the 128 TMEM lanes of a tile).
constexpr int kTcThreads = 128;
__global__ void __launch_bounds__(kTcThreads) k_batch_depth_tc(BatchArgs ba) {
  constexpr int kThreads = kTcThreads;
  extern __shared__ __align__(16) unsigned char smem_raw[];
  __shared__ unsigned int s_next;
  __shared__ uint64_t s_wsum[kThreads / 32];
  __shared__ unsigned int s_cnt, s_stop, s_capped, s_last, s_broken;
  const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5, nwarps = kThreads / 32;
  BatchScratch sc = batch_scratch(ba.scratch + (size_t)blockIdx.x * ba.scratch_stride, ba.pmax, ba.qc, ba.m_max);
  // tensor-core form: operands in shared memory, 128 TMEM columns, two mbarriers
  uint32_t ph_b = 0, ph_m = 0;
  BatchTcSmem tw = batch_tc_smem(smem_raw);
  if (tid == 0) {
    t5::bar_init(t5::saddr(tw.bars), 1);
    t5::bar_init(t5::saddr(tw.bars + 1), 1);
    asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
    s_broken = 0;
  }
  if (warp == 0) {
    asm volatile("tcgen05.alloc.cta_group::1.sync.aligned.shared::cta.b32 [%0], %1;" ::"r"(t5::saddr(tw.tmem_slot)),
                 "r"((uint32_t)t5::kT5NC));
    asm volatile("tcgen05.relinquish_alloc_permit.cta_group::1.sync.aligned;");
  }
  t5::fence_before_sync();
  __syncthreads();
  t5::fence_after_sync();
  const uint32_t tmem = *tw.tmem_slot;
  for (;;) {
    if (tid == 0) s_next = atomicAdd(ba.queue + ba.launch, 1u);
    __syncthreads();
    const int32_t si = (int32_t)s_next;
    __syncthreads();
    if (si >= ba.n) break;
    if (s_broken) break;
    BatchSys* bs = ba.sys + si;
    const int32_t d = bs->cur_depth + 1;
    if (bs->done || d > bs->target_depth) continue;
    BatchDepthStat* stat = bs->stats + d;
    const int64_t cap = bs->cap, budget = bs->budget;
    const int32_t max_expand = bs->max_expand;
    const DevSys S = bs->sys;
    const int m = S.m;
    const int64_t P = bs->level_hi - bs->level_lo;
    const int32_t* parents = bs->pool + (size_t)bs->level_lo * m;
    if (tid == 0) {
      ChunkState z = {};
      *sc.st = z;
    }
    // step (a) and Psi, one thread per parent
    bool over = false;
    for (int64_t p = tid; p < P; p += kThreads) {
      const int32_t* row = parents + (size_t)p * m;
      uint64_t prod = 1;
      bool skip = false, ov = false;
      for (int n = 0; n < m; ++n) {
        const int32_t x = row[n];
        const bool small = (uint32_t)x < (uint32_t)kDirect;
        const uint32_t cnt = __popc(small ? __ldg(S.dmask + (size_t)n * kDirect + x) : (uint32_t)appl(S, n, x));
        if (cnt > 1) prod = __umul64hi(prod, cnt) ? kSat : prod * cnt;
        if (!small || !S.gain_small) ov |= x > INT32_MAX - __ldg(S.gain + n);
        skip |= max_expand >= 0 && x > max_expand;
      }
      sc.off[p] = skip ? 0ull : prod;
      over |= ov && !skip;
    }
    if (tid == 0) sc.off[P] = 0;
    if (__any_sync(0xffffffffu, over) && lane == 0) atomicOr(&bs->error, kErrOverflow);
    __threadfence();
    __syncthreads();
    block_scan_sat(sc.off, P + 1, s_wsum);
    __threadfence();
    __syncthreads();
    const uint64_t total = sc.off[P];
    const uint64_t T = budget > 0 ? min(total, (uint64_t)budget) : total;
    uint64_t remaining = cap > 0 ? (uint64_t)cap : ~0ull;
    uint64_t g0 = 0, examined = 0;
    int64_t nnew = 0, n_rows = bs->n_rows;
    int32_t chunks = 0;
    bool capped = false;
    if (tid == 0) s_stop = bs->error ? 1u : 0u;
    __syncthreads();
    while (g0 < T && !capped && !s_stop) {
      const uint32_t Q = (uint32_t)min((uint64_t)ba.qc, T - g0);
      ClaimArgs a;
      a.sys = S;
      a.parents = parents;
      a.off = sc.off;
      a.P = P;
      a.g0 = g0;
      a.Q = Q;
      a.run = 0;
      a.table = DevTable{bs->slots, bs->bmask};
      a.pool = bs->pool;
      a.staging = sc.staging;
      a.gmin = sc.gmin;
      a.slot_of = sc.slot_of;
      a.ownbits = sc.own;
      a.prec = nullptr;
      a.ctr = nullptr;
      a.pperm = nullptr;
      a.store_ctr = nullptr;
      a.sidx_of = nullptr;
      a.store_cap = 0;
      a.st = sc.st;
      if (!batch_tc_rows(a, bs, tw, tmem, sc.hash, sc.red, ph_b, ph_m)) {
        if (tid == 0) {
          s_broken = 1;
          atomicOr(&bs->error, kErrTimeout);
        }
        __syncthreads();
        break;
      }
      __threadfence();
      __syncthreads();
      // step (d) for the pass's rows, 32 candidates per warp at a time
      for (uint32_t b0 = (uint32_t)warp * 32u; b0 < Q; b0 += (uint32_t)nwarps * 32u) {
        const uint32_t lid = b0 + (uint32_t)lane;
        const bool todo = lid < Q && !sc.red[lid];
        const uint64_t key = todo ? mix64(sc.hash[lid]) : 0ull;
        const int32_t* row = sc.staging + (size_t)(lid < Q ? lid : 0) * m;
        if ((m & 3) == 0)
          resolve_warp_body<RowI32V>(a, row, key, lid, todo);
        else
          resolve_warp_body<RowI32>(a, row, key, lid, todo);
      }
      __threadfence();
      __syncthreads();
      // first-occurrence marks
      const uint32_t nwords = (Q + 31) / 32;
      if (tid == 0) s_cnt = 0;
      __syncthreads();
      uint32_t cnt = 0;
      for (uint32_t wd = tid; wd < nwords; wd += kThreads) {
        uint32_t word = sc.own[wd];
        if (!word) continue;
        sc.own[wd] = 0;
        cnt += __popc(word);
        while (word) {
          const uint32_t o = wd * 32u + (uint32_t)(__ffs(word) - 1);
          word &= word - 1;
          const uint32_t f = o < Q ? sc.gmin[o] : 0xFFFFFFFFu;
          if (f >= Q) {  // not a claim of this pass: record and skip
            atomicOr(&sc.st->error, kErrInternal);
            continue;
          }
          atomicOr(sc.bits + (f >> 5), 1u << (f & 31));
          sc.srow[f] = o;
        }
      }
      if (cnt) atomicAdd(&s_cnt, cnt);
      __threadfence();
      __syncthreads();
      const uint32_t n_alloc = s_cnt;
      // ranks: exclusive scan of the words' popcounts
      uint64_t* ranks = sc.psi;
      for (uint32_t wd = tid; wd < nwords; wd += kThreads) ranks[wd] = __popc(__ldcg(sc.bits + wd));
      __syncthreads();
      block_scan_sat(ranks, nwords, s_wsum);
      __threadfence();
      __syncthreads();
      // commit: warp per word, lane per set bit
      const uint64_t accept = remaining;
      for (uint32_t wd = warp; wd < nwords; wd += nwarps) {
        const uint32_t word = __ldcg(sc.bits + wd);
        if (!((word >> lane) & 1u)) continue;
        const uint32_t lid = wd * 32u + (uint32_t)lane;
        const uint64_t rank = __ldcg(ranks + wd) + __popc(word & ((1u << lane) - 1u));
        const uint32_t o = __ldcg(sc.srow + lid);
        unsigned long long* slot = bs->slots + __ldcg(sc.slot_of + o);
        const unsigned long long hi = (*slot) & 0xFFFFFFFF00000000ull;
        if (rank < accept) {
          const int64_t row = n_rows + (int64_t)rank;
          const int32_t* src = sc.staging + (size_t)o * m;
          int32_t* dst = bs->pool + (size_t)row * m;
          copy_row_cg(src, dst, m);
          *slot = hi | (uint32_t)row;
          if (rank + 1 == accept) {
            sc.st->capped = 1;
            sc.st->last_lid = lid;
          }
        } else {
          *slot = hi | kRowTomb;
        }
      }
      __threadfence();
      __syncthreads();
      const uint64_t acc = min((uint64_t)n_alloc, accept);
      nnew += (int64_t)acc;
      n_rows += (int64_t)acc;
      if (remaining != ~0ull) remaining -= acc;
      if (tid == 0) {
        s_capped = sc.st->capped;
        s_last = sc.st->last_lid;
        if (sc.st->error) atomicOr(&bs->error, sc.st->error);
        s_stop = bs->error ? 1u : 0u;
      }
      for (uint32_t wd = tid; wd < nwords; wd += kThreads) sc.bits[wd] = 0;
      __threadfence();
      __syncthreads();
      capped = s_capped != 0;
      examined = capped ? g0 + s_last + 1 : g0 + Q;
      g0 += Q;
      ++chunks;
    }
    __syncthreads();
    if (tid == 0) {
      stat->new_configs = nnew;
      stat->examined = (int64_t)examined;
      stat->candidates = total;
      stat->truncated = examined < total ? 1 : 0;
      stat->chunks = chunks;
      bs->n_rows = n_rows;
      bs->cur_depth = d;
      if (nnew == 0) {
        bs->done = 1;
      } else {
        bs->depth_reached = d;
        bs->level_lo = bs->level_hi;
        bs->level_hi = n_rows;
      }
    }
    __syncthreads();
  }
  // products of a pass whose wait ran out may still be in flight
  if (s_broken && tid == 0) (void)t5::bar_wait(t5::saddr(tw.bars + 1), ph_m ^ 1u);
  t5::fence_before_sync();
  __syncthreads();
  if (warp == 0)
    asm volatile("tcgen05.dealloc.cta_group::1.sync.aligned.b32 %0, %1;" ::"r"(tmem), "r"((uint32_t)t5::kT5NC));
}

size_t batch_scratch_bytes(int64_t pmax, uint32_t qc, int m_max) {
  auto r = [](size_t b) { return (b + 255) & ~size_t(255); };
  return r((size_t)std::max<int64_t>(pmax + 1, qc / 32 + 1) * 8) + r((pmax + 1) * 8) + r((size_t)qc * m_max * 4) +
         3 * r(qc * 4) + 3 * r((qc / 32 + 1) * 4) +
         r(sizeof(ChunkState)) + r((size_t)qc * 8) + r(qc);
}

void launch_batch_depth_tc(const BatchArgs& a, int blocks, cudaStream_t st) {
  const size_t smem = batch_tc_smem_bytes() + 1024;
  cudaFuncSetAttribute(k_batch_depth_tc, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem);
  k_batch_depth_tc<<<blocks, kTcThreads, smem, st>>>(a);
}

}  // namespace snp
