// Kernels of the single-system BFS over SNP-system configurations.
//
// One depth (Algorithm 1, one round of steps II-IV) runs as:
//   k_psi      step (a) for every frontier configuration: applicable rules,
//              Psi = prod_n max(1, omega_n) (Eq. psi), saturating, and its
//              exclusive prefix sums, which give each parent's first candidate
//              (a lane per row, or a warp per row for small frontiers; after a
//              depth whose Psi sum saturated, the first 8192 rows go first and
//              the others are skipped when those hold 2^64 - 1 candidates);
//   per chunk of candidates [g0, g0 + Q) in canonical order:
//     k_expand steps (b)-(d) (snp_expand.cu; k_expand_wide for rows of more
//              than kWideM neurons): decode the spiking vector, C' = C + S . M_Pi
//              (Eq. next-config), fingerprint, look C' up; a key never seen is
//              claimed in the table and its row written (to the store, or to
//              staging row lid), and every candidate holding such a pending
//              key lowers that key's first-occurrence index;
//     k_mark   one bit per first occurrence;
//     k_commit ranks of the first occurrences in candidate order; the first
//              `remaining` of them get their discovery index, in rank order
//              (the row map entry; or a copy of the staged row into the
//              discovery-ordered pool), and their table slots point at their
//              rows; the rest become tombstones (the cap stops the depth).
#include <algorithm>
#include <type_traits>

#include "snp_kernels.cuh"

namespace snp {

namespace {

constexpr int kWarpsPerBlock = 4;

__device__ __forceinline__ void set_error(ChunkState* st, uint32_t bits) { atomicOr(&st->error, bits); }

}  // namespace

// Step (a), Eq. psi and its saturating exclusive scan for every frontier row:
// off[p] = the sum of Psi over rows before p, off[P] = the total; with REC the
// rows' ParentRecs.  Rows not to be expanded (max_expand) get Psi = 0, rows
// whose children could leave int32 raise kErrOverflow.  A CTA takes one run of
// a.sub consecutive tiles, a warp an eighth of them; runs are handed out in
// order, at most one per resident CTA, and chained by decoupled look-back at
// their ends (a hop per 32 runs; a chain over all tiles of 2^20 rows cost over
// 100 us).
//   WARP = false: tiles of 256 rows, a lane per row.  A warp moves its 32 rows
//     through shared memory 32 columns at a time (16-byte pieces where rows
//     are whole pieces, else one coalesced 128-byte load per row), unpacked to
//     int32; lane r then reads row r's slab at a stride of 33 words.
//   WARP = true: tiles of 8 rows, a warp per row, lane l visiting neurons
//     l, l + 32, ...: for small frontiers, so that a row of many neurons is not
//     one lane's serial walk (launch_psi has the rule).
// Both keep eight table lookups in flight per lane; what bounds them is those
// lookups' latency and the instructions per visit, not the rows' bytes.  With
// the scan in the same launch (it was a Psi launch, one to three scan launches,
// two clears and two copies per depth), the 3-neuron example to depth 10 went
// from 855 us to 601 us and 61 neurons with records from 2051 us to 1840 us.
template <class RF, bool REC, bool WARP>
__global__ void __launch_bounds__(256, REC ? 2 : 3) k_psi(PsiArgs a) {
  constexpr int R = WARP ? 8 : 256;
  __shared__ int32_t slabs[WARP ? 1 : 8][32][33];
  __shared__ uint64_t s_w[8];
  __shared__ uint64_t s_prefix;
  __shared__ uint32_t s_run;
  __shared__ int s_ok, s_last;
  const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
  const DevSys& s = a.s;
  const int m = s.m;
  int64_t P = a.P;
  uint32_t sub = a.sub;
  if (a.prev) {  // the frontier is what the depth before found, if it is complete
    P = __ldcg(&a.prev->go) && __ldcg(&a.prev->complete) ? (int64_t)__ldcg(a.ctr) - a.level_lo : 0;
    if (P > a.P) P = 0;  // more than the buffers hold: the host takes over
  }
  const uint32_t ntiles = (uint32_t)((P + R - 1) / R);
  if (a.prev) sub = max(1u, (ntiles + gridDim.x - 1) / gridDim.x);
  const uint64_t base = a.carry ? __ldcg(a.carry) : 0ull;
  if (a.off && base == kSat) {
    // these rows lie past the last candidate: Psi is not needed
    for (int64_t p = (int64_t)blockIdx.x * 256 + tid; p < P; p += (int64_t)gridDim.x * 256) a.off[p + 1] = kSat;
  } else {
    bool over = false;
    if (tid == 0) s_run = a.off ? atomicAdd(a.ticket, 1u) : blockIdx.x;
    __syncthreads();
    const uint32_t run = s_run, tile0 = run * sub, tile1 = min(tile0 + sub, ntiles);
    uint64_t through = 0;  // sum of the warp's rows so far
    // The run's rows: each warp takes a share of consecutive ones, so that the
    // warps meet only at the run's end (a barrier per tile cost a quarter).
    constexpr int W = R / 8;  // rows of a warp's step
    const int64_t wrow0 = (int64_t)tile0 * R + (int64_t)warp * sub * W;
    for (uint32_t j = 0; j < sub && tile0 < ntiles; ++j) {
      const int64_t p0 = wrow0 + (int64_t)j * W;  // this step's first row
      if (p0 >= P) break;
      PsiAcc acc;
      uint64_t v = 0;  // Psi of this lane's row (WARP: lane 0's)
      if (WARP) {
        if (p0 < P) {
          const typename RF::T* row = row_at<RF>(a.rows, a.perm ? __ldg(a.perm + p0) : (uint64_t)p0, m);
          ParentRec* rec = REC ? a.rec + p0 : nullptr;
          for (int n0 = 0; n0 < m; n0 += 32 * kPsiBatch) {
            int nn[kPsiBatch];
            int32_t x[kPsiBatch];
            uint32_t mask[kPsiBatch];
            uint64_t hx[kPsiBatch];
#pragma unroll
            for (int u = 0; u < kPsiBatch; ++u) {
              const int n = n0 + 32 * u + lane;  // past the row: neuron 0 without spikes, dropped below
              nn[u] = n < m ? n : 0;
              x[u] = n < m ? (int32_t)__ldcg(row + n) : 0;
            }
            acc.look_batch<REC>(s, nn, x, a.max_expand, mask, hx);
#pragma unroll
            for (int u = 0; u < kPsiBatch; ++u)
              if (n0 + 32 * u + lane >= m) {
                mask[u] = 0;
                hx[u] = 0;
              }
            acc.times(mask);
            if (REC) {
#pragma unroll
              for (int u = 0; u < kPsiBatch; ++u) {
                acc.hb += hx[u];
                const bool nt = __popc(mask[u]) > 1;
                const uint32_t b = __ballot_sync(0xffffffffu, nt);
                const uint32_t wide = __ballot_sync(0xffffffffu, nt && mask[u] >= 65536u);
                if (acc.nnt == kRecFull || wide || acc.nnt + __popc(b) > (uint32_t)kRecNt) {
                  if (b) acc.nnt = kRecFull;
                } else {
                  if (nt) rec->nt[acc.nnt + __popc(b & ((1u << lane) - 1u))] = ((uint32_t)nn[u] << 16) | mask[u];
                  acc.nnt += __popc(b);
                }
              }
            }
          }
          uint64_t prod = acc.prod;
#pragma unroll
          for (int o = 16; o > 0; o >>= 1) prod = sat_mul(prod, __shfl_xor_sync(0xffffffffu, prod, o));
          const bool skip = __any_sync(0xffffffffu, acc.skip);
          over |= __any_sync(0xffffffffu, acc.ov) && !skip;
          v = skip ? 0ull : prod;
          if (REC) {
            const uint64_t hb = warp_sum_u64(acc.hb);
            if (lane == 0) {
              rec->hbase = hb;
              rec->nnt = acc.nnt;
            }
          }
        }
      } else {
        int32_t(*slab)[33] = slabs[warp];
        const int nr = (int)max((int64_t)0, min((int64_t)32, P - p0));
        const uint64_t pr = lane < nr ? (a.perm ? __ldg(a.perm + p0 + lane) : (uint64_t)(p0 + lane)) : 0ull;
        ParentRec* rec = REC ? a.rec + p0 + lane : nullptr;
        for (int n0 = 0; n0 < m && nr > 0; n0 += 32) {
          const int w = min(32, m - n0);
          __syncwarp();
          // rows stream through L2 only, so that they do not evict the tables
          if constexpr (RF::VEC) {
            const int q4 = w / RF::PER16, total = nr * q4;
            for (int i0 = 0; i0 < total; i0 += 32) {
              const int i = i0 + lane, r = min(i / q4, nr - 1), q = i - r * q4;
              const uint64_t at = __shfl_sync(0xffffffffu, pr, r);
              if (i < total) {
                const uint4 y = __ldcg(reinterpret_cast<const uint4*>(row_at<RF>(a.rows, at, m) + n0) + q);
                int32_t x[RF::PER16];
                unpack_piece<RF>(y, x);
                int32_t* dst = &slab[r][RF::PER16 * q];
#pragma unroll
                for (int j = 0; j < RF::PER16; ++j) dst[j] = x[j];
              }
            }
          } else {
            for (int r0 = 0; r0 < nr; r0 += 16) {
              int32_t x[16];
#pragma unroll
              for (int u = 0; u < 16; ++u) {
                const uint64_t at = __shfl_sync(0xffffffffu, pr, (r0 + u) & 31);
                if (r0 + u < nr && lane < w) x[u] = __ldcg(row_at<RF>(a.rows, at, m) + n0 + lane);
              }
#pragma unroll
              for (int u = 0; u < 16; ++u)
                if (r0 + u < nr && lane < w) slab[r0 + u][lane] = x[u];
            }
          }
          __syncwarp();
          if (lane < nr) acc.visit_run<REC>(s, n0, slab[lane], w, a.max_expand, rec);
        }
        if (lane < nr) {
          v = acc.psi();
          over |= acc.overflow();
          if (REC) {
            rec->hbase = acc.hb;
            rec->nnt = acc.nnt;
          }
        }
      }
      if (!a.off) continue;
      // sums within the warp's share: exclusive ones to off, to be raised below
      if (WARP) {
        if (lane == 0) a.off[p0] = through;
        through = sat_add(through, v);
      } else {
        uint64_t inc = v;
#pragma unroll
        for (int o = 1; o < 32; o <<= 1) {
          const uint64_t y = __shfl_up_sync(0xffffffffu, inc, o);
          if (lane >= o) inc = sat_add(y, inc);
        }
        uint64_t before = __shfl_up_sync(0xffffffffu, inc, 1);
        if (lane == 0) before = 0;
        if (p0 + lane < P) a.off[p0 + lane] = sat_add(through, before);
        through = sat_add(through, __shfl_sync(0xffffffffu, inc, 31));
      }
    }
    if (a.off && tile0 < ntiles) {
      if (lane == 0) s_w[warp] = through;
      __syncthreads();
      uint64_t wbase = 0, all = 0;  // what the run's earlier warps hold; the run's sum
#pragma unroll
      for (int w = 0; w < 8; ++w) {
        if (w < warp) wbase = sat_add(wbase, s_w[w]);
        all = sat_add(all, s_w[w]);
      }
      if (warp == 0) {
        uint64_t prefix = 0;
        const bool ok = lookback_sat(a.tiles, run, a.epoch, base, all, prefix, lane);
        if (lane == 0) {
          s_prefix = prefix;
          s_ok = ok ? 1 : 0;
          if (!ok) atomicOr(&a.st->error, kErrTimeout);
        }
      }
      __syncthreads();
      if (s_ok) {
        const uint64_t prefix = sat_add(s_prefix, wbase);
        if (prefix != 0) {  // each lane raises what it wrote
          for (uint32_t j = 0; j < sub; ++j) {
            const int64_t p = wrow0 + (int64_t)j * W + (WARP ? 0 : lane);
            if (p < P && (!WARP || lane == 0)) a.off[p] = sat_add(prefix, a.off[p]);
          }
        }
        if (tile1 == ntiles && tid == 0) a.off[P] = sat_add(s_prefix, all);
      }
    }
    if (__any_sync(0xffffffffu, over) && lane == 0) set_error(a.st, kErrOverflow);
  }
  if (!a.off) return;
  __threadfence();
  __syncthreads();
  if (tid == 0) s_last = atomicAdd(a.ticket + 1, 1u) + 1 == gridDim.x ? 1 : 0;
  __syncthreads();
  if (!s_last || tid != 0) return;
  __threadfence();
  a.ticket[0] = 0;
  a.ticket[1] = 0;
  if (a.dyn) {
    DepthDyn y;
    y.P = P;
    y.total = P > 0 ? __ldcg(a.off + P) : 0ull;
    y.T = a.budget ? min(y.total, (uint64_t)a.budget) : y.total;
    y.Q = (uint32_t)min(y.T, (uint64_t)a.pass_max);
    y.go = P > 0 && y.T > 0 && __ldcg(&a.st->error) == 0 ? 1u : 0u;
    y.complete = 0;
    y.pad = 0;
    *a.dyn = y;
    if (P > 0) a.ctr[1] = a.remaining;
  }
  if (a.host_total) {  // the depth's candidates and errors to the host; the depth's counter starts
    if (a.ctr) a.ctr[1] = a.remaining;
    *a.host_total = __ldcg(a.off + P);
    a.host->error = __ldcg(&a.st->error);
    __threadfence_system();
  }
}

namespace {

template <class RF, bool REC>
void psi_launch(PsiArgs a, bool warp, cudaStream_t st, int nsm) {
  const int64_t tiles = (a.P + (warp ? 7 : 255)) / (warp ? 8 : 256);
  const int64_t resident = (int64_t)nsm * (REC ? 2 : 3);
  a.sub = (uint32_t)std::max<int64_t>(1, (tiles + resident - 1) / resident);
  const int blocks = (int)std::max<int64_t>(1, (tiles + a.sub - 1) / a.sub);
  if (warp)
    k_psi<RF, REC, true><<<blocks, 256, 0, st>>>(a);
  else
    k_psi<RF, REC, false><<<blocks, 256, 0, st>>>(a);
}

}  // namespace

// Tiles of 8 rows for small frontiers: a warp per row takes P / (16 nsm)
// rounds of a fixed latency and m / 32 visits, a lane per row m / 8 batches of
// lookups (in units of about 0.1 us: 12 + m / 32 a round, m).
static bool psi_by_warp(int64_t P, int m, int nsm) {
  const int64_t warps = 16 * nsm;
  return (P + warps - 1) / warps * (12 + m / 32) <= (P + 32 * warps - 1) / (32 * warps) * std::max(m, 16);
}

size_t psi_runs(int nsm) { return (size_t)nsm * 3; }

int launch_psi(PsiArgs a, int w, cudaStream_t st, int nsm) {
  const bool warp = psi_by_warp(a.expect > 0 ? a.expect : a.P, a.s.m, nsm);
  if (w == 1)
    a.rec ? psi_launch<RowU8, true>(a, warp, st, nsm) : psi_launch<RowU8, false>(a, warp, st, nsm);
  else if (w == 2)
    a.rec ? psi_launch<RowU16, true>(a, warp, st, nsm) : psi_launch<RowU16, false>(a, warp, st, nsm);
  else if (a.s.m % 4 == 0 && aligned16(a.rows))
    a.rec ? psi_launch<RowI32V, true>(a, warp, st, nsm) : psi_launch<RowI32V, false>(a, warp, st, nsm);
  else
    a.rec ? psi_launch<RowI32, true>(a, warp, st, nsm) : psi_launch<RowI32, false>(a, warp, st, nsm);
  return 1;
}

// One bit per first occurrence: every candidate lid that claimed a key
// (ownbits) names the key's first candidate gmin[lid]; clears ownbits and
// counts the first occurrences of each commit tile.  A warp takes four words, a
// lane per claim, so that the four words' gmin loads are in flight together (a
// thread per word walked its claims one after another: 8 us per pass of 2^16,
// 11 us per pass of 2^20).
__global__ void __launch_bounds__(256) k_mark(uint32_t* ownbits, const uint32_t* gmin, uint32_t* bits, uint32_t* srow,
                                              uint32_t nwords, uint32_t* counts, int tile_log, ChunkState* st,
                                              const DepthDyn* dyn) {
  constexpr int U = kMarkWords;
  if (dyn && !__ldcg(&dyn->go)) return;
  const int lane = threadIdx.x & 31;
  const uint32_t limit = nwords * 32u;
  const uint32_t nw = gridDim.x * (blockDim.x >> 5);
  for (uint32_t w0 = (blockIdx.x * (blockDim.x >> 5) + (threadIdx.x >> 5)) * U; w0 < nwords; w0 += nw * U) {
    uint32_t word[U], f[U];
#pragma unroll
    for (int u = 0; u < U; ++u) word[u] = w0 + u < nwords ? ownbits[w0 + u] : 0u;
    __syncwarp();
#pragma unroll
    for (int u = 0; u < U; ++u) {
      if (lane == 0 && word[u]) ownbits[w0 + u] = 0u;
      f[u] = (word[u] >> lane) & 1u ? gmin[(w0 + u) * 32u + lane] : 0u;
    }
#pragma unroll
    for (int u = 0; u < U; ++u) {
      bool ok = (word[u] >> lane) & 1u;
      if (ok && f[u] >= limit) {  // not a claim of this pass: record and skip
        atomicOr(&st->error, kErrInternal);
        ok = false;
      }
      if (ok) {
        atomicOr(bits + (f[u] >> 5), 1u << (f[u] & 31));
        srow[f[u]] = (w0 + u) * 32u + lane;
      }
      // one addition per tile the warp's claims fall into (mostly one)
      const uint32_t tile = ok ? f[u] >> tile_log : 0xFFFFFFFFu;
      const uint32_t same = __match_any_sync(0xffffffffu, tile);
      if (ok && lane == __ffs(same) - 1) atomicAdd(counts + tile, (uint32_t)__popc(same));
    }
  }
}

// Position of the n-th set bit (0-based; n < popc(v)).
__device__ __forceinline__ int nth_bit(uint32_t v, int n) {
  int pos = 0;
#pragma unroll
  for (int h = 16; h > 0; h >>= 1) {
    const int c = __popc(v & ((1u << h) - 1u));
    if (n >= c) {
      n -= c;
      v >>= h;
      pos += h;
    }
  }
  return pos;
}

// rows staged rows (row r: staging row s of lane r) to consecutive rows at dst,
// `per` elements each, by the whole warp with eight loads in flight.
template <typename T>
__device__ __forceinline__ void copy_staged(const T* staging, T* dst, uint32_t s, uint32_t rows, uint32_t per,
                                            int lane) {
  const uint32_t total = rows * per;
  for (uint32_t i0 = 0; i0 < total; i0 += 32 * 8) {
    T v[8];
#pragma unroll
    for (int u = 0; u < 8; ++u) {
      const uint32_t i = i0 + 32u * u + lane, q = min(i / per, 31u);
      const uint32_t src = __shfl_sync(0xffffffffu, s, (int)q);
      if (i < total) v[u] = __ldcg(staging + (size_t)src * per + (i - q * per));
    }
#pragma unroll
    for (int u = 0; u < 8; ++u)
      if (i0 + 32u * u + lane < total) dst[i0 + 32u * u + lane] = v[u];
  }
}

// One first occurrence of the given rank, candidate lid of the chunk: its row map
// entry, its slot (which keeps its fingerprint, the high half) and its parent
// record; or a tombstone past the cap.  p0, p1: parents that bound lid's.
// Returns the candidate that claimed the key.
__device__ __forceinline__ uint32_t commit_one(const CommitArgs& a, uint32_t lid, uint64_t rank, int64_t row_base,
                                               uint64_t remaining, int64_t p0, int64_t p1) {
  const uint32_t s = a.srow[lid];
  uint32_t* slot = reinterpret_cast<uint32_t*>(a.table.slots + a.slot_of[s]);
  if (rank >= remaining) {
    *slot = kRowTomb;
    return s;
  }
  const int64_t row = row_base + (int64_t)rank;
  const uint32_t at = a.perm ? a.sidx_of[s] : (uint32_t)row;
  if (a.perm) a.perm[row] = at;
  *slot = at;
  if (rank + 1 == remaining) {
    a.st->capped = 1;
    a.st->last_lid = lid;
  }
  if (a.rec_parent) {
    const uint64_t g = a.g0 + lid;
    int64_t lo = p0, hi = p1 + 1;  // largest p with off[p] <= g
    while (hi - lo > 1) {
      const int64_t mid = lo + (hi - lo) / 2;
      if (__ldg(a.off + mid) <= g) lo = mid; else hi = mid;
    }
    a.rec_parent[row] = a.parent_base + lo;
    a.rec_index[row] = g - __ldg(a.off + lo);
  }
  return s;
}

// The chunk is committed (one thread, after all others): the device counters
// move on, the chunk's counters go to the host and are cleared.
__device__ __forceinline__ void finish_chunk(const CommitArgs& a, uint32_t total, int64_t row_base,
                                             uint64_t remaining) {
  ChunkState c;
  c.n_alloc = total;
  c.error = __ldcg(&a.st->error);
  c.total_first = total;
  c.capped = __ldcg(&a.st->capped);
  c.last_lid = __ldcg(&a.st->last_lid);
  c.reserved = 0;
  c.p_first = __ldcg(&a.st->p_first);
  c.p_last = __ldcg(&a.st->p_last);
  if (a.ctr && !(a.dyn && !__ldcg(&a.dyn->go))) {
    const unsigned long long left = remaining;
    const unsigned long long acc = min((unsigned long long)total, left);
    a.ctr[0] = (unsigned long long)row_base + acc;
    if (left != ~0ull) a.ctr[1] = left - acc;
  }
  if (a.dyn) {
    DepthDyn y = *a.dyn;
    y.complete = y.go && !c.error && (c.capped || y.Q == y.T) ? 1u : 0u;
    a.dyn->complete = y.complete;
    a.host_depth->d = y;
    a.host_depth->cs = c;
    __threadfence_system();
    *a.st = ChunkState{};
  } else if (a.host) {
    *a.host = c;
    __threadfence_system();
    *a.st = ChunkState{};
  } else {
    *a.st = c;
  }
}

// Ranks the chunk's first occurrences in candidate order and commits them: the
// first `remaining` get their discovery index (store mode: perm[row] = the
// store row their owner wrote; else the staged row is copied to pool row
// row_base + rank) and their table slot pointed at it, the others become
// tombstones.  A CTA takes a tile of the bitmap; the marks counted every
// tile's first occurrences, so the CTA adds up the counts before its own (at
// most kCommitTiles of them) and deals its set bits out one per thread, 64
// words at a time.  The last CTA to finish advances the device counters,
// hands the chunk's counters to the host and clears them.  Bound by the
// latency of its dependent loads (owner, slot and store row).  (Ranks by
// decoupled look-back cost a hop of about 1 us per 32 tiles: 64 neurons, 18
// passes of about 2^20: 10.5 ms with 512 tiles a pass, 12.2 ms with 2048.)
constexpr int kCommitChunk = 64;  // bitmap words a CTA ranks at a time
__global__ void __launch_bounds__(256) k_commit(CommitArgs a, uint32_t tile_words) {
  __shared__ uint32_t s_word[kCommitChunk], s_pre[kCommitChunk];
  __shared__ uint32_t s_part[8], s_cnt, s_prefix;
  __shared__ int s_last;
  __shared__ int64_t s_p0, s_p1;
  const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
  const int64_t row_base = a.ctr ? (int64_t)__ldcg(a.ctr) : a.row_base;
  const uint64_t remaining = a.ctr ? __ldcg(a.ctr + 1) : a.remaining;
  const uint32_t tile = blockIdx.x, t0 = tile * tile_words, t1 = min(t0 + tile_words, a.nwords);
  const uint32_t mine = __ldcg(a.counts + tile);
  const int64_t P = a.dyn ? __ldcg(&a.dyn->P) : a.P;
  const uint32_t Q = a.dyn ? __ldcg(&a.dyn->Q) : a.Q;
  {  // first occurrences of the tiles before this one (the last CTA: of all)
    uint32_t sum = 0;
    for (uint32_t i = tid; i < tile; i += 256) sum += __ldcg(a.counts + i);
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) sum += __shfl_xor_sync(0xffffffffu, sum, o);
    if (lane == 0) s_part[warp] = sum;
  }
  if (warp == 1 && a.rec_parent && mine) {  // the parents of the tile's candidates
    const uint64_t gf = a.g0 + (uint64_t)t0 * 32u, gl = min(a.g0 + (uint64_t)t1 * 32u, a.g0 + Q) - 1;
    const int64_t p0 = warp_find_parent(a.off, P, gf, lane), p1 = warp_find_parent(a.off, P, gl, lane);
    if (lane == 0) {
      s_p0 = p0;
      s_p1 = p1;
    }
  }
  __syncthreads();
  uint32_t prefix = 0;
#pragma unroll
  for (int w = 0; w < 8; ++w) prefix += s_part[w];
  const uint32_t through = prefix + mine;  // the last tile's: all of the chunk's
  const int m = a.sys.m;
  for (uint32_t w0 = t0; mine && w0 < t1; w0 += kCommitChunk) {
    __syncthreads();
    if (warp == 0) {  // two words per lane
      const uint32_t i0 = w0 + 2u * lane, i1 = i0 + 1;
      const uint32_t x0 = i0 < t1 ? a.bits[i0] : 0u, x1 = i1 < t1 ? a.bits[i1] : 0u;
      if (x0) a.bits[i0] = 0u;  // clear for the next chunk
      if (x1) a.bits[i1] = 0u;
      const uint32_t c0 = __popc(x0), c1 = __popc(x1);
      uint32_t inc = c0 + c1;
#pragma unroll
      for (int o = 1; o < 32; o <<= 1) {
        const uint32_t y = __shfl_up_sync(0xffffffffu, inc, o);
        if (lane >= o) inc += y;
      }
      s_word[2 * lane] = x0;
      s_word[2 * lane + 1] = x1;
      s_pre[2 * lane] = inc - c0 - c1;
      s_pre[2 * lane + 1] = inc - c1;
      if (lane == 31) s_cnt = inc;
    }
    __syncthreads();
    const uint32_t cnt = s_cnt;
    for (uint32_t r0 = (uint32_t)warp * 32u; r0 < cnt; r0 += blockDim.x) {
      const uint32_t r = r0 + (uint32_t)lane;
      const uint64_t rank0 = (uint64_t)prefix + r0, rank = rank0 + lane;
      uint32_t s = 0;
      if (r < cnt) {
        int w = 0;  // the word holding rank r of the chunk
#pragma unroll
        for (int step = kCommitChunk / 2; step > 0; step >>= 1)
          if (s_pre[w + step] <= r) w += step;
        const uint32_t lid = (w0 + (uint32_t)w) * 32u + (uint32_t)nth_bit(s_word[w], (int)(r - s_pre[w]));
        s = commit_one(a, lid, rank, row_base, remaining, s_p0, s_p1);
      }
      if (!a.perm && rank0 < remaining) {  // staged rows to consecutive pool rows, by the whole warp
        const uint32_t rows = (uint32_t)min((uint64_t)min(cnt - r0, 32u), remaining - rank0);
        int32_t* dst = a.pool + (size_t)(row_base + (int64_t)rank0) * m;
        if ((m & 3) == 0 && (reinterpret_cast<uintptr_t>(a.pool) & 15) == 0)
          copy_staged(reinterpret_cast<const int4*>(a.staging), reinterpret_cast<int4*>(dst), s, rows, (uint32_t)m >> 2,
                      lane);
        else
          copy_staged(a.staging, dst, s, rows, (uint32_t)m, lane);
      }
    }
    prefix += cnt;
  }
  __threadfence();
  __syncthreads();
  if (tid == 0) {
    if (tile + 1 == gridDim.x) a.ticket[1] = through;
    __threadfence();
    s_last = atomicAdd(a.ticket, 1u) + 1 == gridDim.x ? 1 : 0;
  }
  __syncthreads();
  if (!s_last) return;
  for (uint32_t i = tid; i < gridDim.x; i += 256) a.counts[i] = 0u;
  if (tid != 0) return;
  __threadfence();
  const uint32_t total = __ldcg(a.ticket + 1);
  a.ticket[0] = 0;
  finish_chunk(a, total, row_base, remaining);
}

// Bitmap words per commit tile, as a power of two: 8 (256 candidates, so that a
// pass of 2^16 is 256 CTAs), more when that would make over kCommitTiles tiles.
static int commit_words_log(uint32_t nwords) {
  int lg = 3;
  while (((uint64_t)nwords + (1ull << lg) - 1) >> lg > kCommitTiles) ++lg;
  return lg;
}

// Marks, ranks and commit of a small chunk (at most kSmallWords bitmap words,
// store mode) by one CTA, the bitmap in shared memory: one launch in place of
// two where the launches are most of the time (3 neurons to depth 10: 525 us with
// up to 2048 candidates, 460 with 4096, 8192 or 16384; 20, 64, 128 and 300 neurons
// with caps of 1000 to 2500: within 2% for any of these limits; a pass of 6107
// candidates by one CTA made 919 neurons 3% slower).
constexpr uint32_t kSmallWords = 128;
__global__ void __launch_bounds__(1024) k_commit_small(CommitArgs a, uint32_t* ownbits, const uint32_t* gmin,
                                                       uint32_t* srow) {
  __shared__ uint32_t s_word[kSmallWords], s_pre[kSmallWords];
  __shared__ uint32_t s_sum[kSmallWords / 32];
  __shared__ int64_t s_p0, s_p1;
  const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
  const int64_t row_base = (int64_t)__ldcg(a.ctr);
  const uint64_t remaining = __ldcg(a.ctr + 1);
  const bool run = !a.dyn || __ldcg(&a.dyn->go);
  uint32_t cnt = 0;
  if (run) {
    const uint32_t limit = a.nwords * 32u;
    if (tid < (int)kSmallWords) s_word[tid] = 0u;
    __syncthreads();
    for (uint32_t w = warp; w < a.nwords; w += 32) {
      const uint32_t word = ownbits[w];
      __syncwarp();
      if (!word) continue;
      if (lane == 0) ownbits[w] = 0u;
      if ((word >> lane) & 1u) {
        const uint32_t f = gmin[w * 32u + lane];
        if (f >= limit) {  // not a claim of this pass: record and skip
          atomicOr(&a.st->error, kErrInternal);
        } else {
          atomicOr(s_word + (f >> 5), 1u << (f & 31));
          srow[f] = w * 32u + lane;
        }
      }
    }
    if (warp == 31 && a.rec_parent) {  // the parents of the chunk's candidates
      const int64_t P = a.dyn ? __ldcg(&a.dyn->P) : a.P;
      const uint32_t Q = a.dyn ? __ldcg(&a.dyn->Q) : a.Q;
      const int64_t p0 = warp_find_parent(a.off, P, a.g0, lane), p1 = warp_find_parent(a.off, P, a.g0 + Q - 1, lane);
      if (lane == 0) {
        s_p0 = p0;
        s_p1 = p1;
      }
    }
    __syncthreads();
    uint32_t inc = 0, own = 0;
    if (tid < (int)kSmallWords) {
      own = inc = __popc(s_word[tid]);
#pragma unroll
      for (int o = 1; o < 32; o <<= 1) {
        const uint32_t y = __shfl_up_sync(0xffffffffu, inc, o);
        if (lane >= o) inc += y;
      }
      if (lane == 31) s_sum[warp] = inc;
    }
    __syncthreads();
    uint32_t before = 0;
#pragma unroll
    for (int w = 0; w < (int)kSmallWords / 32; ++w) {
      if (w < warp) before += s_sum[w];
      cnt += s_sum[w];
    }
    if (tid < (int)kSmallWords) s_pre[tid] = before + inc - own;
    __syncthreads();
    for (uint32_t r = tid; r < cnt; r += 1024) {
      int w = 0;  // the word holding rank r
#pragma unroll
      for (int step = kSmallWords / 2; step > 0; step >>= 1)
        if (s_pre[w + step] <= r) w += step;
      commit_one(a, (uint32_t)w * 32u + (uint32_t)nth_bit(s_word[w], (int)(r - s_pre[w])), r, row_base, remaining, s_p0,
                 s_p1);
    }
    __threadfence();
    __syncthreads();
  }
  if (tid == 0) finish_chunk(a, cnt, row_base, remaining);
}

int launch_mark_commit(const CommitArgs& c, uint32_t* ownbits, const uint32_t* gmin, cudaStream_t st, int nsm) {
  if (c.nwords <= kSmallWords && c.perm && c.ctr) {
    k_commit_small<<<1, 1024, 0, st>>>(c, ownbits, gmin, const_cast<uint32_t*>(c.srow));
    return 1;
  }
  const uint32_t per = 8 * kMarkWords;
  const int blocks = (int)std::min<uint32_t>((c.nwords + per - 1) / per, (uint32_t)nsm * 16);
  const int lg = commit_words_log(c.nwords);
  k_mark<<<blocks, 256, 0, st>>>(ownbits, gmin, c.bits, const_cast<uint32_t*>(c.srow), c.nwords, c.counts, lg + 5, c.st, c.dyn);
  k_commit<<<(c.nwords + (1u << lg) - 1) >> lg, 256, 0, st>>>(c, 1u << lg);
  return 2;
}

__global__ void k_iota_u32(uint32_t* out, int64_t n) {
  for (int64_t k = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; k < n; k += (int64_t)gridDim.x * blockDim.x)
    out[k] = (uint32_t)k;
}

void launch_iota_u32(uint32_t* out, int64_t n, cudaStream_t st) {
  const int blocks = (int)std::max<int64_t>(1, std::min<int64_t>((n + 255) / 256, 152 * 32));
  k_iota_u32<<<blocks, 256, 0, st>>>(out, n);
}

// out[k] = pool[perm[k]] (pool[k] without perm) for k < n as int32 rows.  A
// warp takes 8 rows and moves them as one run of 16-byte pieces of the output
// (4-byte ones where m is no multiple of four), eight loads in flight; packed
// rows are widened four counts at a time.  For rows of up to kGatherPieces
// pieces: with a warp per row, 2^23 rows of 64 counts (4.1 GB moved) took
// 1084 us, half of every warp idle.
constexpr uint32_t kGatherPieces = 96;
template <class RF>
__global__ void __launch_bounds__(256) k_gather_short(const int32_t* pool, const uint32_t* perm, int64_t n, int m,
                                                     int32_t* out) {
  constexpr int kRows = 8, U = 8;
  const int lane = threadIdx.x & 31;
  const int64_t nw = (int64_t)gridDim.x * (blockDim.x >> 5);
  const uint32_t per = RF::VEC ? (uint32_t)m >> 2 : (uint32_t)m;  // pieces per row
  for (int64_t k0 = ((int64_t)blockIdx.x * (blockDim.x >> 5) + (threadIdx.x >> 5)) * kRows; k0 < n; k0 += nw * kRows) {
    const uint32_t rows = (uint32_t)min((int64_t)kRows, n - k0), total = rows * per;
    const uint32_t mine = lane < (int)rows ? (perm ? __ldg(perm + k0 + lane) : (uint32_t)(k0 + lane)) : 0u;
    for (uint32_t i0 = 0; i0 < total; i0 += 32 * U) {
      if constexpr (RF::VEC) {
        using Piece = typename std::conditional<RF::W == 1, uint32_t, typename std::conditional<RF::W == 2, uint2, int4>::type>::type;
        Piece v[U];
#pragma unroll
        for (int u = 0; u < U; ++u) {
          const uint32_t i = i0 + 32u * u + lane, q = min(i / per, (uint32_t)kRows - 1);
          const uint32_t src = __shfl_sync(0xffffffffu, mine, (int)q);
          if (i < total) v[u] = __ldcs(reinterpret_cast<const Piece*>(row_at<RF>(pool, src, m)) + (i - q * per));
        }
        int4* d = reinterpret_cast<int4*>(out) + (size_t)k0 * per;
#pragma unroll
        for (int u = 0; u < U; ++u) {
          const uint32_t i = i0 + 32u * u + lane;
          if (i >= total) continue;
          if constexpr (RF::W == 1) __stcs(d + i, unpack4_u8(v[u]));
          else if constexpr (RF::W == 2) __stcs(d + i, unpack4_u16(v[u]));
          else __stcs(d + i, v[u]);
        }
      } else {
        int32_t v[U];
#pragma unroll
        for (int u = 0; u < U; ++u) {
          const uint32_t i = i0 + 32u * u + lane, q = min(i / per, (uint32_t)kRows - 1);
          const uint32_t src = __shfl_sync(0xffffffffu, mine, (int)q);
          if (i < total) v[u] = __ldcs(pool + (size_t)src * m + (i - q * per));
        }
#pragma unroll
        for (int u = 0; u < U; ++u) {
          const uint32_t i = i0 + 32u * u + lane;
          if (i < total) __stcs(out + (size_t)k0 * m + i, v[u]);
        }
      }
    }
  }
}

// The same with a warp per row, for longer rows (1024 counts: at the copy rate).
template <class RF>
__global__ void __launch_bounds__(256) k_gather_rows(const int32_t* pool, const uint32_t* perm, int64_t n, int m,
                                                     int32_t* out) {
  const int lane = threadIdx.x & 31;
  const int64_t nw = (int64_t)gridDim.x * (blockDim.x >> 5);
  for (int64_t k = (int64_t)blockIdx.x * (blockDim.x >> 5) + (threadIdx.x >> 5); k < n; k += nw) {
    const typename RF::T* src = row_at<RF>(pool, perm ? __ldg(perm + k) : (uint64_t)k, m);
    int32_t* dst = out + (size_t)k * m;
    if constexpr (RF::VEC) {
      int4* d4 = reinterpret_cast<int4*>(dst);
      for (int j = lane; j < (m >> 2); j += 32) {
        if constexpr (RF::W == 1)
          d4[j] = unpack4_u8(__ldg(reinterpret_cast<const uint32_t*>(src) + j));
        else if constexpr (RF::W == 2)
          d4[j] = unpack4_u16(__ldg(reinterpret_cast<const uint2*>(src) + j));
        else
          d4[j] = __ldg(reinterpret_cast<const int4*>(src) + j);
      }
    } else {
      for (int j = lane; j < m; j += 32) dst[j] = __ldg(src + j);
    }
  }
}

void launch_gather_rows(const int32_t* pool, int w, const uint32_t* perm, int64_t n, int m, int32_t* out,
                        cudaStream_t st) {
  // whole 16-byte pieces where the rows are that and the caller's buffer starts on such a boundary
  const bool vec = (m & 3) == 0 && aligned16(out);
  const uint32_t pieces = vec ? (uint32_t)m / 4 : (uint32_t)m;
  const int64_t per = pieces <= kGatherPieces ? 64 : 8;  // rows per CTA
  const int blocks = (int)std::max<int64_t>(1, std::min<int64_t>((n + per - 1) / per, 152 * 64));
  auto fn = pieces <= kGatherPieces
                ? (w == 1 ? k_gather_short<RowU8> : w == 2 ? k_gather_short<RowU16>
                   : vec ? k_gather_short<RowI32V> : k_gather_short<RowI32>)
                : (w == 1 ? k_gather_rows<RowU8> : w == 2 ? k_gather_rows<RowU16>
                   : vec ? k_gather_rows<RowI32V> : k_gather_rows<RowI32>);
  fn<<<blocks, 256, 0, st>>>(pool, perm, n, m, out);
}

// Testing hook: the slot holding store row `row` as being claimed.
__global__ void k_hold_slot_of_row(unsigned long long* slots, uint64_t n, uint32_t row) {
  for (uint64_t i = blockIdx.x * (uint64_t)blockDim.x + threadIdx.x; i < n; i += (uint64_t)gridDim.x * blockDim.x) {
    const unsigned long long v = slots[i];
    if (v != kEmpty && (uint32_t)v == row) slots[i] = (v & 0xFFFFFFFF00000000ull) | kRowReserved;
  }
}

// Inserts committed rows [r0, r1) (all distinct) into an empty or partly
// filled table: used for C0 and to rebuild the table when it grows.
template <class RF>
__global__ void __launch_bounds__(kWarpsPerBlock * 32) k_insert_rows(DevSys s, const int32_t* pool,
                                                                     const uint32_t* perm, int64_t r0, int64_t r1,
                                                                     DevTable t, ChunkState* st) {
  const int lane = threadIdx.x & 31, wib = threadIdx.x >> 5;
  const int64_t nw = (int64_t)gridDim.x * kWarpsPerBlock;
  for (int64_t r = r0 + (int64_t)blockIdx.x * kWarpsPerBlock + wib; r < r1; r += nw) {
    const uint32_t sr = perm ? __ldg(perm + r) : (uint32_t)r;  // the row's place in the pool (the store)
    const typename RF::T* row = row_at<RF>(pool, sr, s.m);
    const uint64_t h = fingerprint(s, row, lane);
    if (lane == 0) {
      const unsigned long long val = ((unsigned long long)fp32_of(h) << 32) | sr;
      uint64_t b = h & t.bmask;
      bool done = false;
      for (uint64_t probes = 0; probes <= t.bmask && !done; ++probes, b = (b + 1) & t.bmask) {
        for (int k = 0; k < kBucket; ++k)
          if (atomicCAS(t.slots + b * kBucket + k, kEmpty, val) == kEmpty) {
            done = true;
            break;
          }
      }
      if (!done) set_error(st, kErrTableFull);
    }
  }
}

// *out = max(*out, x[0 .. n)) (*out starts at 0; the counts are >= 0).
__global__ void k_count_max(const int32_t* x, int64_t n, int32_t* out) {
  int32_t v = 0;
  for (int64_t i = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; i < n; i += (int64_t)gridDim.x * blockDim.x)
    v = max(v, __ldg(x + i));
#pragma unroll
  for (int o = 16; o > 0; o >>= 1) v = max(v, __shfl_xor_sync(0xffffffffu, v, o));
  if ((threadIdx.x & 31) == 0) atomicMax(out, v);
}

void launch_count_max(const int32_t* x, int64_t n, int32_t* out, cudaStream_t st) {
  const int blocks = (int)std::max<int64_t>(1, std::min<int64_t>((n + 255) / 256, 152 * 16));
  k_count_max<<<blocks, 256, 0, st>>>(x, n, out);
}

// n int32 rows into rows of format RF (counts within its range), four counts
// per thread.
template <class RF>
__global__ void k_pack_rows(const int32_t* src, int64_t n4, int32_t* dst) {
  for (int64_t i = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; i < n4; i += (int64_t)gridDim.x * blockDim.x) {
    const int4 v = __ldg(reinterpret_cast<const int4*>(src) + i);
    if constexpr (RF::W == 1)
      reinterpret_cast<uint32_t*>(dst)[i] = pack4_u8(v);
    else
      reinterpret_cast<uint2*>(dst)[i] = pack4_u16(v);
  }
}

void launch_pack_rows(const int32_t* src, int64_t n, int m, int w, int32_t* dst, cudaStream_t st) {
  const int64_t n4 = n * (m / 4);
  const int blocks = (int)std::max<int64_t>(1, std::min<int64_t>((n4 + 255) / 256, 152 * 32));
  if (w == 1)
    k_pack_rows<RowU8><<<blocks, 256, 0, st>>>(src, n4, dst);
  else
    k_pack_rows<RowU16><<<blocks, 256, 0, st>>>(src, n4, dst);
}

void launch_insert_rows(DevSys s, const int32_t* pool, int w, const uint32_t* perm, int64_t r0, int64_t r1,
                        DevTable t, ChunkState* st, int blocks, cudaStream_t stream) {
  auto fn = w == 1 ? k_insert_rows<RowU8> : w == 2 ? k_insert_rows<RowU16> : k_insert_rows<RowI32>;
  fn<<<blocks, kWarpsPerBlock * 32, 0, stream>>>(s, pool, perm, r0, r1, t, st);
}

__global__ void k_fill_u64(unsigned long long* p, uint64_t n, unsigned long long v) {
  for (uint64_t i = (uint64_t)blockIdx.x * blockDim.x + threadIdx.x; i < n; i += (uint64_t)gridDim.x * blockDim.x)
    p[i] = v;
}

}  // namespace snp
