// The single-system expand kernels (device code in snp_expand.cuh), the wide
// mode's base-child cache, and the resolve step for rows already in memory.
#include <algorithm>

#include "snp_expand.cuh"

namespace snp {

namespace {

template <class RF>
__global__ void __launch_bounds__(1024) k_wide_base(ClaimArgs a) {
  extern __shared__ __align__(16) int32_t brow[];  // [m]
  __shared__ int64_t s_p0;
  __shared__ unsigned long long s_h;
  const DevSys& s = a.sys;
  const int m = s.m;
  if (a.dyn && !__ldcg(&a.dyn->go)) return;
  const int64_t P = a.dyn ? __ldcg(&a.dyn->P) : a.P;
  const uint32_t Q = a.dyn ? __ldcg(&a.dyn->Q) : a.Q;
  BaseSlot* hdr = reinterpret_cast<BaseSlot*>(a.bcache);
  int32_t* out = reinterpret_cast<int32_t*>(reinterpret_cast<unsigned char*>(a.bcache) + base_rows_offset()) +
                 (size_t)blockIdx.x * round4(m);
  if (threadIdx.x == 0) {
    int64_t lo = 0, hi = P;  // largest p with off[p] <= g0 (off is sorted, off[0] = 0)
    while (hi - lo > 1) {
      const int64_t mid = lo + (hi - lo) / 2;
      if (__ldg(a.off + mid) <= a.g0) lo = mid; else hi = mid;
    }
    s_p0 = lo;
    s_h = 0;
  }
  __syncthreads();
  const int64_t p = s_p0 + blockIdx.x;
  bool use = !(a.ctr && __ldcg(a.ctr + 1) == 0) && p < P;
  if (use) {
    const uint64_t lo = max(__ldg(a.off + p), a.g0), hi = min(__ldg(a.off + p + 1), a.g0 + Q);
    use = hi > lo && hi - lo >= kBaseMin;
  }
  if (!use) {
    if (threadIdx.x == 0) hdr[blockIdx.x].parent = -1;
    return;
  }
  const typename RF::T* prow = parent_row<RF>(a, p);
  for (int n = threadIdx.x; n < m; n += blockDim.x) brow[n] = (int32_t)prow[n];
  __syncthreads();
  uint64_t h = 0;
  for (int n = threadIdx.x; n < m; n += blockDim.x) {
    const int32_t x = (int32_t)prow[n];
    h += col_hash(s, n, x);
    const uint32_t mask = (uint32_t)appl(s, n, x);
    if (!mask) continue;
    const int r = __ldg(s.first_rule + n) + __ffs(mask) - 1;
    h += __ldg(s.rowkey + r);
    const int e0 = __ldg(&s.rule[r].w), e1 = __ldg(&s.rule[r + 1].w);
    for (int e = e0; e < e1; e += 8) {  // eight loads in flight before their adds
      int2 cv[8];
#pragma unroll
      for (int u = 0; u < 8; ++u) cv[u] = e + u < e1 ? __ldg(s.csr + e + u) : make_int2(-1, 0);
#pragma unroll
      for (int u = 0; u < 8; ++u)
        if (cv[u].x >= 0) atomicAdd(&brow[cv[u].x], cv[u].y);
    }
  }
  h = warp_sum_u64(h);
  if ((threadIdx.x & 31) == 0) atomicAdd(&s_h, (unsigned long long)h);
  __syncthreads();
  for (int n = threadIdx.x; n < m; n += blockDim.x) out[n] = brow[n];
  if (threadIdx.x == 0) {
    hdr[blockIdx.x].hash = s_h;
    hdr[blockIdx.x].parent = p;
  }
}

constexpr uint32_t kMinRun = 32, kMinRunWide = 16;  // least candidates of a task (launch_expand has the figures)

// DYN: a depth without the host (a.dyn).
template <class RF, bool DYN>
__global__ void __launch_bounds__(256, 2) k_expand(ClaimArgs a, int B, int ts) {
  extern __shared__ __align__(16) unsigned char smem_raw[];
  if (DYN && !__ldcg(&a.dyn->go)) return;
  if (a.ctr && __ldcg(a.ctr + 1) == 0) return;  // the depth is full: a chunk enqueued ahead has nothing to do
  const int lane = threadIdx.x & 31, wib = threadIdx.x >> 5, wpb = blockDim.x >> 5;
  ExpandSmem w = expand_smem(smem_raw + (size_t)wib * expand_warp_bytes(a.sys.m, B, ts), a.sys.m, B, ts);
  expand_warp<RF, 0, DYN>(a, B, ts, w, (uint64_t)blockIdx.x * wpb + wib, (uint64_t)gridDim.x * wpb, kMinRun, lane);
}

// The wide mode of k_expand (rows of more than kWideM neurons).  WARPS per CTA,
// one CTA per SM: 16 (128 registers each) where their shared memory fits, else
// kWideWarps.  The passes are latency-bound: 301 neurons, cap 2^18: 6874 us with
// 11 warps, 5510 us with 16.
template <class RF, int WARPS, bool DYN>
__global__ void __launch_bounds__(WARPS * 32, 1) k_expand_wide(ClaimArgs a) {
  extern __shared__ __align__(16) unsigned char smem_raw[];
  if (DYN && !__ldcg(&a.dyn->go)) return;
  if (a.ctr && __ldcg(a.ctr + 1) == 0) return;
  const int lane = threadIdx.x & 31, wib = threadIdx.x >> 5, wpb = blockDim.x >> 5;
  ExpandSmem w = expand_smem_wide(smem_raw + (size_t)wib * expand_wide_bytes(a.sys.m), a.sys.m);
  expand_warp<RF, kWide, DYN>(a, kWideB, 0, w, (uint64_t)blockIdx.x * wpb + wib, (uint64_t)gridDim.x * wpb, kMinRunWide,
                              lane);
}

// Step (d) for rows already built in global memory (the tensor-core forms):
// one lane per candidate, the same bounded wait-free passes as k_expand.  (A
// lane that copied its own row of 1024 counts to the store: 195 us per 65536
// candidates.)
template <class RF>
__global__ void __launch_bounds__(256) k_resolve_rows(ClaimArgs a, const int32_t* rows,
                                                      const unsigned long long* hash, const uint8_t* redundant) {
  const int m = a.sys.m;
  if (a.ctr && __ldcg(a.ctr + 1) == 0) return;
  for (uint64_t base = (uint64_t)blockIdx.x * blockDim.x; base < a.Q; base += (uint64_t)gridDim.x * blockDim.x) {
    const uint64_t lid = base + threadIdx.x;
    bool done = lid >= a.Q || redundant[lid];
    const uint64_t key = done ? 0ull : mix64(hash[lid]);
    uint64_t t0 = 0;
    for (int pass = 0;; ++pass) {
      unsigned long long* owned = nullptr;
      const int status = done ? kDone : resolve_lane<RF>(a, rows + lid * m, key, (uint32_t)lid, owned);
      if (a.inplace) {
        if (status == kOwner) finish_owner_inplace(a, key, (uint32_t)lid, owned, a.inplace_base + lid);
      } else {  // the owners take consecutive store rows; the whole warp copies each row
        const int lane = threadIdx.x & 31;
        const uint32_t ob = __ballot_sync(0xffffffffu, status == kOwner);
        if (ob) {
          unsigned long long first = 0;
          if (lane == 0) first = atomicAdd(a.store_ctr, (unsigned long long)__popc(ob));
          first = __shfl_sync(0xffffffffu, first, 0);
          for (uint32_t o = ob, k = 0; o; o &= o - 1, ++k) {
            const uint64_t src = __shfl_sync(0xffffffffu, lid, __ffs(o) - 1);
            if (first + k < a.store_cap) warp_store_row<RF>(rows + src * m, row_at<RF>(a.pool, first + k, m), m, lane);
          }
          __threadfence();
          __syncwarp();
          if (status == kOwner)
            finish_owner_inplace(a, key, (uint32_t)lid, owned, first + __popc(ob & ((1u << lane) - 1u)));
        }
      }
      done = done || status != kRetry;
      if (__all_sync(0xffffffffu, done)) break;
      if (wait_expired(pass, a.wait_ns, t0)) {
        if (!done) atomicOr(&a.st->error, kErrTimeout);
        break;
      }
      __nanosleep(32);
    }
  }
}

}  // namespace

void launch_resolve_rows(ClaimArgs a, const int32_t* rows, const unsigned long long* hash, const uint8_t* redundant,
                         cudaStream_t st, int nsm) {
  const int blocks = (int)std::max<uint64_t>(1, std::min<uint64_t>(((uint64_t)a.Q + 255) / 256, (uint64_t)nsm * 8));
  if (a.sys.m % 4 == 0)
    k_resolve_rows<RowI32V><<<blocks, 256, 0, st>>>(a, rows, hash, redundant);
  else
    k_resolve_rows<RowI32><<<blocks, 256, 0, st>>>(a, rows, hash, redundant);
}

size_t wide_base_bytes(int m) { return base_rows_offset() + (size_t)kBaseSlots * round4(m) * 4; }

int launch_expand(ClaimArgs a, cudaStream_t st, int nsm) {
  const int m = a.sys.m;
  // rows of whole 16-byte pieces on 16-byte boundaries (snp_explore_static's
  // rows lie in the caller's buffer, which may start off one)
  const bool vec = m % 4 == 0 && aligned16(a.parents) && aligned16(a.pool) && aligned16(a.staging);
  if (m > kWideM) {
    const size_t per_warp = expand_wide_bytes(m);
    const bool many = per_warp * kWideWarpsMany <= (226u << 10);
    const int wpb = many ? kWideWarpsMany : (int)std::max<size_t>(1, std::min<size_t>(kWideWarps, (226u << 10) / per_warp));
    const size_t smem = per_warp * wpb;
    // one task per warp: a task's first block costs a full decode (C + S . M
    // over every neuron), which wide rows make expensive; at least 16
    // candidates (919 neurons, passes of a few thousand: 1031 us per
    // exploration with 256 or more, 552 with 32, 498 with 16, 502 with 8)
    const uint64_t warps = (uint64_t)nsm * wpb;
    a.run = (uint32_t)std::max<uint64_t>(kMinRunWide, ((uint64_t)a.Q + warps - 1) / warps);
    const uint64_t ntasks = ((uint64_t)a.Q + a.run - 1) / a.run;
    const int blocks = (int)std::min<uint64_t>((ntasks + wpb - 1) / wpb, (uint64_t)nsm);
    if (a.bcache) {  // base children of the pass's largest parents
      const size_t bs = (size_t)round4(m) * 4;
      auto fb = a.w == 2 ? k_wide_base<RowU16> : a.w == 1 ? k_wide_base<RowU8>
                : vec ? k_wide_base<RowI32V> : k_wide_base<RowI32>;
      fb<<<kBaseSlots, std::min(1024, (m + 31) / 32 * 32), bs, st>>>(a);
    }
    constexpr int kM = kWideWarpsMany, kF = kWideWarps;
    auto pick = [&](auto rf) -> void (*)(ClaimArgs) {
      using RF = decltype(rf);
      if (a.dyn) return many ? k_expand_wide<RF, kM, true> : k_expand_wide<RF, kF, true>;
      return many ? k_expand_wide<RF, kM, false> : k_expand_wide<RF, kF, false>;
    };
    auto fn = a.w == 2 ? pick(RowU16()) : a.w == 1 ? pick(RowU8()) : vec ? pick(RowI32V()) : pick(RowI32());
    allow_smem(fn);
    fn<<<blocks > 0 ? blocks : 1, wpb * 32, smem, st>>>(a);
    return a.bcache ? 2 : 1;
  }
  const int ts = round4(m) + 4;  // tile row stride (words): 16-byte aligned, rotates banks
  const int B = (int)std::min<size_t>(32, std::max<size_t>(1, (32u << 10) / (4u * ts)));
  const size_t per_warp = expand_warp_bytes(m, B, ts);
  const int wpb = (int)std::max<size_t>(1, std::min<size_t>(8, (100u << 10) / per_warp));
  const size_t smem = per_warp * wpb;
  const int per_sm = (int)std::max<size_t>(1, (220u << 10) / smem);
  // a task (run of candidates) pays one decode of its first block: in small
  // passes every warp takes one task of at least 32 candidates (20 neurons,
  // passes of at most 2^16: 404 us per exploration with 256 or more, 308 with
  // 32); from 256 candidates per warp on, two tasks per warp (16 neurons,
  // passes of half a million: two tasks of 103 each run 9% slower)
  {
    const uint64_t warps = (uint64_t)nsm * per_sm * wpb, each = ((uint64_t)a.Q + warps - 1) / warps;
    a.run = (uint32_t)std::max<uint64_t>(kMinRun, each <= 256 ? each : std::max<uint64_t>(256, (each + 1) / 2));
  }
  const uint64_t ntasks = ((uint64_t)a.Q + a.run - 1) / a.run;
  const int blocks = (int)std::min<uint64_t>((ntasks + wpb - 1) / wpb, (uint64_t)nsm * per_sm);
  auto pick = [&](auto rf) -> void (*)(ClaimArgs, int, int) {
    using RF = decltype(rf);
    return a.dyn ? k_expand<RF, true> : k_expand<RF, false>;
  };
  auto fn = a.w == 2 ? pick(RowU16()) : a.w == 1 ? pick(RowU8()) : vec ? pick(RowI32V()) : pick(RowI32());
  allow_smem(fn);
  fn<<<blocks > 0 ? blocks : 1, wpb * 32, smem, st>>>(a, B, ts);
  return 1;
}

}  // namespace snp

