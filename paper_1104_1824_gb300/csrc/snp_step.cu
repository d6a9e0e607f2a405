// One transition step of one configuration (snp_step): every child C + S . M_Pi
// in canonical order (Eq. next-config for every valid spiking vector,
// Algorithm 2), without deduplication.
//
//   k_step_plan      Psi(C), the multi-choice neurons least significant first,
//                    and the base child (every firing neuron on its first
//                    applicable rule);
//   k_step_children  a warp walks a run of consecutive children in one row in
//                    shared memory: the first from the base child by swapping
//                    the neurons whose digit is not 0, each next one by the
//                    odometer (mostly one swap), and writes the row out.
//
// Bound by the rows written and, below that, by the latency of a swap.  The
// whole call for 2^15 children of 1024 neurons (134 MB) takes 74 us; with a
// child built from C and every firing neuron's row (26 k shared-memory atomics
// each) it took 4333 us.
#include <algorithm>

#include "snp_kernels.cuh"

namespace snp {

namespace {

constexpr int kPlanThreads = 256;
constexpr int kStepWarps = 8;  // per CTA

// Block 0: Psi and the list.  The other blocks: a warp per neuron adds its
// first applicable rule's row to base (atomics in L2; base holds C on entry).
// Bound by latency: 1024 neurons of 65 entries are 66 k additions, which one
// CTA's shared memory would take 20 us for.
__global__ void __launch_bounds__(kPlanThreads) k_step_plan(DevSys s, const int32_t* C, int32_t* base,
                                                            StepPlan* plan) {
  const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
  const int m = s.m;
  if (blockIdx.x > 0) {
    const int n = (blockIdx.x - 1) * (kPlanThreads / 32) + warp;
    if (n >= m) return;
    const uint32_t mask = (uint32_t)appl(s, n, __ldg(C + n));
    if (!mask) return;
    const int r = __ldg(s.first_rule + n) + __ffs(mask) - 1;
    const int e1 = __ldg(&s.rule[r + 1].w);
    for (int e = __ldg(&s.rule[r].w) + lane; e < e1; e += 32) {
      const int2 cv = __ldg(s.csr + e);
      atomicAdd(base + cv.x, cv.y);
    }
    return;
  }
  __shared__ uint32_t masks[1024];  // m <= 1024
  __shared__ uint64_t part[kPlanThreads / 32];
  uint64_t prod = 1;
  for (int n = tid; n < m; n += kPlanThreads) {
    const uint32_t mask = (uint32_t)appl(s, n, __ldg(C + n));
    masks[n] = mask;
    prod = sat_mul(prod, mask ? (uint64_t)__popc(mask) : 1ull);
  }
#pragma unroll
  for (int o = 16; o > 0; o >>= 1) prod = sat_mul(prod, __shfl_xor_sync(0xffffffffu, prod, o));
  if (lane == 0) part[warp] = prod;
  __syncthreads();
  if (warp != 0) return;
  int count = 0;
  for (int top = m - 1; top >= 0 && count < kStepList; top -= 32) {
    const int n = top - lane;
    const bool nt = n >= 0 && __popc(masks[n]) > 1;
    const uint32_t b = __ballot_sync(0xffffffffu, nt);
    const int at = count + __popc(b & ((1u << lane) - 1u));
    if (nt && at < kStepList) {
      plan->neuron[at] = n;
      plan->mask[at] = masks[n];
    }
    count += __popc(b);
  }
  if (lane == 0) {
    uint64_t psi = 1;
    for (int w = 0; w < kPlanThreads / 32; ++w) psi = sat_mul(psi, part[w]);
    plan->psi = psi;
    plan->len = min(count, kStepList);
  }
}

// VEC: rows of a multiple of four counts at a 16-byte aligned out.
template <bool VEC>
__global__ void __launch_bounds__(kStepWarps * 32) k_step_children(DevSys s, const int32_t* base,
                                                                   const StepPlan* plan, uint64_t capacity,
                                                                   int32_t* out) {
  extern __shared__ __align__(16) int32_t smem[];
  __shared__ uint8_t digs[kStepWarps][kStepList];
  const int lane = threadIdx.x & 31, wib = threadIdx.x >> 5;
  const int m = s.m;
  const uint64_t n = min((uint64_t)__ldg(&plan->psi), capacity);
  const uint64_t nw = (uint64_t)gridDim.x * kStepWarps;
  const uint64_t run = (n + nw - 1) / nw;
  const uint64_t t0 = ((uint64_t)blockIdx.x * kStepWarps + wib) * run;
  if (t0 >= n) return;
  const uint64_t t1 = min(n, t0 + run);
  const int len = __ldg(&plan->len);
  int32_t* row = smem + (size_t)wib * ((m + 3) & ~3);
  uint8_t* dig = digs[wib];
  for (int j = lane; j < m; j += 32) row[j] = __ldg(base + j);
  for (int i = lane; i < kStepList; i += 32) dig[i] = 0;
  __syncwarp();
  uint64_t q = t0;
  for (int i = 0; i < len && q != 0; ++i) {
    const uint32_t mask = __ldg(plan->mask + i);
    const int d = (int)next_digit(q, __popc(mask));
    if (d == 0) continue;
    const int r0 = __ldg(s.first_rule + __ldg(plan->neuron + i));
    warp_swap_rule(s, row, r0 + __ffs(mask) - 1, r0 + nth_set_bit(mask, d), lane);
    if (lane == 0) dig[i] = (uint8_t)d;
  }
  __syncwarp();
  for (uint64_t t = t0;;) {
    if constexpr (VEC) {
      const int4* a = reinterpret_cast<const int4*>(row);
      int4* b = reinterpret_cast<int4*>(out + t * m);
#pragma unroll 4
      for (int j = lane; j < (m >> 2); j += 32) __stcs(b + j, a[j]);
    } else {
      for (int j = lane; j < m; j += 32) __stcs(out + t * m + j, row[j]);
    }
    __syncwarp();
    if (++t >= t1) break;
    for (int i = 0; i < len; ++i) {  // the odometer, every lane following the same digits
      const uint32_t mask = __ldg(plan->mask + i);
      const int d = dig[i];
      const int nd = d + 1 == __popc(mask) ? 0 : d + 1;
      const int r0 = __ldg(s.first_rule + __ldg(plan->neuron + i));
      warp_swap_rule(s, row, r0 + nth_set_bit(mask, d), r0 + nth_set_bit(mask, nd), lane);
      if (lane == 0) dig[i] = (uint8_t)nd;
      if (nd != 0) break;
    }
    __syncwarp();
  }
}

}  // namespace

void launch_step_plan(DevSys s, const int32_t* C, int32_t* base, StepPlan* plan, cudaStream_t st) {
  const int per = kPlanThreads / 32;
  k_step_plan<<<1 + (s.m + per - 1) / per, kPlanThreads, 0, st>>>(s, C, base, plan);
}

void launch_step_children(DevSys s, const int32_t* base, const StepPlan* plan, uint64_t capacity, int32_t* out,
                          cudaStream_t st, int nsm) {
  // 32 warps per SM where there are that many children: at 1024 neurons a
  // child costs its 4 KB of stores and about one swap's round trip
  const uint64_t want = (capacity + kStepWarps - 1) / kStepWarps;
  const int blocks = (int)std::max<uint64_t>(1, std::min<uint64_t>(want, (uint64_t)nsm * 4));
  const size_t smem = (size_t)kStepWarps * ((s.m + 3) / 4 * 4) * sizeof(int32_t);
  if (s.m % 4 == 0 && (reinterpret_cast<uintptr_t>(out) & 15) == 0)
    k_step_children<true><<<blocks, kStepWarps * 32, smem, st>>>(s, base, plan, capacity, out);
  else
    k_step_children<false><<<blocks, kStepWarps * 32, smem, st>>>(s, base, plan, capacity, out);
}

}  // namespace snp
