// Exact int8 tensor-core form of step (c): C' = C + S . M_Pi (Eq. next-config)
// as a dense product of the chunk's spiking vectors S (0/1, int8, Q x R) with
// M_Pi (int8, R x m), accumulated in int32 by mma.sync m16n8k32 (the int8
// tensor-core instruction sm_103a accepts).  The product is exact: each row of
// S holds at most one 1 per neuron, so every output is a sum of at most m
// entries of M_Pi, each in [-127, 127], far inside int32.
//
// Per chunk:
//   k_tc_masks   a warp per run of candidates: parent, the spiking vector as one
//                bit per rule, its child's linear hash, whether it repeats an
//                earlier candidate;
//   k_tc_rows    128 candidates x 256 columns per CTA, 64 x 64 per warp;
//   then the rows are resolved against the hash table as in the sparse path.
#include <algorithm>

#include "snp_kernels.cuh"

namespace snp {

namespace {

constexpr int kTcWarps = 8;      // per CTA: 2 (candidates) x 4 (columns)
constexpr int kTcM = 64;         // candidates per warp
constexpr int kTcN = 64;         // columns per warp

__device__ __forceinline__ void mma_s8(int (&c)[4], uint32_t a0, uint32_t a1, uint32_t a2, uint32_t a3, uint32_t b0,
                                       uint32_t b1) {
  asm volatile(
      "mma.sync.aligned.m16n8k32.row.col.s32.s8.s8.s32 {%0,%1,%2,%3}, {%4,%5,%6,%7}, {%8,%9}, {%0,%1,%2,%3};"
      : "+r"(c[0]), "+r"(c[1]), "+r"(c[2]), "+r"(c[3])
      : "r"(a0), "r"(a1), "r"(a2), "r"(a3), "r"(b0), "r"(b1));
}

// Bits 4 i .. 4 i + 3 of w as four 0/1 bytes.
__device__ __forceinline__ uint32_t nibble_bytes(uint32_t w, int i) {
  return (((w >> (4 * i)) & 0xFu) * 0x00204081u) & 0x01010101u;
}

// Per-warp shared memory of k_tc_masks.
struct MaskSmem {
  uint32_t* msk;   // [m] applicable rules
  uint32_t* word;  // [nb] the spiking vector's bits
  uint16_t* ntl;   // [m] neurons with two or more applicable rules, least significant first
  uint8_t* dig;    // [m] digits over ntl
};
__host__ __device__ inline size_t mask_smem_bytes(int m, int nb) {
  return ((size_t)m * 7 + (size_t)nb * 4 + 15) / 16 * 16;
}

}  // namespace

// Step (b) for the chunk: per candidate the bits of its chosen rules
// (bits[lid * nb + r / 32], bit r % 32), its parent's store row (perm[p] when
// the frontier is reached through a row map, else p), linear hash and repeat
// flag.  A warp sets the first candidate of its run up from the parent and
// goes on by the odometer (a digit or two per candidate).  (Decoding every
// neuron of every candidate took 0.83 ms per 65536 candidates of 1024 neurons.)
__global__ void __launch_bounds__(256) k_tc_masks(DevSys s, const int32_t* parents, const uint32_t* perm,
                                                  const uint64_t* off, int64_t P, uint64_t g0, uint32_t Q,
                                                  uint32_t run, uint32_t* bits, int nb, uint32_t* pidx,
                                                  unsigned long long* hash, uint8_t* redundant, ChunkState* st) {
  extern __shared__ __align__(16) unsigned char tc_smem[];
  const int lane = threadIdx.x & 31, wib = threadIdx.x >> 5;
  const int m = s.m;
  MaskSmem w;
  w.msk = reinterpret_cast<uint32_t*>(tc_smem + (size_t)wib * mask_smem_bytes(m, nb));
  w.word = w.msk + m;
  w.ntl = reinterpret_cast<uint16_t*>(w.word + nb);
  w.dig = reinterpret_cast<uint8_t*>(w.ntl + m);
  const uint64_t la = ((uint64_t)blockIdx.x * (blockDim.x >> 5) + wib) * run;
  if (la >= Q) return;
  const uint64_t lb = min(la + run, (uint64_t)Q);
  int64_t p = warp_find_parent(off, P, g0 + la, lane);
  for (uint64_t l = la; l < lb; ++p) {
    const uint64_t p_lo = __ldg(off + p), p_hi = __ldg(off + p + 1);
    if (g0 + l >= p_hi) continue;  // a parent without candidates
    const uint32_t prow = perm ? __ldg(perm + p) : (uint32_t)p;
    const int32_t* row = parents + (size_t)prow * m;
    __syncwarp();
    for (int i = lane; i < nb; i += 32) w.word[i] = 0u;
    __syncwarp();
    // the base child: every firing neuron on its first applicable rule
    uint64_t h = 0;
    for (int n = lane; n < m; n += 32) {
      const int32_t x = __ldg(row + n);
      const uint32_t mask = appl_mask(s, n, x);
      w.msk[n] = mask;
      h += col_hash(s, n, x);
      if (!mask) continue;
      const int r = __ldg(s.first_rule + n) + __ffs(mask) - 1;
      atomicOr(w.word + (r >> 5), 1u << (r & 31));
      h += __ldg(s.rowkey + r);
    }
    h = warp_sum_u64(h);
    __syncwarp();
    int len = 0;
    for (int top = m - 1; top >= 0; top -= 32) {
      const int n = top - lane;
      const bool nt = n >= 0 && __popc(w.msk[n]) > 1;
      const uint32_t b = __ballot_sync(0xffffffffu, nt);
      const int at = len + __popc(b & ((1u << lane) - 1u));
      if (nt) {
        w.ntl[at] = (uint16_t)n;
        w.dig[at] = 0;
      }
      len += __popc(b);
    }
    __syncwarp();
    int red = 0;
    // neuron ntl[i] moves from digit d to nd (every lane follows; lane 0 writes)
    auto move = [&](int i, int d, int nd) {
      const int n = w.ntl[i];
      const uint32_t mask = w.msk[n];
      const int f = __ldg(s.first_rule + n);
      const int ro = f + nth_set_bit(mask, d), rn = f + nth_set_bit(mask, nd);
      h += __ldg(s.rowkey + rn) - __ldg(s.rowkey + ro);
      red += (redundant_choice(s, mask, rn) ? 1 : 0) - (redundant_choice(s, mask, ro) ? 1 : 0);
      if (lane == 0) {
        w.word[ro >> 5] &= ~(1u << (ro & 31));
        w.word[rn >> 5] |= 1u << (rn & 31);
        w.dig[i] = (uint8_t)nd;
      }
    };
    uint64_t q = g0 + l - p_lo;
#pragma unroll 1
    for (int i = 0; i < len && q != 0; ++i) {
      const int d = (int)next_digit(q, __popc(w.msk[w.ntl[i]]));
      if (d != 0) move(i, 0, d);
    }
    if (q != 0 && lane == 0) atomicOr(&st->error, kErrInternal);  // not an index of this parent
    for (;;) {
      __syncwarp();
      for (int i = lane; i < nb; i += 32) bits[l * nb + i] = w.word[i];
      if (lane == 0) {
        pidx[l] = prow;
        hash[l] = h;
        redundant[l] = red > 0 ? 1 : 0;
      }
      __syncwarp();
      ++l;
      if (l >= lb || g0 + l >= p_hi) break;
#pragma unroll 1
      for (int i = 0; i < len; ++i) {  // the odometer
        const int d = w.dig[i], nd = d + 1 == __popc(w.msk[w.ntl[i]]) ? 0 : d + 1;
        move(i, d, nd);
        if (nd != 0) break;
      }
    }
  }
}

// C' = C + S . M_Pi: 64 candidates x 64 columns per warp, no shared memory and
// no barriers.  The operands come as the instruction wants them: a lane's
// bytes of S are two nibbles of its candidates' rule bits, and M_Pi^T is laid
// out fragment by fragment at load (tc_pack), so that a warp's share of 8
// columns x 64 rules is one 16-byte load per lane (4 MB in all at 1024
// neurons: from L2).  Bound by the int8 tensor pipe (one mma.sync in about 66
// cycles per quarter of an SM); the version before it staged S byte by byte in
// shared memory and ran at 28% of that rate (11.5 ms per 65536 candidates of
// 1024 neurons).
//   MF: [col tiles of 8][nb / 2][32 lanes] 16 bytes.
__global__ void __launch_bounds__(kTcWarps * 32, 1) k_tc_rows(DevSys s, const int32_t* parents, const uint32_t* bits,
                                                              int nb, const uint32_t* pidx, uint32_t Q,
                                                              const uint4* MF, int32_t* rows) {
  const int m = s.m;
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
  const int g = lane >> 2, t4 = lane & 3;
  const uint32_t row0 = (blockIdx.x * 2u + (warp & 1)) * kTcM;
  const int col0 = ((int)blockIdx.y * 4 + (warp >> 1)) * kTcN;
  if (row0 >= Q || col0 >= m) return;
  int acc[4][8][4];
#pragma unroll
  for (int i = 0; i < 4; ++i)
#pragma unroll
    for (int j = 0; j < 8; ++j) acc[i][j][0] = acc[i][j][1] = acc[i][j][2] = acc[i][j][3] = 0;
  // rows of this lane: row0 + 16 i + g and + 8
  const uint32_t* bp[4][2];
#pragma unroll
  for (int i = 0; i < 4; ++i)
#pragma unroll
    for (int k = 0; k < 2; ++k) bp[i][k] = bits + (size_t)min(row0 + 16u * i + 8u * k + g, Q - 1) * nb;
  const uint4* mf = MF + (size_t)(col0 / 8) * (nb / 2) * 32 + lane;
  for (int k2 = 0; k2 < nb / 2; ++k2) {
    uint2 aw[4][2];
#pragma unroll
    for (int i = 0; i < 4; ++i)
#pragma unroll
      for (int k = 0; k < 2; ++k) aw[i][k] = __ldg(reinterpret_cast<const uint2*>(bp[i][k] + 2 * k2));
    uint4 b[8];
#pragma unroll
    for (int j = 0; j < 8; ++j) b[j] = __ldg(mf + ((size_t)j * (nb / 2) + k2) * 32);
#pragma unroll
    for (int ks = 0; ks < 2; ++ks) {
      uint32_t a[4][4];
#pragma unroll
      for (int i = 0; i < 4; ++i) {
        const uint32_t lo = ks ? aw[i][0].y : aw[i][0].x, hi = ks ? aw[i][1].y : aw[i][1].x;
        a[i][0] = nibble_bytes(lo, t4);
        a[i][1] = nibble_bytes(hi, t4);
        a[i][2] = nibble_bytes(lo, t4 + 4);
        a[i][3] = nibble_bytes(hi, t4 + 4);
      }
#pragma unroll
      for (int j = 0; j < 8; ++j)
#pragma unroll
        for (int i = 0; i < 4; ++i)
          mma_s8(acc[i][j], a[i][0], a[i][1], a[i][2], a[i][3], ks ? b[j].z : b[j].x, ks ? b[j].w : b[j].y);
    }
  }
#pragma unroll
  for (int i = 0; i < 4; ++i)
#pragma unroll
    for (int k = 0; k < 2; ++k) {
      const uint32_t r = row0 + 16u * i + 8u * k + g;
      if (r >= Q) continue;
      const int32_t* prow = parents + (size_t)__ldg(pidx + r) * m;
      int32_t* out = rows + (size_t)r * m;
#pragma unroll
      for (int j = 0; j < 8; ++j) {
        const int col = col0 + 8 * j + 2 * t4;
        const int v0 = acc[i][j][2 * k], v1 = acc[i][j][2 * k + 1];
        if ((m & 1) == 0 && col + 1 < m) {
          const int2 x = __ldg(reinterpret_cast<const int2*>(prow + col));
          __stcg(reinterpret_cast<int2*>(out + col), make_int2(x.x + v0, x.y + v1));
        } else {
          if (col < m) __stcg(out + col, __ldg(prow + col) + v0);
          if (col + 1 < m) __stcg(out + col + 1, __ldg(prow + col + 1) + v1);
        }
      }
    }
}

// Peak of mma.sync m16n8k32 s8 on this GPU: each warp issues `iters` rounds of
// 8 independent products; out receives a value that depends on every product.
__global__ void __launch_bounds__(128) k_tc_peak(int iters, int* out) {
  int acc[8][4];
#pragma unroll
  for (int k = 0; k < 8; ++k) acc[k][0] = acc[k][1] = acc[k][2] = acc[k][3] = 0;
  const uint32_t a = 0x01010101u * (threadIdx.x & 3), b = 0x01010101u;
  for (int it = 0; it < iters; ++it) {
#pragma unroll
    for (int k = 0; k < 8; ++k) mma_s8(acc[k], a, a + it, a, a, b, b + k);
  }
  int sum = 0;
#pragma unroll
  for (int k = 0; k < 8; ++k) sum += acc[k][0] + acc[k][1] + acc[k][2] + acc[k][3];
  out[blockIdx.x * blockDim.x + threadIdx.x] = sum;
}

// M_Pi^T in the order k_tc_rows reads it: for each tile of 8 columns and each
// pair of 32-rule blocks, 16 bytes per lane (column lane / 4; of each block the
// rules 4 (lane % 4) .. + 3 and 16 + 4 (lane % 4) .. + 3).
std::vector<int8_t> tc_pack(const int32_t* M, int R, int m, int nb) {
  const int tiles = tc_col_tiles(m);
  std::vector<int8_t> out((size_t)tiles * (nb / 2) * 32 * 16, 0);
  for (int r = 0; r < R; ++r) {
    const int blk = r >> 5, k = r & 31;
    const int t4 = (k & 15) >> 2, byte = (blk & 1) * 8 + (k >> 4) * 4 + (k & 3);
    for (int j = 0; j < m; ++j)
      out[(((size_t)(j >> 3) * (nb / 2) + (blk >> 1)) * 32 + (j & 7) * 4 + t4) * 16 + byte] = (int8_t)M[(size_t)r * m + j];
  }
  return out;
}

int tc_blocks(int R) { return ((R + 63) / 64) * 2; }

int tc_col_tiles(int m) { return (m + kTcN - 1) / kTcN * (kTcN / 8); }

void launch_tc_masks(DevSys s, const int32_t* parents, const uint32_t* perm, const uint64_t* off, int64_t P,
                     uint64_t g0, uint32_t Q, uint32_t* bits, int nb, uint32_t* pidx, unsigned long long* hash,
                     uint8_t* redundant, ChunkState* st, cudaStream_t stream, int nsm) {
  const size_t per = mask_smem_bytes(s.m, nb);
  int warps = 8;
  while (warps > 1 && per * warps > (200u << 10)) warps >>= 1;
  const size_t smem = per * warps;
  if (smem > (48u << 10)) allow_smem(k_tc_masks);
  const uint32_t run = std::max<uint32_t>(8, (uint32_t)(((uint64_t)Q + 16ull * nsm - 1) / (16ull * nsm)));
  const uint32_t tasks = (Q + run - 1) / run;
  k_tc_masks<<<(tasks + warps - 1) / warps, warps * 32, smem, stream>>>(s, parents, perm, off, P, g0, Q, run, bits, nb,
                                                                        pidx, hash, redundant, st);
}

void launch_tc_rows(DevSys s, const int32_t* parents, const uint32_t* bits, int nb, const uint32_t* pidx, uint32_t Q,
                    const int8_t* MF, int32_t* rows, cudaStream_t st) {
  const dim3 grid((Q + 2 * kTcM - 1) / (2 * kTcM), (s.m + 4 * kTcN - 1) / (4 * kTcN));
  k_tc_rows<<<grid, kTcWarps * 32, 0, st>>>(s, parents, bits, nb, pidx, Q, reinterpret_cast<const uint4*>(MF), rows);
}

}  // namespace snp

extern "C" int snp_tc_peak_tops(int32_t iters, double* tops) {
  if (!tops || iters < 1) return 1;
  int dev = 0, nsm = 0;
  if (cudaGetDevice(&dev) != cudaSuccess) return 4;
  cudaDeviceGetAttribute(&nsm, cudaDevAttrMultiProcessorCount, dev);
  const int blocks = nsm * 8, threads = 128;
  int* out = nullptr;
  if (cudaMalloc(&out, sizeof(int) * blocks * threads) != cudaSuccess) return 3;
  cudaEvent_t e0, e1;
  cudaEventCreate(&e0);
  cudaEventCreate(&e1);
  snp::k_tc_peak<<<blocks, threads>>>(iters / 10 + 1, out);  // warm-up
  cudaEventRecord(e0);
  snp::k_tc_peak<<<blocks, threads>>>(iters, out);
  cudaEventRecord(e1);
  cudaError_t err = cudaEventSynchronize(e1);
  float ms = 0.f;
  cudaEventElapsedTime(&ms, e0, e1);
  cudaEventDestroy(e0);
  cudaEventDestroy(e1);
  cudaFree(out);
  if (err != cudaSuccess) return 4;
  const double ops = 2.0 * 16 * 8 * 32 * 8.0 * iters * (double)blocks * (threads / 32);
  *tops = ops / (ms * 1e-3) / 1e12;
  return 0;
}
