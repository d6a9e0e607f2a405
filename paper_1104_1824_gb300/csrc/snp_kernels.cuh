// Kernel entry points of the single-system BFS (declarations shared by the
// launch code in snp_api.cu and the definitions in snp_kernels.cu).
#pragma once

#include <cuda.h>

#include <vector>

#include "snp_device.cuh"

namespace snp {

// True for a 16-byte boundary: device buffers of the caller may start off one,
// and the kernels' vector forms must not be given such rows.
inline bool aligned16(const void* p) { return (reinterpret_cast<uintptr_t>(p) & 15) == 0; }

// Lets a kernel (without static shared memory) launch with as much dynamic
// shared memory as a block can have.  Always this much, whatever the launch at
// hand needs: the limit belongs to the function, handles are used from several
// threads, and one that a thread lowered to its own launch would refuse a
// larger launch of another.
template <class F>
inline void allow_smem(F fn) {
  cudaFuncSetAttribute(fn, cudaFuncAttributeMaxDynamicSharedMemorySize, 227 << 10);
}

// A depth that runs without the host: what its kernels need to know of the
// depth before it and of one another (device memory).
struct DepthDyn {
  int64_t P;                  // frontier rows; 0: the depth does not run (yet)
  uint64_t total, T;          // candidates, and those within the budget
  uint32_t Q;                 // candidates of its first pass
  uint32_t go;                // 1: the pass runs
  uint32_t complete;          // 1: the pass was all the depth needed
  uint32_t pad;
};
// The same for the host, with the pass's counters (pinned memory).
struct HostDepth {
  DepthDyn d;
  ChunkState cs;
};

struct ClaimArgs {
  DevSys sys;
  const int32_t* parents;     // frontier rows: parents + pperm[p] * m, or parents + p * m without pperm
  const uint32_t* pperm;      // [P] store rows of the frontier, or nullptr
  const uint64_t* off;        // [P + 1] exclusive prefix sums of Psi (saturating)
  int64_t P;
  uint64_t g0;                // first candidate of the chunk
  uint32_t Q;                 // candidates in the chunk
  uint32_t run;               // consecutive candidates per warp task
  DevTable table;
  int32_t* pool;              // committed configurations (store mode: every claimed row, in claim order)
  int32_t* staging;           // [Q x m] row lid = candidate lid's configuration if lid claimed a new key
  // Store mode (store_ctr set): an owner takes the next row of the store
  // (pool) instead of staging row lid, and records it in sidx_of[lid].
  unsigned long long* store_ctr;
  uint32_t* sidx_of;          // [Q]
  uint64_t store_cap;         // rows the store holds
  uint32_t* gmin;             // [Q] per claiming lid: smallest chunk-local candidate holding its key
  uint32_t* slot_of;          // [Q] per claiming lid: its table slot
  uint32_t* ownbits;          // [Q / 32 + 1] bit lid set iff candidate lid claimed a new key
  const ParentRec* prec;      // [P] parent summaries, or nullptr (decode from the rows)
  const unsigned long long* ctr;  // device counters {rows, still acceptable} or nullptr; none left: no work
  ChunkState* st;
  // Rows already in the store (the fp8 tensor-core form writes candidate
  // lid's row to store row inplace_base + lid): an owner publishes it there.
  int32_t inplace = 0;
  uint64_t inplace_base = 0;
  uint64_t wait_ns = 0;       // > 0: time limit of a wait for a slot being claimed
  // Bytes per spike count of the rows of parents, pool and staging: 4
  // (int32), or 2 / 1 in a packed store (uint16 / uint8; m a multiple of 8 /
  // 16).  The pointers keep their int32_t type in every case.
  int32_t w = 4;
  // Wide mode: base children of the pass's largest parents (wide_base_bytes;
  // filled by the launch before each pass), or nullptr.
  int32_t* bcache = nullptr;
  // A depth without the host: P and Q (at most this Q) come from here.
  const DepthDyn* dyn = nullptr;
};

// Wide mode: base children cached per pass (headers, then rows of round4(m)).
constexpr int kBaseSlots = 8;
size_t wide_base_bytes(int m);

struct CommitArgs {
  DevSys sys;
  uint32_t Q;                 // candidates in the chunk
  uint32_t nwords;            // ceil(Q / 32)
  uint32_t* bits;             // [nwords] first-occurrence bitmap over chunk-local indices; cleared on the way
  // Counters that start (and are left) at 0: first occurrences of each commit
  // tile (kCommitTiles), and two words (tiles done; all first occurrences).
  uint32_t* counts;
  uint32_t* ticket;
  const uint32_t* srow;       // [Q] owner (candidate that claimed the key) of each first occurrence
  const uint32_t* slot_of;
  const int32_t* staging;
  DevTable table;
  int32_t* pool;
  // Store mode (perm set): rows stay where their owners stored them;
  // perm[row] = sidx_of[owner] records the store row of discovery index row.
  uint32_t* perm;
  const uint32_t* sidx_of;
  int64_t row_base;           // pool row of rank 0
  uint64_t remaining;         // how many more configurations the depth may accept
  unsigned long long* ctr;    // or, when set, both from device counters {rows, still acceptable}, advanced at the end
  // parent records (optional)
  int64_t* rec_parent;        // [rows] or nullptr
  uint64_t* rec_index;
  const uint64_t* off;
  int64_t P;
  int64_t parent_base;        // discovery index of frontier row 0
  uint64_t g0;
  ChunkState* st;             // the chunk's counters; with host, copied there and cleared at the end
  ChunkState* host;           // pinned host copy, or nullptr
  // A depth without the host: P and Q (at most this Q) come from dyn, whose
  // `complete` is set at the end; dyn and the counters go to host_depth.
  DepthDyn* dyn;
  HostDepth* host_depth;
};
constexpr int kMarkWords = 4;     // bitmap words per warp of the mark kernel
constexpr uint32_t kCommitTiles = 2048;  // most commit tiles of a chunk
// First-occurrence marks of the chunk (ownbits cleared on the way), ranks and
// commit; returns the launches made.
int launch_mark_commit(const CommitArgs& c, uint32_t* ownbits, const uint32_t* gmin, cudaStream_t st, int nsm);

// ---------------------------------------------------------------------------
// Batch engine and serving loop: many independent systems advance together.

// What a system of the sparse form does next (snp_many.cu).
constexpr int32_t kPhaseIdle = 0, kPhasePsi = 1, kPhaseExpand = 2;

// One system of a batch (device memory; updated by the batch kernels).
struct BatchSys {
  DevSys sys;
  int32_t* pool;               // configurations, discovery order, pool_rows rows
  unsigned long long* slots;   // the system's own hash table
  uint64_t bmask;              // buckets - 1
  int64_t pool_rows;
  int64_t level_lo, level_hi;  // current frontier: pool rows [level_lo, level_hi)
  int64_t n_rows;
  int32_t done;                // a depth found nothing new: the system is finished
  uint32_t error;              // kErr* bits
  int32_t depth_reached;
  int32_t cur_depth;           // depths completed so far
  int32_t target_depth;        // depths to run
  int32_t max_expand;
  int64_t cap, budget;         // per-depth frontier cap (>= 1) and candidate budget (<= 0: none)
  struct BatchDepthStat* stats;  // [target_depth + 1]
  // fp8 tensor-core form: M_Pi^T in e4m3 (tc5_pack_mt layout), columns rounded to 16, rule blocks
  const uint8_t* MB;
  int32_t np, nblocks;
  // Sparse form (snp_many.cu): the pass's arguments for the expand code (its
  // scratch among them), and where the depth stands.
  ClaimArgs a;
  uint64_t* off;               // [cap + 1] Psi, then its saturating exclusive scan
  ParentRec* rec;              // [cap]
  uint32_t* srow;              // [qc] owner of each first occurrence
  uint32_t* order;             // [qc] owners in rank order
  int32_t phase, tile;         // kPhase*; rows of the expand tile (narrow rows)
  uint32_t qc;                 // largest pass the scratch holds
  uint32_t overshoot;          // claims past the cap that the table has room for, per depth
  int32_t fixed_q;             // 1: passes of qc candidates whatever the cap still takes (the caller's pass size)
  int32_t chunks;
  uint32_t copy_n, copy_acc;   // first occurrences of the last pass; the accepted ones (ranks 0 .. copy_acc - 1)
  int64_t copy_row0;           // pool row of rank 0
  uint64_t total, T;           // candidates of the depth; those within the budget
  uint64_t remaining, examined, tombs;
  int64_t nnew;
  float rate;                  // first occurrences per candidate of the last pass
  int32_t few;                 // 1: the last depth had at most 256 candidates per parent (records pay)
};

// Work items {system, first element} of one iteration of the sparse form.
struct ManyQueue {
  int2* expand[2];             // runs of a.run candidates: this iteration's and the next one's; kMqForms regions of `cap`
  int2* copy;                  // kCopyRows first occurrences each
  int2* psi[2];                // 32 frontier rows each: without and with parent records
  uint32_t* ctr;               // counters, kMq*
  int64_t cap;                 // items of one region
};
// Systems by the form of the expand code they take (rows within or beyond
// kWideM neurons, of whole 16-byte units or not): items of one form together.
constexpr int kMqForms = 4;
enum { kMqExpand = 0, kMqHead = 2 * kMqForms, kMqCopy = 4 * kMqForms, kMqPsi, kMqActive = kMqPsi + 2, kMqCounters = 20 };

// Shape of the sparse form's expand launch.
struct ManyPlan {
  size_t warp_bytes = 0;       // shared memory per warp
  int warps = 8, ctas_per_sm = 2;
};
// Plan for systems of these neuron counts; tile, warps: the caller's settings
// (<= 0: automatic).  many_tile: rows of the expand tile for m neurons.
ManyPlan many_plan(const int32_t* ms, int64_t n, int tile, int warps);
int many_tile(const ManyPlan& p, int m, int tile);
// Candidates per pass for a frontier cap when the caller sets none.
uint32_t many_default_qc(int64_t cap);
// Scratch of one system: size, and its pointers (and pass arguments) in b,
// whose sys, pool, slots, bmask and cap are set.
size_t many_scratch_bytes(int64_t cap, uint32_t qc, int m);
void many_carve(BatchSys& b, unsigned char* base, uint32_t qc, uint32_t run);
// Work items a system can have queued at once (expand, copy or psi).
int64_t many_items(int64_t cap, uint32_t qc, uint32_t run);
// C0 into pool and table, scratch bitmaps cleared, first frontier queued:
// systems idx[i] (i without idx) for i < n.
void launch_many_init(BatchSys* sys, const int32_t* idx, const int32_t* c0, const int64_t* c0_off, int32_t n,
                      const ManyQueue& q, cudaStream_t st);
// One iteration over the systems [0, n): each finishes the Psi scan of a new
// frontier and at most one pass.  par alternates 0, 1.  Returns the launches made.
int launch_many_iteration(BatchSys* sys, int32_t n, const ManyQueue& q, int par, const ManyPlan& p, cudaStream_t st,
                          int nsm);

struct BatchDepthStat {
  int64_t new_configs;
  int64_t examined;
  uint64_t candidates;
  int32_t truncated;
  int32_t chunks;
};

// Tensor-core form: one launch advances every system by one depth (cur_depth
// + 1), unless it is finished or has run target_depth depths.
struct BatchArgs {
  BatchSys* sys;               // [n]
  int32_t n;
  int32_t launch;              // index of this launch (its work counter)
  uint32_t qc;                 // candidates per pass
  unsigned int* queue;         // work counters, one per launch, zero before it
  unsigned char* scratch;      // per-CTA scratch
  size_t scratch_stride;
  int64_t pmax;                // largest frontier a system may have (largest cap)
  int32_t m_max;
};

// Bytes of per-CTA scratch for frontiers of up to pmax rows and passes of qc candidates.
size_t batch_scratch_bytes(int64_t pmax, uint32_t qc, int m_max);
void launch_batch_depth_tc(const BatchArgs& a, int blocks, cudaStream_t st);
__global__ void k_batch_init(BatchSys* sys, const int32_t* c0, const int64_t* c0_off, int32_t n);

// Step (a), Psi and its scan for P frontier rows.
struct PsiArgs {
  DevSys s;
  const int32_t* rows;        // rows + perm[p] * m, or rows + p * m without perm (w bytes per count: launch_psi)
  const uint32_t* perm;
  int64_t P;
  int32_t max_expand;
  uint64_t* off;              // [P + 1], or nullptr: records only
  ParentRec* rec;             // [P] or nullptr
  // Look-back state: psi_runs() entries, two counters that start (and are
  // left) at 0, and a number no earlier launch on these entries had.
  ScanTile* tiles;
  uint32_t* ticket;
  uint32_t epoch;
  uint32_t sub;               // tiles per run (set by launch_psi)
  const uint64_t* carry;      // sum of Psi before these rows (nullptr: 0); when it is 2^64 - 1 the rows are not read
  ChunkState* st;             // errors
  // Set on the last launch of a depth: the total and st's errors to pinned
  // host memory; ctr (if any): ctr[1] = remaining.
  uint64_t* host_total;
  ChunkState* host;
  unsigned long long* ctr;
  unsigned long long remaining;
  // A depth without the host (dyn set): with prev, the frontier is what the
  // depth before it found, rows level_lo .. ctr[0] - 1, if that depth is
  // complete and they are at most P; dyn receives the frontier, its candidates
  // and the first pass (at most pass_max of the budget's candidates).
  DepthDyn* dyn;
  const DepthDyn* prev;
  int64_t level_lo;
  int64_t expect;             // frontier rows to choose the kernel by (0: P)
  unsigned long long budget;  // 0: none
  uint32_t pass_max;
};
size_t psi_runs(int nsm);
// rows: w bytes per spike count (4: int32; 2, 1: a packed store).  Returns the launches made.
int launch_psi(PsiArgs a, int w, cudaStream_t st, int nsm);
// Steps (b)-(d) for the chunk's candidates (k_expand); returns the launches made.
// Rows of more than kWideM neurons go through the kernel's wide mode (one
// scratch row per warp, rows built on demand).
constexpr int kWideM = 128;
int launch_expand(ClaimArgs a, cudaStream_t st, int nsm);
// Step (d) for candidate rows already in global memory (rows[lid * m], hash[lid]).
// Candidates with redundant[lid] set repeat an earlier candidate and are skipped.
void launch_resolve_rows(ClaimArgs a, const int32_t* rows, const unsigned long long* hash, const uint8_t* redundant,
                         cudaStream_t st, int nsm);
// Int8 tensor-core form of step (c) (snp_tc.cu).  nb = tc_blocks(R): words of a
// spiking vector's bits; M_Pi^T packed by tc_pack (tc_col_tiles(m) tiles).
int tc_blocks(int R);
int tc_col_tiles(int m);
std::vector<int8_t> tc_pack(const int32_t* M, int R, int m, int nb);
void launch_tc_masks(DevSys s, const int32_t* parents, const uint32_t* perm, const uint64_t* off, int64_t P,
                     uint64_t g0, uint32_t Q, uint32_t* bits, int nb, uint32_t* pidx, unsigned long long* hash,
                     uint8_t* redundant, ChunkState* st, cudaStream_t stream, int nsm);
void launch_tc_rows(DevSys s, const int32_t* parents, const uint32_t* bits, int nb, const uint32_t* pidx, uint32_t Q,
                    const int8_t* MF, int32_t* rows, cudaStream_t st);
// fp8 tensor-core form of step (c) on tcgen05 (snp_tc5.cu): candidate rows
// C' = C + S . M_Pi written to out[lid * m], their linear hashes and repeat flags.
struct Tc5Args {
  DevSys s;
  const int32_t* parents;     // the store (parents + pperm[p] * m) or frontier rows
  const uint32_t* pperm;
  const uint64_t* off;        // [P + 1] saturating exclusive scan of Psi
  int64_t P;
  uint64_t g0;
  uint32_t Q;
  const uint8_t* MB;          // M_Pi^T in e4m3, tc5_pack_mt layout
  int np;                     // columns rounded up to 16
  int nblocks;                // rule blocks: ceil(R / 32)
  int slots;                  // rule blocks held in shared memory at once (tc5_slots)
  int delta;                  // 1: delta form for tiles within one parent
  int32_t* out;               // [Q][m]: row lid = candidate lid's configuration (store row store_row0 + lid)
  uint64_t store_row0;        // store row of candidate 0 (the TMA store's row coordinate)
  int use_map;                // 1: rows go out through the tensor map given at launch
  unsigned long long* hash;   // [Q] linear hash h(C') of each candidate
  uint8_t* red;               // [Q] 1: repeats an earlier candidate of the same parent
  const unsigned long long* ctr;  // device counters {rows, still acceptable}: none left: no work
  ChunkState* st;
};
size_t tc5_smem_bytes(int m, int nblocks, int slots);
int tc5_slots(int m, int nblocks);
// Tensor map of the store (int32 [rows][m]) for the TMA row stores: 32 x 32
// boxes, 128-byte swizzle.  false: not available (m % 4 != 0, m < 32, or no
// driver entry point); rows are then stored by the threads.
bool tc5_store_map(CUtensorMap* map, int32_t* pool, int m, uint64_t rows);
void launch_tc5(const Tc5Args& a, const CUtensorMap& map, cudaStream_t st, int nsm);
void launch_iota_u32(uint32_t* out, int64_t n, cudaStream_t st);
// out[k] = row perm[k] (row k without perm) of a pool of w bytes per count, as
// int32.  w < 4: out on a 16-byte boundary.
void launch_gather_rows(const int32_t* pool, int w, const uint32_t* perm, int64_t n, int m, int32_t* out,
                        cudaStream_t st);
// Testing hook: marks the slot holding store row `row` as being claimed.
__global__ void k_hold_slot_of_row(unsigned long long* slots, uint64_t n, uint32_t row);
// *out = max(*out, x[0 .. n)) for counts x >= 0.
void launch_count_max(const int32_t* x, int64_t n, int32_t* out, cudaStream_t st);
// n int32 rows of m counts (m % 8 == 0, each count within the range of w
// bytes) into rows of w = 1 or 2 bytes per count at dst.
void launch_pack_rows(const int32_t* src, int64_t n, int m, int w, int32_t* dst, cudaStream_t st);
// Inserts rows [r0, r1) of a pool of w bytes per count into the table
// (blocks CTAs of kWarpsPerBlock warps).
void launch_insert_rows(DevSys s, const int32_t* pool, int w, const uint32_t* perm, int64_t r0, int64_t r1,
                        DevTable t, ChunkState* st, int blocks, cudaStream_t stream);
// All children of one configuration (snp_step.cu).  Plan of a step: Psi(C) and
// the multi-choice neurons, least significant first, as far as the first
// `capacity` children reach (each has two or more choices: at most 64).
constexpr int kStepList = 64;
struct StepPlan {
  unsigned long long psi;
  int32_t len;
  int32_t neuron[kStepList];
  uint32_t mask[kStepList];
};
// Reads C, turns base (C on entry) into the base child and fills *plan.
void launch_step_plan(DevSys s, const int32_t* C, int32_t* base, StepPlan* plan, cudaStream_t st);
// Children 0 .. min(Psi, capacity) - 1, canonical order, to out (no deduplication).
void launch_step_children(DevSys s, const int32_t* base, const StepPlan* plan, uint64_t capacity, int32_t* out,
                          cudaStream_t st, int nsm);
__global__ void k_fill_u64(unsigned long long* p, uint64_t n, unsigned long long v);

}  // namespace snp
