// mcm_kernels.cuh -- launch-side declarations of the MCM kernels.
//
// Problem (paper Section IV-A, Eq. (2); recurrence from Cormen et al., which
// the paper cites): for i < j
//     m[i][j] = min_{i <= k < j} m[i][k] + m[k+1][j] + p[i] * p[k+1] * p[j+1]
// and s[i][j] = the smallest minimising k.  The interval-DP instances add a
// per-cell weight w[i][j] to every candidate of cell (i, j) (Eq. (2) with a
// more general f), which they do once, when the cell's minimum is final.
//
// GPU decomposition.  The n x n table is cut into 32 x 32 tiles (I, J), J >= I.
// Tile (I, J) lies on tile-diagonal D = J - I.  For a cell of tile (I, J) the
// splits k fall into
//   * external segments K = I+1 .. J-1 (k in [32K, 32K+32)): the row panel is
//     tile (I, K), the column panel rows 32K+1 .. 32K+32 of tile column J;
//     segment K becomes computable once tile-diagonal r(K) = max(K-I, J-K) is
//     complete, so most of a tile's work is ready long before its neighbours;
//   * the boundary split k = 32I + 31 (needs row 32(I+1) of tile (I+1, J));
//   * the in-tile splits k in [i, 32I+30] and [32J, j-1], which depend on the
//     tile's own cells and are resolved by a wavefront over the tile's
//     diagonals of 2x2 cells (the paper's diagonal computation order, Figs. 5-7,
//     applied inside one tile).
// Work items ("tasks") are (tile, range of r levels).  A bulk task reduces a
// group of external segments and merges its (value, k) minima into the tile's
// partial accumulator with 64-bit atomicMin (deterministic: the packed
// comparison is lexicographic on (value, k)).  The finisher task of a tile
// waits for those, reduces the last segments, adds the boundary split, runs
// the in-tile wavefront, writes the outputs and publishes the tile's flag.
// Tasks are popped from one queue in order of the tile-diagonal at which they
// become ready (finishers of diagonal D after every task they wait for), so a
// block only ever waits for tasks popped before its own: the queue makes
// progress whatever the number of resident blocks.
//
// Cost encodings (exact integer arithmetic throughout):
//   int32 costs: every candidate is at most (n-1)*max(p)^3 =: bound < 2^31
//     (interval DP: (n-1)*(max(p)^3 + max(w))).
//     The packed row-panel entry is (m << S) | (k mod 2^S) and the column
//     panel entry m << S, with S the largest value <= 5 such that
//     (bound + 1) << S <= 2^32.  Then  A + B + (p_i p_j1) (p_k1 << S)
//     = (candidate << S) | (k mod 2^S), so an unsigned min over a chunk of
//     2^min(S,5) aligned splits yields the minimum and its smallest k at once.
//   int64 costs (bound < 2^47): entries are (m << 16) | k and m << 16, so one
//     unsigned 64-bit min yields (value, smallest k) directly.
// The panels of a diagonal tile are read by in-tile solves only: int32, like
// those of any tile; int64, as the tables U and L of mcm_tile.cuh.
#pragma once

#include <cstdint>
#include <cuda_runtime.h>

namespace dpk {

constexpr int kTile = 32;
// the int32 main kernel's blocks
constexpr int kGroupThreads = 128;                     // one compute group
constexpr int kComputeThreads = 2 * kGroupThreads;     // two groups
constexpr int kMcmThreads = kComputeThreads + 32;      // + producer warp
constexpr int kStages = 2;                             // bulk-copy stages per group

// Work split of a tile on tile-diagonal D >= 2: its external levels
// r = (D+1)/2 .. D-1 go to bulk tasks of kLevelsPerPart levels each, except
// the last level, which the finisher keeps; a tile with fewer than
// kMinBulkLevels bulk levels is not split at all.
constexpr int kLevelsPerPart = 8;
constexpr int kMinBulkLevels = 2;
// A tile's bulk levels are cut from the top: the part that ends at the last
// bulk level D-2 -- the part the finisher is likeliest to wait for, since it
// becomes ready only when tile-diagonal D-2 is complete -- holds
// kLastPartLevels levels, and kLevelsPerPart-level parts cover the levels
// below it.
constexpr int kLastPartLevels = 4;
// Queue position of the other parts: not before they become ready, and not
// earlier than kDeferBuckets tile-diagonals before their finisher. Work that
// is not needed soon then waits behind the tasks of the chain in the middle
// diagonals (where blocks are scarce) and fills the blocks that the last
// diagonals leave idle.  int64 chains, against parts cut from the lowest level
// up and queued as they become ready: n = 1500 1006 -> 927 us, n = 2048 1457 ->
// 1264, n = 4096 6154 -> 5896; batches of 50 to 2000 uneven chains within 3 %.
constexpr int kDeferBuckets = 3;

struct McmInstDev {
  const int32_t* p;   // dims p[0..n] (set by the prologue)
  void* m;            // output cost table (set by the prologue)
  int16_t* s;         // output split table (set by the prologue)
  int32_t n;          // matrices
  int32_t nt;         // tiles per side
  int32_t shift;      // packing shift S (set by the prologue)
  int32_t pad_;
  int64_t tile_base;  // first index of this chain's tiles in the per-tile arrays
  int64_t pp_base;    // offset of this chain's padded dims in McmLaunchArgs::pp
  int64_t pk_base;    // offset of this chain's shifted dims in McmLaunchArgs::pk
  const void* w;      // interval DP: per-cell weight table, like m (set by the prologue)
  unsigned long long wmax;  // interval DP: largest weight above the diagonal (weight pass)
};

// kind 0: finisher of tile (I, J) for r levels [r_lo, r_hi], waits for
// `nparts` bulk tasks.  kind 1: bulk task for r levels [r_lo, r_hi].
struct McmTask {
  int32_t inst;
  int16_t I, J;
  int16_t r_lo, r_hi;
  int16_t kind, nparts;
};

// The tasks of a tile on tile-diagonal D: its finisher keeps the levels [lo,
// hi], its bulk parts (0 the last one, then downwards) cover the ones below.
struct McmSplit {
  int lo, hi, nparts, rmin;
};
__host__ __device__ inline McmSplit mcm_split(int D, int levels_per_part) {
  McmSplit t{1, 0, 0, 1};
  if (D < 2) return t;
  t.rmin = (D + 1) / 2;
  t.hi = D - 1;
  t.lo = t.hi - t.rmin < kMinBulkLevels ? t.rmin : t.hi;  // the last level: both neighbours
  const int bulk = t.lo - t.rmin;
  if (bulk > 0) t.nparts = 1 + (bulk > kLastPartLevels ? (bulk - kLastPartLevels + levels_per_part - 1) / levels_per_part : 0);
  return t;
}

// The queue is sorted into bins, 3 per tile-diagonal b: the finishers of
// diagonal b, the last parts of diagonal b + 1 and the other parts of diagonal
// b + kDeferBuckets.  A last part is ready when diagonal b is complete; the
// others were ready earlier, and wait behind the tasks of the chain.  So every
// task comes after every task it waits for.
__host__ __device__ inline int mcm_bin_finisher(int D) { return 3 * D; }
__host__ __device__ inline int mcm_bin_last(int D) { return 3 * (D - 1) + 1; }
__host__ __device__ inline int mcm_bin_other(int D) { return 3 * (D - kDeferBuckets) + 2; }
static_assert(kLastPartLevels + 1 >= kDeferBuckets, "the other parts are ready in their bin");

// Calls emit(bin, place, task) for each task of tile (I, J); place numbers the
// tasks that tiles of one chain have in the bin.
#pragma nv_exec_check_disable
template <typename F>
__host__ __device__ inline void mcm_tile_tasks(int32_t inst, int I, int J, int levels_per_part, F&& emit) {
  const int D = J - I;
  const McmSplit t = mcm_split(D, levels_per_part);
  McmTask task{inst, (int16_t)I, (int16_t)J, (int16_t)t.lo, (int16_t)t.hi, 0, (int16_t)t.nparts};
  emit(mcm_bin_finisher(D), I, task);
  task.kind = 1;
  task.nparts = 0;
  int r1 = t.lo - 1;
  for (int q = 0; q < t.nparts; ++q) {
    const int r0 = r1 - (q == 0 ? kLastPartLevels : levels_per_part) + 1;
    task.r_lo = (int16_t)(r0 > t.rmin ? r0 : t.rmin);
    task.r_hi = (int16_t)r1;
    if (q == 0) emit(mcm_bin_last(D), I, task);
    else emit(mcm_bin_other(D), I * (t.nparts - 1) + q - 1, task);
    r1 = task.r_lo - 1;
  }
}

// Builds the queue and the split-K slots of a plan on the device.  cursors:
// 3 max_nt first places of the bins, then the slot count (0); consumed.
struct McmQueueArgs {
  const McmInstDev* insts;
  McmTask* tasks;
  int32_t* accslot;
  int32_t* cursors;
  int32_t ninst, max_nt, levels_per_part;
};
cudaError_t launch_mcm_queue(const McmQueueArgs& a, cudaStream_t st);

struct McmLaunchArgs {
  McmInstDev* insts;
  const McmInstDev* insts_from;  // static fields of the records, copied by the prologue (nullptr: already there)
  const McmTask* tasks;
  int32_t ninst;
  int32_t ntasks;
  void* af;                      // packed row panels, tile-major, k-major inside a tile
  void* bf;                      // packed column panels (rows shifted by one), tile-major
  int32_t* flags;                // per tile: 1 once the tile is final
  int32_t* counters;             // per tile: bulk tasks merged so far
  const int32_t* accslot;        // per tile: partial-accumulator slot or -1
  unsigned long long* acc;       // per slot: 32*32 packed (value, k) minima
  int32_t* pp;                   // padded dims
  uint32_t* pk;                  // pk[x] = p[x+1] << S
  int32_t* queue;                // task counter
  void* zero;                    // state the prologue sets to zero (16-byte aligned) ...
  int64_t zero_bytes;            // ... and its size; 0: already done
  int32_t* status;               // device status word
  long long spin_limit;          // clock cycles a wait may take before DP_ETIMEOUT
  int32_t drop_task;             // fault injection: this queue entry is popped but never run (-1: none)
  int32_t pad_;
  const int32_t* p_all;          // prologue inputs
  const int64_t* p_off;          // nullptr: single chain at p_all
  const int64_t* tab_off;        // nullptr: single chain at m_all / s_all
  void* m_all;
  int16_t* s_all;
  // Interval DP (nullptr: plain MCM): per-cell weights laid out like m_all
  // (chain b's n x n table at offset tab_off[b]); w[i][j], i < j, is added to
  // the minimum of cell (i, j), and p may then hold zeros.
  const void* w_all;
  uint32_t one = 1;  // 1, as a value the compiler does not see (fold64 in mcm_tile.cuh)
};

// The int64-cost main kernel (mcm64.cu); the functions below route to it.
size_t mcm64_smem_bytes();
cudaError_t mcm64_configure();
cudaError_t mcm64_occupancy(int* blocks_per_sm);
cudaError_t mcm64_preload();
cudaError_t launch_mcm64(const McmLaunchArgs& a, int grid, cudaStream_t st);

// Launches a main kernel; the blocks of a grid of at most kEarlyGrid may become
// resident while the previous kernel of the stream (the prologue) still runs
// (they call grid_dependency_wait before they read anything it writes).  A
// larger grid starts after it: placed around the prologue's blocks, two blocks
// of a one-per-SM grid land on one SM (int64, n = 1500: 926 -> 1357 us).
constexpr int kEarlyGrid = 64;
template <typename K>
cudaError_t launch_dependent(K kernel, int grid, int threads, size_t smem, cudaStream_t st, const McmLaunchArgs& a) {
  cudaLaunchAttribute attr{};
  attr.id = cudaLaunchAttributeProgrammaticStreamSerialization;
  attr.val.programmaticStreamSerializationAllowed = 1;
  cudaLaunchConfig_t cfg{};
  cfg.gridDim = dim3((unsigned)grid);
  cfg.blockDim = dim3((unsigned)threads);
  cfg.dynamicSmemBytes = smem;
  cfg.stream = st;
  cfg.attrs = &attr;
  cfg.numAttrs = grid <= kEarlyGrid ? 1 : 0;
  return cudaLaunchKernelEx(&cfg, kernel, a);
}

size_t mcm_smem_bytes(bool i64);
cudaError_t mcm_configure(bool i64);
cudaError_t mcm_occupancy(bool i64, int* blocks_per_sm);
// With a.w_all set, the prologue and main kernel are the interval-DP
// instances, and launch_mcm_weight_max must run first (it fills
// McmInstDev::wmax, from which the prologue derives the cost bound).  The
// interval DP exists for int32 costs only: these calls return
// cudaErrorNotSupported for i64 with weights.
cudaError_t launch_mcm_weight_max(const McmLaunchArgs& a, bool i64, int sms, cudaStream_t st);
cudaError_t launch_mcm_prologue(const McmLaunchArgs& a, bool i64, int max_n, int sms, cudaStream_t st);
cudaError_t launch_mcm_main(const McmLaunchArgs& a, bool i64, int grid, cudaStream_t st);
// Loads the prologue, main and split-pass kernels into the current context
// (with lazy module loading a kernel is otherwise loaded at its first launch).
cudaError_t mcm_preload(bool i64);

}  // namespace dpk
