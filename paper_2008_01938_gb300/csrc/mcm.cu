// mcm.cu -- sm_103a kernels for the matrix-chain multiplication table
// (paper Section IV-A, Eq. (2)): the main kernel of the int32-cost and
// interval-DP solves, and the set-up kernels of all (mcm64.cu has the main
// kernel of the int64-cost solves).  See mcm_kernels.cuh for the decomposition
// and the packed cost encodings.
#include <cstdint>

#include "dp_common.cuh"
#include "mcm_kernels.cuh"

namespace dpk {

namespace {

constexpr int T = kTile;
constexpr uint32_t kFinPollNs = 64;   // finisher mbarrier waits (int32): longest sleep between polls
constexpr uint32_t kFlagPollNs = 32;  // flag and counter waits (int32): longest sleep between polls

constexpr int kBlk = T / 2;                // 2x2-cell blocks of a tile, per side
constexpr int kDiagRows = 2 * kBlk - 1;    // block diagonals E = bj - bi in [-15, 15]

using E = uint32_t;      // panel entries: (m << S) | (k mod 2^S)
constexpr int KB = 32;   // k bits in the 64-bit (value, k) key

__device__ __forceinline__ int64_t tile_index(const McmInstDev& in, int I, int J) {
  return in.tile_base + (int64_t)I * in.nt - (int64_t)I * (I - 1) / 2 + (J - I);
}

// Shared-memory carve-up (byte offsets); identical for all blocks.
//
// In-tile wavefront arrays (finisher of an off-diagonal tile) start at STA and
// reuse the bulk-copy stages (every copy of the task has landed before they
// are written), as 2x2-cell blocks of 16 bytes.  Rows of L and U blocks that a
// step reaches beside the tables hold zeros where no cell stands behind them
// (before row 0 of L, after row 15 of U); the others are read only for blocks
// that are final already, and hold anything.  The cell-value arrays Xr / Xc live outside the stage area, so their entries for
// cells that do not exist are set to all ones once per block and stay so
// (every existing cell is written before it is read).
struct Smem {
  static constexpr int ES = 4;
  static constexpr int TILE = T * T * ES;
  static constexpr int BARS = 0;                                 // 9 mbarriers + task slot
  static constexpr int STA = 128;                                // [group][stage] row panels
  static constexpr int STB = STA + 4 * TILE;                     // [group][stage] column panels
  static constexpr int STPK = STB + 4 * TILE;                    // [group][stage] 32 x u32 dims
  static constexpr int STEND = STPK + 4 * 128;
  static constexpr int XBYTES = kDiagRows * kBlk * 16;
  static constexpr int kQRows = 3 * kBlk - 3;                    // 45: every block row a step can reach
  static constexpr int kLRow0 = kBlk - 1;                        // row of block row 0 of L, and of U
  static constexpr int kURow0 = kBlk - 2;
  static constexpr int UQW = 4 * kBlk + 4;                       // pitch of U rows: conflict-free down a column
  static constexpr int WLQ = STA;                                // Lq[kLRow0 + u][bj]: L[2u + s][2 bj + c] at 2 s + c
  static constexpr int WUQ = WLQ + kQRows * 4 * kBlk * ES;       // Uq[kURow0 + b][bi]: m[IT+2bi+r][IT+2b+s-1] at 2 r + s
  static constexpr int WPJ = WUQ + kQRows * UQW * ES;            // p[JT + 2u + s + 1]
  static constexpr int WPI = WPJ + kQRows * 8;                   // p[IT + 2b + s]
  static constexpr int WEND = (WPI + kQRows * 8 + 127) / 128 * 128;
  static constexpr int FINU = ((STEND > WEND ? STEND : WEND) + 127) / 128 * 128;  // row panel of (I,I)
  static constexpr int FINL = FINU + TILE;                       // column panel of diagonal tile (J,J)
  static constexpr int FINBROW = FINL + TILE;                    // boundary row (one tile row)
  static constexpr int FINPP = FINBROW + 256;                    // p[32I .. 32I+31]
  static constexpr int FINPKI = FINPP + 128;                     // p[32I+1 ..] << S
  static constexpr int FINPKJ = FINPKI + 128;                    // p[32J+1 ..] << S
  static constexpr int FINACC = FINPKJ + 128;                    // bulk-task partial minima
  static constexpr int BEST = FINACC + T * T * 8;                // running (value, k) keys
  static constexpr int WXR = BEST + T * T * 8;                   // Xr[E+15][bi]: final values of block (bi, bi+E)
  static constexpr int WXC = WXR + XBYTES;                       // Xc[E+15][bj]: final values of block (bj-E, bj)
  static constexpr int TOTAL = WXC + XBYTES;
  static constexpr int XV = STA;                                 // diagonal tiles: the tile's values
  static_assert(WXR % 16 == 0 && WLQ % 16 == 0 && WUQ % 16 == 0 && (UQW * ES) % 16 == 0 && WPJ % 8 == 0,
                "vector rows");
};

__device__ __forceinline__ void bar_compute() {  // the 256 compute threads only
  asm volatile("bar.sync 1, %0;" ::"n"(kComputeThreads) : "memory");
}

// Barrier over the 256 compute threads that also ANDs a predicate, so a
// decision taken after per-thread bounded waits is the same in every thread
// (every later named barrier is then reached by all 256 or by none).
__device__ __forceinline__ bool bar_compute_and(bool v) {
  uint32_t r;
  asm volatile(
      "{\n\t.reg .pred p, q;\n\t"
      "setp.ne.u32 p, %1, 0;\n\t"
      "bar.red.and.pred q, 1, %2, p;\n\t"
      "selp.u32 %0, 1, 0, q;\n\t}"
      : "=r"(r)
      : "r"((uint32_t)v), "n"(kComputeThreads)
      : "memory");
  return r != 0;
}

template <typename E>
__device__ __forceinline__ E umin(E a, E b) { return a < b ? a : b; }

// ---------------------------------------------------------------------------
// In-tile solve of an off-diagonal tile (I, J).
// X is the tile; its in-tile splits are
//   column splits k = IT + t, li <= t <= 30:  U[li][t] + X[t+1][lj] + w
//   row splits    k = JT + u,  0 <= u < lj:   X[li][u] + L[u][lj] + w
// with U = the diagonal tile (I, I), L = rows shifted by one of (J, J) and
// w = p[IT+li] p[k+1] p[JT+lj+1]; the boundary split k = IT + 31 and the
// external splits are known before the solve starts.
//
// A thread owns a block of 2x2 cells, (2 bi + r, 2 bj + c).  The block lies on
// block diagonal E = bj - bi in [-15, 15] and depends only on blocks of lower
// diagonals, so the tile is solved in the paper's diagonal order (Figs. 5-7),
// one block diagonal per step: in step E every block pulls the candidates of
// the two column splits and the two row splits per cell whose operands lie in
// blocks of diagonal E, and the blocks of diagonal E + 1, whose last operands
// those were, become final: their cells depend on one another through one
// split each in one or two more links, in registers.  Warp w owns block rows
// 2w and 2w + 1.
//
// The solve is a chain of steps (barrier, load, minima, store), and on it hangs
// the time between two tile diagonals.  Cell by cell it is 62 steps of 170
// clocks, by blocks 30 of about 210 for the same candidates: n = 128: 45.9 ->
// 38.8 us, 1000 (tables to the host) 389 -> 322, 4096 1980 -> 1798, interval DP
// of 2000 670 -> 579.  (Blocks of 8x8 cells, one warp each without barriers
// inside, took 17.3 k clocks a tile against the cells' 10.5 k.)
//
// Each thread keeps one running minimum per cell (values only).  The operands
// that do not depend on the tile are laid out as blocks, one 16-byte load per
// step each, loaded and multiplied ahead of the barrier.  The cell values
// themselves are exchanged through two arrays of blocks by diagonal, written
// once, when a block becomes final: Xr (indexed by block row, the row-split
// operand) and Xc (indexed by block column, the column-split operand).
//
// Out-of-range operands are read from zero rows (U, L, dims) and from
// all-ones entries (cells that do not exist), so no candidate needs a
// predicate: a missing cell yields an all-ones candidate, and a candidate
// whose operand exists but whose split is outside the cell's range only
// arises after the block was finalised (its running minimum is then dead).
// The smallest minimising split is recovered after the tile is published, by
// scanning the splits of each cell in increasing k.
// ---------------------------------------------------------------------------
__device__ __forceinline__ uint4 lds4(const E* p) { return *reinterpret_cast<const uint4*>(p); }  // 16-byte aligned
__device__ __forceinline__ uint2 lds2(const E* p) { return *reinterpret_cast<const uint2*>(p); }  // 8-byte aligned

// ---------------------------------------------------------------------------
// Bulk segment reductions (one compute group, 128 threads, 4 x 2 cells each).
// ---------------------------------------------------------------------------

// int32 costs, chunks of 2^LOGC aligned splits.
template <int LOGC>
__device__ __forceinline__ void seg_i32(const uint32_t* __restrict__ A, const uint32_t* __restrict__ B,
                                        const uint32_t* __restrict__ PK, const uint32_t (&P)[4][2],
                                        unsigned long long (&best)[4][2], int ty, int tx, int S, int KT) {
  constexpr int C = 1 << LOGC;
#pragma unroll 1
  for (int c0 = 0; c0 < T; c0 += C) {
    uint32_t acc[4][2];
#pragma unroll
    for (int r = 0; r < 4; ++r) acc[r][0] = acc[r][1] = 0xFFFFFFFFu;
    // One split evaluation is a multiply-add on the FMA pipe (weight plus the
    // row-panel key) and a fused add-and-minimum (__viaddmin_u32, one ALU-pipe
    // instruction) that adds the column-panel key and folds the candidate
    // into the running minimum: two instructions, one on each integer pipe.
#pragma unroll
    for (int kk = 0; kk < C; kk += 2) {
      const uint4 a0 = *reinterpret_cast<const uint4*>(A + (c0 + kk) * T + 4 * ty);
      const uint2 b0 = *reinterpret_cast<const uint2*>(B + (c0 + kk) * T + 2 * tx);
      const uint4 a1 = *reinterpret_cast<const uint4*>(A + (c0 + kk + 1) * T + 4 * ty);
      const uint2 b1 = *reinterpret_cast<const uint2*>(B + (c0 + kk + 1) * T + 2 * tx);
      const uint32_t pk0 = PK[c0 + kk], pk1 = PK[c0 + kk + 1];
      const uint32_t av0[4] = {a0.x, a0.y, a0.z, a0.w}, av1[4] = {a1.x, a1.y, a1.z, a1.w};
      const uint32_t bv0[2] = {b0.x, b0.y}, bv1[2] = {b1.x, b1.y};
#pragma unroll
      for (int r = 0; r < 4; ++r)
#pragma unroll
        for (int c = 0; c < 2; ++c) {
          acc[r][c] = __viaddmin_u32(P[r][c] * pk0 + av0[r], bv0[c], acc[r][c]);
          acc[r][c] = __viaddmin_u32(P[r][c] * pk1 + av1[r], bv1[c], acc[r][c]);
        }
    }
#pragma unroll
    for (int r = 0; r < 4; ++r)
#pragma unroll
      for (int c = 0; c < 2; ++c) {
        const unsigned long long v = acc[r][c] >> S;
        const unsigned long long k = (unsigned)(KT + c0) + (acc[r][c] & (C - 1));
        best[r][c] = umin(best[r][c], (v << 32) | k);
      }
  }
}

// Walks the external segments of a task in the order both roles agree on.
template <typename F>
__device__ __forceinline__ void for_each_segment(const McmTask& t, F&& body) {
  int q = 0;
  for (int r = t.r_lo; r <= t.r_hi; ++r) {
#pragma unroll 1
    for (int h = 0; h < 2; ++h) {
      const int K = h == 0 ? t.I + r : t.J - r;
      if (h == 1 && K == t.I + r) continue;
      if (K < t.I + 1 || K > t.J - 1) continue;
      body(K, q);
      ++q;
    }
  }
}

template <bool W>
__global__ void __launch_bounds__(kMcmThreads, 3) mcm_main_kernel(const McmLaunchArgs a) {
  using SM = Smem;
  extern __shared__ __align__(128) uint8_t smem[];
  uint64_t* bar_full = reinterpret_cast<uint64_t*>(smem + SM::BARS);      // [g*2+st]
  uint64_t* bar_empty = bar_full + 4;                                      // [g*2+st]
  uint64_t* bar_fin = bar_full + 8;
  volatile int32_t* task_slot = reinterpret_cast<volatile int32_t*>(smem + SM::BARS + 80);
  E* stA = reinterpret_cast<E*>(smem + SM::STA);
  E* stB = reinterpret_cast<E*>(smem + SM::STB);
  uint32_t* stPK = reinterpret_cast<uint32_t*>(smem + SM::STPK);
  E* finU = reinterpret_cast<E*>(smem + SM::FINU);
  E* finL = reinterpret_cast<E*>(smem + SM::FINL);
  E* finBrow = reinterpret_cast<E*>(smem + SM::FINBROW);
  int32_t* finPP = reinterpret_cast<int32_t*>(smem + SM::FINPP);
  uint32_t* finPKI = reinterpret_cast<uint32_t*>(smem + SM::FINPKI);
  uint32_t* finPKJ = reinterpret_cast<uint32_t*>(smem + SM::FINPKJ);
  unsigned long long* finAcc = reinterpret_cast<unsigned long long*>(smem + SM::FINACC);
  unsigned long long* bestS = reinterpret_cast<unsigned long long*>(smem + SM::BEST);
  E* Xv = reinterpret_cast<E*>(smem + SM::XV);  // in-tile solve only (stage area)

  const int tid = threadIdx.x;
  const int warp = tid >> 5;
  const int lane = tid & 31;
  const long long limit = a.spin_limit;
  int32_t* status = a.status;

  E* x = reinterpret_cast<E*>(smem + SM::WXR);
  for (int i = tid; i < 2 * SM::XBYTES / SM::ES; i += blockDim.x) x[i] = ~(E)0;
  if (tid == 0) {
    for (int i = 0; i < 4; ++i) {
      mbar_init(&bar_full[i], 1);
      mbar_init(&bar_empty[i], kGroupThreads);
    }
    mbar_init(bar_fin, 1);
    fence_mbar_init();
  }
  __syncthreads();

  grid_dependency_wait();  // the set-up kernel's writes

  // Per-role running counters (each role walks the same segment sequence).
  uint32_t use_cnt[2] = {0u, 0u};   // producer: stage uses issued per group; consumer: own group
  uint32_t fin_cnt = 0;             // finisher-barrier uses

  while (true) {
    if (tid == 0) {
      int32_t t = -1;
      if (*reinterpret_cast<volatile int32_t*>(status) == 0) t = atomicAdd(a.queue, 1);
      *task_slot = t;
    }
    __syncthreads();
    const int32_t tix = *task_slot;
    if (tix < 0 || tix >= a.ntasks) break;
    if (tix == a.drop_task) {  // injected fault: the task's flag is never published
      __syncthreads();
      continue;
    }
    const McmTask task = a.tasks[tix];
    const McmInstDev inst = a.insts[task.inst];
    const int I = task.I, J = task.J, D = J - I;
    const int IT = I * T, JT = J * T;
    const int64_t tidx = tile_index(inst, I, J);
    const bool finisher = task.kind == 0;
    const int S = inst.shift;
    const int32_t accslot = a.accslot[tidx];

    if (warp == kComputeThreads / 32) {
      // ===================== producer warp =====================
      // The lanes poll a flag each, so that all the flags waited for cost one
      // round trip together; lane 0 issues the copies.
      //
      // The stage area was written and read through the generic proxy by the
      // previous task's in-tile solve; order that before this task's copies.
      asm volatile("fence.proxy.async.shared::cta;" ::: "memory");
      bool ok = true;
      uint32_t issued = 0u, parity = 0u;  // a bit per group and stage (arrays here lived in local memory: 4096 1799 -> 1781 us)
      bool fin_issued = false;
      const int32_t* const flags = a.flags + inst.tile_base;
      auto tile = [&](int i, int j) { return i * inst.nt - i * (i - 1) / 2 + (j - i); };
      // the lane's flag of segment K, for lanes 0 .. 2: tiles (I, K), (K, J), (K + 1, J)
      auto segment_flag = [&](int K, int x) {
        return flags + tile(x == 0 ? I : x == 1 ? K : K + 1, x == 0 ? K : J);
      };
      auto copy_segment = [&](int K, int g, uint32_t u) {
        const int st = u % kStages;
        const uint32_t round = u / kStages;
        bool got = true;
        if (lane == 0) {
          fence_proxy_async_global();
          got = mbar_wait(&bar_empty[g * kStages + st], (round & 1u) ^ 1u, limit);
          if (got) {
            uint64_t* fb = &bar_full[g * kStages + st];
            mbar_arrive_expect_tx(fb, 2 * SM::TILE + 128);
            bulk_g2s(stA + (g * kStages + st) * T * T,
                     static_cast<const E*>(a.af) + tile_index(inst, I, K) * T * T, SM::TILE, fb);
            bulk_g2s(stB + (g * kStages + st) * T * T,
                     static_cast<const E*>(a.bf) + tile_index(inst, K, J) * T * T, SM::TILE, fb);
            bulk_g2s(stPK + (g * kStages + st) * 32, a.pk + inst.pk_base + (int64_t)K * T, 128, fb);
          } else {
            set_status(status, DP_ETIMEOUT);
          }
        }
        got = __shfl_sync(~0u, (int)got, 0) != 0;
        if (got) {
          const uint32_t bit = 1u << (g * kStages + st);
          issued |= bit;
          parity = (round & 1u) ? parity | bit : parity & ~bit;
        }
        return got;
      };
      // Polls the lanes' flags until `stop` (called with the mask of the lanes
      // that are done) returns true; false after an error or `limit` clocks.
      auto poll = [&](const int32_t* f, int32_t target, bool done, auto&& stop) {
        const long long t0 = clock64();
        for (int32_t failed = 0;; failed = *reinterpret_cast<volatile const int32_t*>(status)) {
          if (!done) done = ld_acquire(f) >= target;
          const uint32_t have = __ballot_sync(~0u, done);
          __syncwarp();
          if (stop(have)) return true;
          const bool late = clock64() - t0 > limit;
          if (late && lane == 0) set_status(status, DP_ETIMEOUT);
          if (__shfl_sync(~0u, (int)(late || failed != 0), 0) != 0) return false;
          __nanosleep(kFlagPollNs);
        }
      };
      // A finisher's last two segments (its neighbours' tiles) and its own
      // operands become ready at about the same time, in no fixed order: their
      // flags are waited for together, one round trip a poll, and the copies
      // of the segments go first.  (Flags one after the other in lane 0: the
      // second segment arrived 1.3 k clocks after the first.  n = 300 89.3 ->
      // 83.4 us, 1000 255 -> 230, 2000 559 -> 529, 3000 985 -> 963, 4096 1798
      // -> 1811, interval DP of 2000 592 -> 569; operands' copies as soon as
      // they may: 1 to 2% slower.)
      int nseg = 0;
      if (finisher) for_each_segment(task, [&](int, int q) { nseg = q + 1; });
      int late_k[2] = {0, 0};
      uint32_t late_u[2] = {0u, 0u};
      for_each_segment(task, [&](int K, int q) {
        const int g = q & 1;
        const uint32_t u = use_cnt[g]++;
        if (finisher && q >= nseg - 2) {
          if (g == 0) late_k[0] = K, late_u[0] = u;
          else late_k[1] = K, late_u[1] = u;
          return;
        }
        if (!ok) return;
        ok = poll(segment_flag(K, lane < 3 ? lane : 0), 1, lane >= 3, [&](uint32_t have) { return have == ~0u; }) &&
             copy_segment(K, g, u);
      });
      if (finisher && ok) {
        // lanes 0 .. 2 and 3 .. 5: the segments; 6 .. 8: tiles (I, I), (J, J),
        // (I+1, J); 9: the bulk-task counter
        bool want[2] = {nseg > 0, nseg > 1}, want_fin = true, got = true;
        const int32_t* f = a.counters + tidx;
        int32_t target = lane == 9 ? task.nparts : 0;
        if (lane < 6) {
          const int g = lane / 3;
          if (nseg > g) f = segment_flag(g == 0 ? late_k[0] : late_k[1], lane - 3 * g), target = 1;
        } else if (lane < 9 && D >= 1) {
          f = flags + (lane == 6 ? tile(I, I) : lane == 7 ? tile(J, J) : tile(I + 1, J));
          target = 1;
        }
        const bool polled = poll(f, target, target == 0, [&](uint32_t have) {
          if (want[0] && (have & 0x7u) == 0x7u) want[0] = false, got = got && copy_segment(late_k[0], 0, late_u[0]);
          if (want[1] && (have & 0x38u) == 0x38u) want[1] = false, got = got && copy_segment(late_k[1], 1, late_u[1]);
          if (want_fin && !want[0] && !want[1] && (have & 0x3C0u) == 0x3C0u) {
            want_fin = false;
            fin_issued = got;
            if (got && lane == 0) {
              fence_proxy_async_global();
              uint32_t bytes = 3 * 128;
              if (D >= 1) bytes += 2 * SM::TILE + T * (uint32_t)sizeof(E);
              if (task.nparts > 0) bytes += T * T * 8;
              mbar_arrive_expect_tx(bar_fin, bytes);
              bulk_g2s(finPP, a.pp + inst.pp_base + IT, 128, bar_fin);
              bulk_g2s(finPKI, a.pk + inst.pk_base + IT, 128, bar_fin);
              bulk_g2s(finPKJ, a.pk + inst.pk_base + JT, 128, bar_fin);
              if (D >= 1) {
                bulk_g2s(finU, static_cast<const E*>(a.af) + tile_index(inst, I, I) * T * T, SM::TILE, bar_fin);
                bulk_g2s(finL, static_cast<const E*>(a.bf) + tile_index(inst, J, J) * T * T, SM::TILE, bar_fin);
                bulk_g2s(finBrow, static_cast<const E*>(a.bf) + tidx * T * T + (T - 1) * T, T * sizeof(E), bar_fin);
              }
              if (task.nparts > 0) bulk_g2s(finAcc, a.acc + (int64_t)accslot * T * T, T * T * 8, bar_fin);
            }
          }
          return !got || (!want[0] && !want[1] && !want_fin);
        });
        ok = polled && got;
      }
      if (lane == 0) {
        // (A finisher whose operands' flags did not come copies nothing, and its
        // compute threads' wait runs out as well: the tile is then neither
        // solved nor published, and with the status word set this is the block's
        // last task.)
        // No bulk copy may still be in flight when the task ends.
        for (int g = 0; g < 2; ++g)
          for (int st = 0; st < kStages; ++st)
            if (issued >> (g * kStages + st) & 1u)
              mbar_wait(&bar_full[g * kStages + st], parity >> (g * kStages + st) & 1u, limit * 4);
        if (fin_issued) mbar_wait(bar_fin, fin_cnt & 1u, limit * 4);
      }
    } else {
      // ===================== compute threads (2 groups) =====================
      const int g = warp >> 2;
      const int tg = tid & (kGroupThreads - 1);
      const int ty = tg >> 4, tx = tg & 15;
      unsigned long long best[4][2];
      uint32_t P[4][2];
#pragma unroll
      for (int r = 0; r < 4; ++r) {
        const uint32_t pi = (uint32_t)a.pp[inst.pp_base + IT + 4 * ty + r];
#pragma unroll
        for (int c = 0; c < 2; ++c) {
          P[r][c] = pi * (uint32_t)a.pp[inst.pp_base + JT + 2 * tx + c + 1];
          best[r][c] = ~0ull;
        }
      }
      bool ok = true;
      for_each_segment(task, [&](int K, int q) {
        if ((q & 1) != g) return;
        const uint32_t u = use_cnt[g]++;
        const int st = u % kStages;
        const uint32_t round = u / kStages;
        if (!ok) return;
        // a finisher's segments are on the critical path: poll more often
        const bool got = finisher ? mbar_wait_cap(&bar_full[g * kStages + st], round & 1u, limit, kFinPollNs)
                                  : mbar_wait(&bar_full[g * kStages + st], round & 1u, limit);
        if (!got) {
          set_status(status, DP_ETIMEOUT);
          ok = false;
          return;
        }
        const E* A = stA + (g * kStages + st) * T * T;
        const E* B = stB + (g * kStages + st) * T * T;
        const uint32_t* PK = stPK + (g * kStages + st) * 32;
        const int logc = S < 5 ? S : 5;
        switch (logc) {
          case 5: seg_i32<5>(A, B, PK, P, best, ty, tx, S, K * T); break;
          case 4: seg_i32<4>(A, B, PK, P, best, ty, tx, S, K * T); break;
          case 3: seg_i32<3>(A, B, PK, P, best, ty, tx, S, K * T); break;
          case 2: seg_i32<2>(A, B, PK, P, best, ty, tx, S, K * T); break;
          default: seg_i32<1>(A, B, PK, P, best, ty, tx, S, K * T); break;
        }
        mbar_arrive(&bar_empty[g * kStages + st]);
      });

      // (a finisher's look at the error status, early enough to be there when it is needed)
      const int32_t failed = finisher ? *reinterpret_cast<volatile const int32_t*>(status) : 0;
      // merge the two groups' minima: group 1 publishes, group 0 combines
      if (g == 1) {
#pragma unroll
        for (int r = 0; r < 4; ++r)
#pragma unroll
          for (int c = 0; c < 2; ++c) bestS[(4 * ty + r) * T + 2 * tx + c] = best[r][c];
      }
      bar_compute();
      if (g == 0) {
#pragma unroll
        for (int r = 0; r < 4; ++r)
#pragma unroll
          for (int c = 0; c < 2; ++c) {
            const int cell = (4 * ty + r) * T + 2 * tx + c;
            const unsigned long long v = umin(best[r][c], bestS[cell]);
            if (finisher)
              bestS[cell] = v;
            else if (v != ~0ull)
              atomicMin(a.acc + (int64_t)accslot * T * T + cell, v);
          }
      }

      if (finisher) {
        bar_compute();
        // ------------------ in-tile wavefront (finisher) ------------------
        // The thread's 4 cells: off-diagonal tiles, the 2x2 block (bi, bj); the
        // diagonal tile, rows 4w .. 4w + 3 of column lane.
        const int w = warp;
        const int bi = 2 * w + (lane >> 4), bj = lane & (kBlk - 1);
        // interval DP: the weights of the cells, loaded while the copies land
        E wt[4] = {0, 0, 0, 0};
        if constexpr (W) {
#pragma unroll
          for (int r = 0; r < 4; ++r) {
            const int64_t i = IT + (D >= 1 ? 2 * bi + (r >> 1) : 4 * w + r), j = JT + (D >= 1 ? 2 * bj + (r & 1) : lane);
            if (i < j && j < inst.n) wt[r] = static_cast<const E*>(inst.w)[i * inst.n + j];
          }
        }
        const uint32_t fpar = fin_cnt & 1u;
        const bool fin_ok = mbar_wait_cap(bar_fin, fpar, limit, kFinPollNs);
        if (!fin_ok) set_status(status, DP_ETIMEOUT);
        const bool go = bar_compute_and(fin_ok && failed == 0);
        const int n = inst.n;
        const E pj1 = (E)(finPKJ[lane] >> S);  // p[JT + lane + 1]
        if (go) {
          if (D >= 1) {
            E* Lq = reinterpret_cast<E*>(smem + SM::WLQ);
            E* Uq = reinterpret_cast<E*>(smem + SM::WUQ);
            E* PJ = reinterpret_cast<E*>(smem + SM::WPJ);
            E* PI = reinterpret_cast<E*>(smem + SM::WPI);
            E* Xr = reinterpret_cast<E*>(smem + SM::WXR);
            E* Xc = reinterpret_cast<E*>(smem + SM::WXC);
            // operands in blocks (thread: block row tid / 16, block column tid % 16)
            {
              const int y = tid >> 4, x = tid & (kBlk - 1);
              const uint2 l0 = lds2(finL + 2 * y * T + 2 * x), l1 = lds2(finL + (2 * y + 1) * T + 2 * x);
              const bool in1 = y < kBlk - 1;  // L has 31 rows
              *reinterpret_cast<uint4*>(Lq + ((SM::kLRow0 + y) * kBlk + x) * 4) =
                  make_uint4(l0.x >> S, l0.y >> S, in1 ? l1.x >> S : 0u, in1 ? l1.y >> S : 0u);
              const uint2 u1 = lds2(finU + 2 * y * T + 2 * x), u0 = lds2(finU + (y > 0 ? 2 * y - 1 : 0) * T + 2 * x);
              *reinterpret_cast<uint4*>(Uq + (SM::kURow0 + y) * SM::UQW + 4 * x) =
                  make_uint4(u0.x >> S, u1.x >> S, u0.y >> S, u1.y >> S);
              if (y < kBlk - 1) {  // block rows that do not exist: -15 .. -1 of L, 16 .. 30 of U
                *reinterpret_cast<uint4*>(Lq + (y * kBlk + x) * 4) = make_uint4(0u, 0u, 0u, 0u);
                *reinterpret_cast<uint4*>(Uq + (SM::kURow0 + kBlk + y) * SM::UQW + 4 * x) = make_uint4(0u, 0u, 0u, 0u);
              }
              if (tid < T) {
                PJ[2 * SM::kLRow0 + tid] = finPKJ[tid] >> S;
                PI[2 * SM::kURow0 + tid] = finPP[tid];
              } else if (tid < 2 * T - 2) {
                PJ[tid - T] = 0u;
                PI[2 * (SM::kURow0 + kBlk) + tid - T] = 0u;
              }
            }
            // boundary split k = IT + 31: U[li][31] + m[IT+32][j] + w
            const E pI32 = (E)(finPKI[T - 1] >> S);
            const E pib = finPP[2 * bi + 1], pjb = finPKJ[2 * bj] >> S;  // p[IT + 2 bi + 1], p[JT + 2 bj + 1]
            E m[4], wv[4];  // cell (2 bi + r, 2 bj + c) at 2 r + c
            E ib[4];        // multiplier terms of the splits inside the block: 0,0 / 1,1 / 0,1 by row / 0,1 by column
            {
              const uint2 br = lds2(finBrow + 2 * bj), pj = lds2(finPKJ + 2 * bj);
              const uint2 ub = lds2(finU + (T - 1) * T + 2 * bi), pp = lds2(reinterpret_cast<const E*>(finPP) + 2 * bi);
              wv[0] = pp.x * (pj.x >> S), wv[1] = pp.x * (pj.y >> S);
              wv[2] = pp.y * (pj.x >> S), wv[3] = pp.y * (pj.y >> S);
#pragma unroll
              for (int r = 0; r < 2; ++r) {
                ulonglong2* own = reinterpret_cast<ulonglong2*>(bestS + (2 * bi + r) * T + 2 * bj);
                ulonglong2 cb = *own;
                if (task.nparts > 0) {
                  const ulonglong2 ac = *reinterpret_cast<const ulonglong2*>(finAcc + (2 * bi + r) * T + 2 * bj);
                  cb.x = umin(cb.x, ac.x);
                  cb.y = umin(cb.y, ac.y);
                  *own = cb;  // external minimum: (value, smallest k)
                }
                const E u31 = (r ? ub.y : ub.x) >> S;
                m[2 * r] = umin((E)(cb.x >> KB), u31 + (br.x >> S) + wv[2 * r] * pI32);
                m[2 * r + 1] = umin((E)(cb.y >> KB), u31 + (br.y >> S) + wv[2 * r + 1] * pI32);
              }
              ib[0] = wv[0] * pib, ib[1] = wv[3] * pjb, ib[2] = wv[1] * pjb, ib[3] = wv[1] * pib;
            }
            // The block's final values, in the order of its cell diagonals; the
            // one split inside it adds a table value 0.
            auto block_values = [&]() {
              uint4 v;
              v.z = m[2];
              if constexpr (W) v.z += wt[2];
              v.x = __viaddmin_u32(v.z, ib[0], m[0]);
              v.w = __viaddmin_u32(v.z, ib[1], m[3]);
              if constexpr (W) v.x += wt[0], v.w += wt[3];
              v.y = __viaddmin_u32(v.x, ib[2], __viaddmin_u32(v.w, ib[3], m[1]));
              if constexpr (W) v.y += wt[1];
              return v;
            };
            const int fd = bj - bi;  // the block's diagonal
            E* const xr0 = Xr + (kBlk - 1) * kBlk * 4 + 4 * bi;  // + 4 kBlk E: block (bi, bi + E)
            E* const xc0 = Xc + (kBlk - 1) * kBlk * 4 + 4 * bj;  // + 4 kBlk E: block (bj - E, bj)
            if (fd == 1 - kBlk) {  // block (15, 0), the only one of its diagonal
              const uint4 v = block_values();
              *reinterpret_cast<uint4*>(xr0 + 4 * kBlk * (1 - kBlk)) = v;
              *reinterpret_cast<uint4*>(xc0 + 4 * kBlk * (1 - kBlk)) = v;
            }
            bar_compute();
            // 30 steps, unrolled: every shared-memory operand is a constant
            // offset from a per-thread base.  What does not depend on the tile
            // is loaded at the start of the step before and multiplied at its
            // end, so that after a barrier a candidate is one fused
            // add-and-minimum.
            const E* const l0 = Lq + (SM::kLRow0 + bi) * kBlk * 4 + 4 * bj;   // + 4 kBlk E
            const E* const u0 = Uq + (SM::kURow0 + bj) * SM::UQW + 4 * bi;    // - UQW E
            const E* const pj0 = PJ + 2 * (SM::kLRow0 + bi);                  // + 2 E
            const E* const pi0 = PI + 2 * (SM::kURow0 + bj);                  // - 2 E
            const int e_last = kBlk - 2 - 2 * w;  // the warp's last block, (2w, 15), is final after this step
            E rc[8], cc[8];  // candidates less the tile value: cell 2 r + c, operand s at 2 (2 r + c) + s
            auto terms = [&](const uint4& l, const uint4& u, const uint2& qj, const uint2& qi) {
              rc[0] = l.x + wv[0] * qj.x, rc[1] = l.z + wv[0] * qj.y;
              rc[2] = l.y + wv[1] * qj.x, rc[3] = l.w + wv[1] * qj.y;
              rc[4] = l.x + wv[2] * qj.x, rc[5] = l.z + wv[2] * qj.y;
              rc[6] = l.y + wv[3] * qj.x, rc[7] = l.w + wv[3] * qj.y;
              cc[0] = u.x + wv[0] * qi.x, cc[1] = u.y + wv[0] * qi.y;
              cc[2] = u.x + wv[1] * qi.x, cc[3] = u.y + wv[1] * qi.y;
              cc[4] = u.z + wv[2] * qi.x, cc[5] = u.w + wv[2] * qi.y;
              cc[6] = u.z + wv[3] * qi.x, cc[7] = u.w + wv[3] * qi.y;
            };
            terms(lds4(l0 + 4 * kBlk * (1 - kBlk)), lds4(u0 - SM::UQW * (1 - kBlk)), lds2(pj0 + 2 * (1 - kBlk)),
                  lds2(pi0 - 2 * (1 - kBlk)));
#pragma unroll
            for (int e = 1 - kBlk; e <= kBlk - 2; ++e) {
              if (e <= e_last) {
                const uint4 xr = lds4(xr0 + 4 * kBlk * e);  // X[2 bi + r][2 (bi + e) + s] at 2 r + s
                const uint4 xc = lds4(xc0 + 4 * kBlk * e);  // X[2 (bj - e) + s][2 bj + c] at 2 s + c
                uint4 l = {}, u = {};
                uint2 qj = {}, qi = {};
                if (e < kBlk - 2) {
                  l = lds4(l0 + 4 * kBlk * (e + 1));
                  u = lds4(u0 - SM::UQW * (e + 1));
                  qj = lds2(pj0 + 2 * (e + 1));
                  qi = lds2(pi0 - 2 * (e + 1));
                }
                m[2] = __viaddmin_u32(rc[4], xr.z, m[2]);
                m[0] = __viaddmin_u32(rc[0], xr.x, m[0]);
                m[3] = __viaddmin_u32(rc[6], xr.z, m[3]);
                m[1] = __viaddmin_u32(rc[2], xr.x, m[1]);
                m[2] = __viaddmin_u32(rc[5], xr.w, m[2]);
                m[0] = __viaddmin_u32(rc[1], xr.y, m[0]);
                m[3] = __viaddmin_u32(rc[7], xr.w, m[3]);
                m[1] = __viaddmin_u32(rc[3], xr.y, m[1]);
                m[2] = __viaddmin_u32(cc[4], xc.x, m[2]);
                m[0] = __viaddmin_u32(cc[0], xc.x, m[0]);
                m[3] = __viaddmin_u32(cc[6], xc.y, m[3]);
                m[1] = __viaddmin_u32(cc[2], xc.y, m[1]);
                m[2] = __viaddmin_u32(cc[5], xc.z, m[2]);
                m[0] = __viaddmin_u32(cc[1], xc.z, m[0]);
                m[3] = __viaddmin_u32(cc[7], xc.w, m[3]);
                m[1] = __viaddmin_u32(cc[3], xc.w, m[1]);
                // blocks on diagonal e + 1 are final now
                const uint4 v = block_values();
                if (fd == e + 1) {
                  *reinterpret_cast<uint4*>(xr0 + 4 * kBlk * (e + 1)) = v;
                  *reinterpret_cast<uint4*>(xc0 + 4 * kBlk * (e + 1)) = v;
                }
                if (e < kBlk - 2) terms(l, u, qj, qi);
              }
              bar_compute();
            }
            // ---------------- panels needed by other tiles, then publish ----------------
            const int64_t nn = n;
            E vals[4];
#pragma unroll
            for (int r = 0; r < 4; ++r)  // cell (4w + r, lane)
              vals[r] = Xc[(((lane >> 1) - 2 * w - (r >> 1) + kBlk - 1) * kBlk + (lane >> 1)) * 4 + 2 * (r & 1) + (lane & 1)];
            {
              E* af = static_cast<E*>(a.af) + tidx * T * T;
              E pa[4];
#pragma unroll
              for (int r = 0; r < 4; ++r) {
                pa[r] = (vals[r] << S) | (E)(lane & ((1 << (S < 5 ? S : 5)) - 1));
              }
              *reinterpret_cast<uint4*>(af + lane * T + 4 * w) = make_uint4(pa[0], pa[1], pa[2], pa[3]);
              E* bf = static_cast<E*>(a.bf);
#pragma unroll
              for (int r = 0; r < 4; ++r) {
                const int li = 4 * w + r;
                const E pb = vals[r] << S;
                if (li >= 1)
                  bf[tidx * T * T + (li - 1) * T + lane] = pb;
                else if (I >= 1)
                  bf[tile_index(inst, I - 1, J) * T * T + (T - 1) * T + lane] = pb;
              }
            }
            bar_compute();
            // release: the panel stores of every compute thread, ordered before
            // this store by the barrier, are visible to whoever acquires the flag
            if (tid == 0) st_release(a.flags + tidx, 1);
            // ---------------- the tables themselves (not read by other tiles) ----------------
#pragma unroll
            for (int r = 0; r < 4; ++r) {
              const int li = 4 * w + r;
              const int64_t i = IT + li, j = JT + lane;
              if (i < nn && j < nn) {
                static_cast<int32_t*>(inst.m)[i * nn + j] = (int32_t)vals[r];
              }
              const int64_t i2 = JT + li, j2 = IT + lane;  // mirror tile (J, I)
              if (i2 < nn && j2 < nn) {
                static_cast<int32_t*>(inst.m)[i2 * nn + j2] = 0;
                inst.s[i2 * nn + j2] = -1;
              }
            }
            // ---------------- split table (off the critical path) ----------------
            // The smallest k reaching the final value, scanning in increasing
            // k: column splits IT+li .. IT+30, the boundary IT+31, the
            // external splits (smallest one kept with the external minimum),
            // row splits JT .. j-1.
            const unsigned long long kmask = (1ull << KB) - 1ull;
            const E brow = finBrow[lane] >> S;
            const int cb = lane >> 1, cc1 = lane & 1;  // the column's block, and which of its columns
            // word offset of row or column x (x = t + 1 for column splits) in an
            // array of blocks
            auto at = [](int x, int pitch, int odd) { return (x >> 1) * pitch + (x & 1) * odd; };
#pragma unroll 1
            for (int r = 0; r < 4; ++r) {
              // warp w scans rows w, w + 8, w + 16 and w + 24, a mix of
              // long and short column scans, so that the warps finish together
              // (the value, weight and multiplier of the row are read again)
              const int li = w + 8 * r;
              const int64_t i = IT + li, j = JT + lane;
              if (i >= nn || j >= nn) continue;
              const int lb = li >> 1, lr = li & 1;
              E v;   // the minimum, less the cell's own weight
              E wr;  // the row's multiplier p[i] p[j+1]
              v = Xc[((cb - lb + kBlk - 1) * kBlk + cb) * 4 + 2 * lr + cc1];
              if constexpr (W) v -= static_cast<const E*>(inst.w)[i * inst.n + j];
              wr = (E)finPP[li] * pj1;
              int k = -1;
              // four splits per round with independent loads, the
              // smallest matching one kept; a lane stops after the first
              // round with a match (reads past the last split stay inside
              // shared memory and are not used)
              const E* us = Uq + SM::kURow0 * SM::UQW + 4 * lb + 2 * lr;            // + at(x, UQW, 1)
              const E* xs = Xc + ((cb + kBlk - 1) * kBlk + cb) * 4 + cc1;           // + at(x, -4 kBlk, 2)
              const E* ps = PI + 2 * SM::kURow0;                                    // + x
              int uo[4], xo[4];
#pragma unroll
              for (int d = 0; d < 4; ++d) uo[d] = at(li + 1 + d, SM::UQW, 1), xo[d] = at(li + 1 + d, -4 * kBlk, 2);
              for (int t0 = li; t0 <= T - 2 && k < 0; t0 += 4) {
                E c4[4];
#pragma unroll
                for (int d = 0; d < 4; ++d) c4[d] = us[uo[d]] + xs[xo[d]] + wr * ps[t0 + 1 + d];
#pragma unroll
                for (int d = 3; d >= 0; --d)
                  if (t0 + d <= T - 2 && c4[d] == v) k = IT + t0 + d;
                us += 2 * SM::UQW;
                xs -= 8 * kBlk;
              }
              if (k < 0 && (finU[(T - 1) * T + li] >> S) + brow + wr * pI32 == v) k = IT + T - 1;
              if (k < 0) {
                const unsigned long long ek = bestS[li * T + lane];
                if ((E)(ek >> KB) == v) k = (int)(ek & kmask);
              }
              if (k < 0) {
                const E* rs = Xr + ((kBlk - 1 - lb) * kBlk + lb) * 4 + 2 * lr;  // + at(u, 4 kBlk, 1)
                const E* ls = Lq + (SM::kLRow0 * kBlk + cb) * 4 + cc1;          // + at(u, 4 kBlk, 2)
                for (int u0 = 0; u0 < lane && k < 0; u0 += 4) {
                  E c4[4];
#pragma unroll
                  for (int d = 0; d < 4; ++d)
                    c4[d] = rs[at(d, 4 * kBlk, 1)] + ls[at(d, 4 * kBlk, 2)] + wr * PJ[2 * SM::kLRow0 + u0 + d];
#pragma unroll
                  for (int d = 3; d >= 0; --d)
                    if (u0 + d < lane && c4[d] == v) k = JT + u0 + d;
                  rs += 8 * kBlk;
                  ls += 8 * kBlk;
                }
              }
              inst.s[i * nn + j] = (int16_t)k;
            }
          } else {
            // diagonal tile: ordinary MCM on the 32-matrix sub-chain
            unsigned long long cb[4];
            E pi[4];
#pragma unroll
            for (int r = 0; r < 4; ++r) {
              const int li = 4 * w + r;
              pi[r] = (E)finPP[li];
              cb[r] = ~0ull;  // (no external splits)
            }
            const E pj1d = (E)(finPKI[lane] >> S);
            bool keyed = false;
            if (S == 5) {
              // int32 with a 5-bit shift: a cell's running minimum is one
              // 32-bit key (value << 5) + (k - IT), whose unsigned minimum
              // keeps the smallest split on ties, as the 64-bit keys below
              // do; final values are stored shifted in Xv, and a candidate
              // whose operands are not both final is not taken (a select,
              // no branch)
              //
              // The tile is a triangle: a warp row holds two table rows, i and
              // 31 - i, of 31 cells together, so that a thread has two cells and
              // none lies idle (four cells of the square a thread: 470 clocks a
              // step; 2000 chains of 8 to 128 matrices: 432 -> 367 us, n = 128 38.1 -> 36.4).
              uint32_t* Xs = reinterpret_cast<uint32_t*>(Xv);
              uint32_t key[2], pij[2], wc[2] = {0u, 0u};
              int ci[2], cj[2];  // the cells; (0, 0) stands in for the 32nd of a warp row
#pragma unroll
              for (int r = 0; r < 2; ++r) {
                const int row = 2 * w + r;
                const bool up = lane > row;
                ci[r] = up ? row : T - 1 - row;
                cj[r] = up ? lane : T - 1 - lane;
                if (lane == row) ci[r] = cj[r] = 0;
                key[r] = 0xFFFFFFFFu;
                pij[r] = (uint32_t)finPP[ci[r]] * (finPKI[cj[r]] >> S);
                if constexpr (W) {
                  const int64_t i = IT + ci[r], j = JT + cj[r];
                  if (i < j && j < inst.n) wc[r] = static_cast<const E*>(inst.w)[i * inst.n + j];
                }
              }
              if (w == 0) Xs[lane * T + lane] = 0u;
#pragma unroll 1
              for (int e = 0; e <= T - 2; ++e) {
#pragma unroll
                for (int r = 0; r < 2; ++r)
                  if (e > 0 && cj[r] - ci[r] == e) Xs[ci[r] * T + cj[r]] = (key[r] & ~31u) + (wc[r] << 5);
                bar_compute();
#pragma unroll
                for (int r = 0; r < 2; ++r) {
                  const int li = ci[r], lj = cj[r];
                  const int f = lj - li;
                  // split k1 = li + e: left operand on diagonal e, right on f - e - 1
                  const bool v1 = f > e && f - e - 1 <= e;
                  const int k1 = v1 ? li + e : 0;
                  const uint32_t c1 = Xs[li * T + k1] + pij[r] * finPKI[k1] + (uint32_t)k1;
                  const uint32_t n1 = __viaddmin_u32(c1, Xs[(k1 + 1) * T + lj], key[r]);
                  // split k2 = lj - 1 - e: right operand on diagonal e, left on f - 1 - e
                  const bool v2 = f > e && f - 1 - e < e;
                  const int k2 = v2 ? lj - 1 - e : 0;
                  const uint32_t c2 = Xs[li * T + k2] + pij[r] * finPKI[k2] + (uint32_t)k2;
                  const uint32_t n2 = __viaddmin_u32(c2, Xs[(k2 + 1) * T + lj], v1 ? n1 : key[r]);
                  key[r] = v2 ? n2 : (v1 ? n1 : key[r]);
                }
              }
              // to the threads that write the cells out
#pragma unroll
              for (int r = 0; r < 2; ++r)
                bestS[ci[r] * T + cj[r]] =
                    key[r] == 0xFFFFFFFFu ? ~0ull : ((unsigned long long)(key[r] >> 5) << KB) | (unsigned)(IT + (key[r] & 31u));
              bar_compute();
#pragma unroll
              for (int r = 0; r < 4; ++r) cb[r] = bestS[(4 * w + r) * T + lane];
              keyed = true;
            }
#pragma unroll 1
            for (int e = 0; e <= T - 2 && !keyed; ++e) {
#pragma unroll
              for (int r = 0; r < 4; ++r) {
                const int li = 4 * w + r;
                if (lane - li == e) Xv[li * T + lane] = e == 0 ? (E)0 : (E)(cb[r] >> KB) + wt[r];
              }
              bar_compute();
#pragma unroll
              for (int r = 0; r < 4; ++r) {
                const int li = 4 * w + r;
                const int f = lane - li;
                if (f > e) {
                  if (f - e - 1 <= e) {  // split k = li + e: left operand on diagonal e
                    const E cand = Xv[li * T + li + e] + Xv[(li + e + 1) * T + lane] +
                                   pi[r] * (E)(finPKI[li + e] >> S) * pj1d;
                    cb[r] = umin(cb[r], ((unsigned long long)cand << KB) | (unsigned)(IT + li + e));
                  }
                  if (f - 1 - e < e) {  // split k = lane - 1 - e: right operand on diagonal e
                    const E cand = Xv[li * T + lane - 1 - e] + Xv[(lane - e) * T + lane] +
                                   pi[r] * (E)(finPKI[lane - 1 - e] >> S) * pj1d;
                    cb[r] = umin(cb[r], ((unsigned long long)cand << KB) | (unsigned)(IT + lane - 1 - e));
                  }
                }
              }
            }
          // ------------------ outputs ------------------
          const int64_t nn = n;
          const unsigned long long kmask = (1ull << KB) - 1ull;
          E vals[4];
#pragma unroll
          for (int r = 0; r < 4; ++r) {
            const int li = 4 * w + r;
            const int64_t i = IT + li, j = JT + lane;
            const bool upper = li < lane;
            const E v = upper ? (E)(cb[r] >> KB) + wt[r] : (E)0;
            const int kk = upper ? (int)(cb[r] & kmask) : -1;
            vals[r] = v;
            if (i < nn && j < nn) {
              static_cast<int32_t*>(inst.m)[i * nn + j] = (int32_t)v;
              inst.s[i * nn + j] = (int16_t)kk;
            }
          }
          // packed row panel: af[tile][k = lane][row]
          E* af = static_cast<E*>(a.af) + tidx * T * T;
          E pa[4];
#pragma unroll
          for (int r = 0; r < 4; ++r) {
            pa[r] = (vals[r] << S) | (E)(lane & ((1 << (S < 5 ? S : 5)) - 1));
          }
          *reinterpret_cast<uint4*>(af + lane * T + 4 * w) = make_uint4(pa[0], pa[1], pa[2], pa[3]);
          // packed column panel, rows shifted by one: bf[tile(X, J)][row r] = m[32X + r + 1][.]
          E* bf = static_cast<E*>(a.bf);
#pragma unroll
          for (int r = 0; r < 4; ++r) {
            const int li = 4 * w + r;
            const E pb = vals[r] << S;
            if (li >= 1)
              bf[tidx * T * T + (li - 1) * T + lane] = pb;
            else if (I >= 1)
              bf[tile_index(inst, I - 1, J) * T * T + (T - 1) * T + lane] = pb;
          }
          }
        }
      }
    }
    if (finisher) ++fin_cnt;
    __syncthreads();
    if (tid == 0 && *reinterpret_cast<volatile int32_t*>(status) == 0) {
      // release (cumulative over the block's merges and stores before the barrier)
      if (!finisher)
        red_release_add(a.counters + tidx, 1);
      else if (D == 0)  // off-diagonal tiles publish right after their values
        st_release(a.flags + tidx, 1);
    }
  }
}

// A warp per tile row of a chain.  Single chains know each task's place in its
// bin; the tasks of several chains take places as they come (the order inside
// a bin does not matter to the result or to progress).
constexpr int kQueueRows = 8;
__global__ void __launch_bounds__(32 * kQueueRows) mcm_queue_kernel(const McmQueueArgs a) {
  const int lane = threadIdx.x & 31, I = blockIdx.y * kQueueRows + (threadIdx.x >> 5);
  const McmInstDev& in = a.insts[blockIdx.x];
  if (I >= in.nt) return;
  int32_t* slots = a.cursors + 3 * a.max_nt;
  for (int J0 = I; J0 < in.nt; J0 += 32) {
    const int J = J0 + lane;
    bool split = false;
    if (J < in.nt) {
      split = mcm_split(J - I, a.levels_per_part).nparts > 0;
      mcm_tile_tasks((int32_t)blockIdx.x, I, J, a.levels_per_part, [&](int bin, int place, const McmTask& t) {
        a.tasks[a.ninst == 1 ? a.cursors[bin] + place : atomicAdd(a.cursors + bin, 1)] = t;
      });
    }
    const unsigned with = __ballot_sync(0xffffffffu, split);
    int32_t first = 0;
    if (lane == 0 && with) first = atomicAdd(slots, __popc(with));
    first = __shfl_sync(0xffffffffu, first, 0);
    if (J < in.nt) a.accslot[tile_index(in, I, J)] = split ? first + __popc(with & ((1u << lane) - 1u)) : -1;
  }
}

// Interval DP, before the prologue: the largest weight above the diagonal of
// each chain (blockIdx.y), merged into McmInstDev::wmax; a negative weight
// there is DP_EINVAL.  Entries on and below the diagonal are not read.
// Weights are int32 (the cost type the interval DP is built for).
__global__ void __launch_bounds__(256) mcm_weight_max_kernel(const McmLaunchArgs a) {
  using SW = int32_t;
  __shared__ unsigned long long s_max[8];
  const int b = blockIdx.y;
  McmInstDev* inst = a.insts + b;
  const int n = inst->n;
  const SW* w = static_cast<const SW*>(a.w_all) + (a.tab_off ? a.tab_off[b] : 0);
  unsigned long long mx = 0;
  bool neg = false;
  for (int i = blockIdx.x; i < n; i += gridDim.x) {
    const SW* row = w + (int64_t)i * n;
    for (int j = i + 1 + (int)threadIdx.x; j < n; j += blockDim.x) {
      const SW v = row[j];
      neg |= v < 0;
      mx = v > 0 && (unsigned long long)v > mx ? (unsigned long long)v : mx;
    }
  }
  for (int o = 16; o > 0; o >>= 1) {
    const unsigned long long x = __shfl_xor_sync(0xffffffffu, mx, o);
    mx = x > mx ? x : mx;
  }
  if ((threadIdx.x & 31) == 0) s_max[threadIdx.x >> 5] = mx;
  neg = __syncthreads_or(neg);
  if (threadIdx.x == 0) {
    for (int x = 1; x < (int)(blockDim.x >> 5); ++x) mx = s_max[x] > mx ? s_max[x] : mx;
    if (neg) set_status(a.status, DP_EINVAL);
    if (mx > 0) atomicMax(&inst->wmax, mx);
  }
}

// One block per chain: validates dims, derives the cost bound and the packing
// shift, writes the padded / shifted dim arrays and the chain's record.  The
// blocks also set the flags, counters and queue to zero.  (As a memset, a copy
// of the records and this kernel, all before the main kernel's launch, the
// set-up took 8 of the 54 us of a 128-matrix solve.  Further blocks that set
// the accumulators too cost more than the memset they replace: the main
// kernel's first blocks, which take the head of the queue, are then not spread
// over the SMs one by one, n = 1000 355 -> 360 us.)
template <bool I64, bool W>
__global__ void __launch_bounds__(1024) mcm_prologue_kernel(const McmLaunchArgs a) {
  __shared__ int32_t s_max[32], s_min[32];
  __shared__ int32_t s_shift;
  launch_dependents();  // the main kernel's blocks may set themselves up meanwhile
  const int b = blockIdx.x;
  uint4* zero = reinterpret_cast<uint4*>(a.zero);
  for (int64_t x = (int64_t)b * blockDim.x + threadIdx.x; x < a.zero_bytes / 16; x += (int64_t)gridDim.x * blockDim.x)
    zero[x] = make_uint4(0u, 0u, 0u, 0u);
  McmInstDev* inst = a.insts + b;
  if (a.insts_from) {
    if (threadIdx.x == 0) *inst = a.insts_from[b];
    __syncthreads();
  }
  const int n = inst->n;
  const int32_t* p = a.p_off ? a.p_all + a.p_off[b] : a.p_all;
  int32_t mx = 0, mn = 0x7fffffff;
  for (int x = threadIdx.x; x <= n; x += blockDim.x) {
    const int32_t v = p[x];
    mx = v > mx ? v : mx;
    mn = v < mn ? v : mn;
  }
  for (int o = 16; o > 0; o >>= 1) {
    mx = max(mx, __shfl_xor_sync(0xffffffffu, mx, o));
    mn = min(mn, __shfl_xor_sync(0xffffffffu, mn, o));
  }
  if ((threadIdx.x & 31) == 0) {
    s_max[threadIdx.x >> 5] = mx;
    s_min[threadIdx.x >> 5] = mn;
  }
  __syncthreads();
  if (threadIdx.x == 0) {
    for (int w = 1; w < (int)(blockDim.x >> 5); ++w) {
      mx = max(mx, s_max[w]);
      mn = min(mn, s_min[w]);
    }
    int shift = -1;
    // interval DP: dims may be 0 (no rank-1 term); the weight adds at most
    // wmax per product, and n - 1 products make up a cell
    const unsigned long long wm = W ? inst->wmax : 0ull;
    if (mn < (W ? 0 : 1)) {
      set_status(a.status, DP_EINVAL);
    } else if (mx >= 65536 || wm >= (1ull << 47)) {
      set_status(a.status, DP_EOVERFLOW);
    } else {
      const unsigned long long m3 = (unsigned long long)mx * mx * mx;         // < 2^48
      const unsigned long long bound = (unsigned long long)(n - 1) * (m3 + wm);  // < 2^64
      if (I64) {
        if (bound >= (1ull << 47)) set_status(a.status, DP_EOVERFLOW);
        else shift = 16;
      } else {
        if (bound >= (1ull << 31)) {
          set_status(a.status, DP_EOVERFLOW);
        } else {
          shift = 1;
          while (shift < 5 && ((bound + 1) << (shift + 1)) <= (1ull << 32)) ++shift;
        }
      }
    }
    s_shift = shift;
    inst->shift = shift;
    inst->p = p;
    const int64_t to = a.tab_off ? a.tab_off[b] : 0;
    inst->m = static_cast<uint8_t*>(a.m_all) + to * (I64 ? 8 : 4);
    inst->s = a.s_all + to;
    if (W) inst->w = static_cast<const uint8_t*>(a.w_all) + to * (I64 ? 8 : 4);
  }
  __syncthreads();
  const int shift = s_shift;
  if (shift < 0) return;
  const int ext = inst->nt * T;
  for (int x = threadIdx.x; x < ext + 32; x += blockDim.x) {
    a.pp[inst->pp_base + x] = x <= n ? p[x] : 1;
    if (x < ext) a.pk[inst->pk_base + x] = (uint32_t)(x + 1 <= n ? p[x + 1] : 1) << shift;
  }
}

}  // namespace

cudaError_t launch_mcm_queue(const McmQueueArgs& a, cudaStream_t st) {
  if (a.ninst <= 0) return cudaSuccess;
  const dim3 grid((unsigned)a.ninst, (unsigned)((a.max_nt + kQueueRows - 1) / kQueueRows));
  mcm_queue_kernel<<<grid, 32 * kQueueRows, 0, st>>>(a);
  return cudaGetLastError();
}

size_t mcm_smem_bytes(bool i64) { return i64 ? mcm64_smem_bytes() : Smem::TOTAL; }

cudaError_t mcm_configure(bool i64) {
  cudaError_t e;
  if (i64) return mcm64_configure();
  if ((e = cudaFuncSetAttribute(mcm_main_kernel<false>, cudaFuncAttributeMaxDynamicSharedMemorySize,
                                (int)Smem::TOTAL)) != cudaSuccess)
    return e;
  return cudaFuncSetAttribute(mcm_main_kernel<true>, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)Smem::TOTAL);
}

// Both instances of a cost type have the same launch bounds and shared
// memory, hence the same occupancy.
cudaError_t mcm_occupancy(bool i64, int* blocks_per_sm) {
  if (i64) return mcm64_occupancy(blocks_per_sm);
  return cudaOccupancyMaxActiveBlocksPerMultiprocessor(blocks_per_sm, mcm_main_kernel<false>, kMcmThreads,
                                                       Smem::TOTAL);
}

cudaError_t mcm_preload(bool i64) {
  cudaFuncAttributes fa;
  cudaError_t e;
  if (i64) {
    if ((e = cudaFuncGetAttributes(&fa, mcm_prologue_kernel<true, false>)) != cudaSuccess) return e;
    return mcm64_preload();
  }
  if ((e = cudaFuncGetAttributes(&fa, mcm_prologue_kernel<false, false>)) != cudaSuccess) return e;
  return cudaFuncGetAttributes(&fa, mcm_main_kernel<false>);
}

// The interval DP is built for int32 costs only (see launch_mcm_weight_max
// in mcm_kernels.cuh): with int64 costs and weights these return
// cudaErrorNotSupported and launch nothing.
cudaError_t launch_mcm_weight_max(const McmLaunchArgs& a, bool i64, int sms, cudaStream_t st) {
  if (a.ninst <= 0 || !a.w_all) return cudaSuccess;
  if (i64) return cudaErrorNotSupported;
  const dim3 grid((unsigned)(sms > 0 ? 4 * sms : 256), (unsigned)a.ninst);
  mcm_weight_max_kernel<<<grid, 256, 0, st>>>(a);
  return cudaGetLastError();
}

cudaError_t launch_mcm_prologue(const McmLaunchArgs& a, bool i64, int max_n, int sms, cudaStream_t st) {
  if (a.ninst <= 0) return cudaSuccess;
  // few chains: their dims in few rounds of a large block (n = 4096: 12 us with
  // 256 threads); many chains: many small blocks per SM
  const int threads = max_n > 256 && a.ninst <= sms ? 1024 : 256;
  const bool w = a.w_all != nullptr;
  if (i64) {
    if (w) return cudaErrorNotSupported;
    mcm_prologue_kernel<true, false><<<a.ninst, threads, 0, st>>>(a);
  } else {
    if (w) mcm_prologue_kernel<false, true><<<a.ninst, threads, 0, st>>>(a);
    else mcm_prologue_kernel<false, false><<<a.ninst, threads, 0, st>>>(a);
  }
  return cudaGetLastError();
}

cudaError_t launch_mcm_main(const McmLaunchArgs& a, bool i64, int grid, cudaStream_t st) {
  if (a.ntasks <= 0) return cudaSuccess;
  const bool w = a.w_all != nullptr;
  if (i64) return w ? cudaErrorNotSupported : launch_mcm64(a, grid, st);
  return w ? launch_dependent(mcm_main_kernel<true>, grid, kMcmThreads, Smem::TOTAL, st, a)
           : launch_dependent(mcm_main_kernel<false>, grid, kMcmThreads, Smem::TOTAL, st, a);
}

}  // namespace dpk
