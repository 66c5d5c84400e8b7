// mcm64.cu -- the main kernel of the int64-cost MCM solves (plain, batched,
// served).  Same decomposition, queue, panels and flags as the int32 kernel
// (mcm_kernels.cuh); a panel entry is (m << 16) | k, so one 64-bit minimum
// carries the cost and its smallest split through every stage, the in-tile
// wavefront included, and no cell's split is searched for afterwards.
//
// What bounds it.  A 64-bit split evaluation is one multiply-add and six
// instructions on the ALU pipe (add, compare and select in two halves each),
// of which the selects are predicated multiply-adds by one on the FMA pipe
// outside the in-tile solve, so the work of a tile is issue
// slots, and a single chain is bound by its tile-diagonals' hand-offs and
// wavefronts.  Batches of short chains are mostly finishers: one block of 256
// threads per tile and two of them per SM keep the ALUs fed while others
// wait at a barrier or for memory.  Two blocks leave 128 registers a thread,
// 127 of them used, with 64 bytes stored to and 48 loaded from local memory;
// three leave 80, and 492 and 660 bytes.
//
// A block needs nothing but plain copies: every flag a task waits for is
// polled by one lane of the first warp before the task starts (its other
// threads wait at the barrier and take no issue slots), the panels of its
// segments then arrive by cp.async into two stages.
#include <cstdint>

#include "dp_common.cuh"
#include "mcm_kernels.cuh"
#include "mcm_tile.cuh"

namespace dpk {

namespace {

constexpr int T = kTile;
constexpr int kThreads = 256;
constexpr int kBlocks = 2;                 // resident blocks per SM
constexpr U64 kInf = ~0ull;
constexpr U64 kValue = ~0xFFFFull;         // the shifted cost of a key
constexpr uint32_t kPollNs = 32;

struct __align__(128) Smem64 {
  union {
    U64 stage[2][2][T * T];                // [stage][row panel, column panel], k-major
    struct {
      U64 xr[T * T], xc[T * T];            // the tile's shifted costs by row and by column (swz)
    } x;
    U64 diag[T * T];                       // diagonal tiles: the tile's shifted costs
  };
  U64 u[T * T], l[T * T];                  // U of (I, I) and L of (J, J), see mcm_tile.cuh
  U64 best[T * T];
  int16_t ks[T * T];
  uint32_t pk[2][T];                       // p[k+1] << 16 of the staged segments
  uint32_t pi[T], pkj[T];                  // p[IT+t] << 16, p[JT+u+1] << 16
  int32_t task;
};

__device__ __forceinline__ int64_t tile_index(const McmInstDev& in, int I, int J) {
  return in.tile_base + (int64_t)I * in.nt - (int64_t)I * (I - 1) / 2 + (J - I);
}

__device__ __forceinline__ U64 umin64(U64 a, U64 b) { return a < b ? a : b; }

__device__ __forceinline__ void cp_async16(void* dst, const void* src) {
  asm volatile("cp.async.cg.shared.global [%0], [%1], 16;" ::"r"(smem_u32(dst)), "l"(src) : "memory");
}
__device__ __forceinline__ void cp_async_commit() { asm volatile("cp.async.commit_group;" ::: "memory"); }
template <int N>
__device__ __forceinline__ void cp_async_wait() {
  asm volatile("cp.async.wait_group %0;" ::"n"(N) : "memory");
}

// The external segments of a task: levels r_lo .. r_hi, segments I + r and
// J - r of each (one where they meet, which only the lowest level can).
struct Segments {
  int I, J, r_lo, one, count;
  __device__ __forceinline__ explicit Segments(const McmTask& t)
      : I(t.I), J(t.J), r_lo(t.r_lo), one(t.r_hi >= t.r_lo && 2 * t.r_lo == t.J - t.I),
        count(t.r_hi >= t.r_lo ? 2 * (t.r_hi - t.r_lo + 1) - one : 0) {}
  __device__ __forceinline__ int operator[](int x) const {
    const int y = x + (one && x >= 1);
    const int r = r_lo + (y >> 1);
    return (y & 1) ? J - r : I + r;
  }
};

__global__ void __launch_bounds__(kThreads, kBlocks) mcm64_kernel(const McmLaunchArgs a) {
  extern __shared__ __align__(128) uint8_t raw[];
  Smem64& sm = *reinterpret_cast<Smem64*>(raw);
  const int tid = threadIdx.x, w = tid >> 5, lane = tid & 31;
  // segment reductions: half the block takes the first 16 splits of every
  // segment, half the others; cells (4 ty + r, 2 tx + c) per thread
  const int half = tid >> 7, ty = (tid >> 4) & 7, tx = tid & 15;
  const U64* const af = static_cast<const U64*>(a.af);
  const U64* const bf = static_cast<const U64*>(a.bf);
  grid_dependency_wait();  // the set-up kernel's writes

  while (true) {
    if (tid == 0) {
      int32_t t = -1;
      if (*reinterpret_cast<volatile int32_t*>(a.status) == 0) t = atomicAdd(a.queue, 1);
      sm.task = t;
    }
    __syncthreads();
    const int32_t tix = sm.task;
    if (tix < 0 || tix >= a.ntasks) break;
    const McmTask task = a.tasks[tix];
    const McmInstDev inst = a.insts[task.inst];
    const int I = task.I, J = task.J, D = J - I, IT = I * T, JT = J * T;
    const int64_t tidx = tile_index(inst, I, J);
    const int32_t accslot = a.accslot[tidx];
    const bool finisher = task.kind == 0;
    const Segments seg(task);
    // an injected fault drops the task: its flag is never published
    bool ok = tix != a.drop_task;
    // every flag the task needs, one lane each: three tiles per segment; for a
    // finisher the diagonal tiles, the tile below and its bulk tasks
    if (w == 0 && ok) {
      const int nflags = 3 * seg.count + (finisher && D >= 1 ? 4 : 0);
      for (int f = lane; f < nflags; f += 32) {
        const int32_t* flag;
        int32_t target = 1;
        if (f < 3 * seg.count) {
          const int K = seg[f / 3], which = f % 3;
          flag = a.flags + (which == 0 ? tile_index(inst, I, K) : tile_index(inst, K + which - 1, J));
        } else {
          const int which = f - 3 * seg.count;
          if (which == 3) target = task.nparts;
          flag = which == 0   ? a.flags + tile_index(inst, I, I)
                 : which == 1 ? a.flags + tile_index(inst, J, J)
                 : which == 2 ? a.flags + tile_index(inst, I + 1, J)
                              : a.counters + tidx;
        }
        ok = ok && wait_flag_geq_cap<kPollNs>(flag, target, a.spin_limit, a.status);
      }
      __syncwarp();
    }
    if (!__syncthreads_and(ok)) continue;  // (a wait that ran out has set the status word: the next pop ends)

    // ---------------- external segments ----------------
    auto issue = [&](int q) {
      const int K = seg[q], st = q & 1;
      const U64* pa = af + tile_index(inst, I, K) * T * T;
      const U64* pb = bf + tile_index(inst, K, J) * T * T;
#pragma unroll
      for (int x = 0; x < 2; ++x) {
        const int at = 2 * (tid + x * kThreads);
        cp_async16(&sm.stage[st][0][at], pa + at);
        cp_async16(&sm.stage[st][1][at], pb + at);
      }
      if (tid < 8) cp_async16(&sm.pk[st][4 * tid], a.pk + inst.pk_base + (int64_t)K * T + 4 * tid);
      cp_async_commit();
    };
    U64 best[4][2];
#pragma unroll
    for (int r = 0; r < 4; ++r) best[r][0] = best[r][1] = kInf;
    U64 ext[2][2], brow0 = 0, brow1 = 0;  // finisher: bulk minima and boundary row of its blocks' cells
    uint32_t pI32 = 0;
    if (finisher && D >= 1) {
      const U64* pu = af + tile_index(inst, I, I) * T * T;
      const U64* pl = bf + tile_index(inst, J, J) * T * T;
#pragma unroll
      for (int x = 0; x < 2; ++x) {
        const int at = 2 * (tid + x * kThreads);
        cp_async16(&sm.u[at], pu + at);
        cp_async16(&sm.l[at], pl + at);
      }
      if (tid < 8) cp_async16(&sm.pkj[4 * tid], a.pk + inst.pk_base + JT + 4 * tid);
      cp_async_commit();
      if (tid < T) sm.pi[tid] = (uint32_t)a.pp[inst.pp_base + IT + tid] << 16;
      pI32 = a.pk[inst.pk_base + IT + T - 1];
      const U64* br = bf + tidx * T * T + (T - 1) * T;  // m[IT+32][.]
      brow0 = __ldcg(br + 8 * tile_block_c(0, w) + (lane & 7));
      brow1 = __ldcg(br + 8 * tile_block_c(1, w) + (lane & 7));
#pragma unroll
      for (int x = 0; x < 4; ++x) {
        const int li = 8 * tile_block_a(x >> 1, w) + (lane >> 3) + 4 * (x & 1), lj = 8 * tile_block_c(x >> 1, w) + (lane & 7);
        ext[x >> 1][x & 1] = task.nparts > 0 ? __ldcg(a.acc + (int64_t)accslot * T * T + li * T + lj) : kInf;
      }
    }
    if (seg.count > 0) {
      issue(0);
      uint32_t P[4][2];
#pragma unroll
      for (int r = 0; r < 4; ++r)
#pragma unroll
        for (int c = 0; c < 2; ++c)
          P[r][c] = (uint32_t)a.pp[inst.pp_base + IT + 4 * ty + r] * (uint32_t)a.pp[inst.pp_base + JT + 2 * tx + c + 1];
#pragma unroll 1
      for (int q = 0; q < seg.count; ++q) {
        if (q + 1 < seg.count) {
          issue(q + 1);
          cp_async_wait<1>();
        } else {
          cp_async_wait<0>();
        }
        __syncthreads();
        const U64* A = sm.stage[q & 1][0] + half * (T / 2) * T + 4 * ty;
        const U64* B = sm.stage[q & 1][1] + half * (T / 2) * T + 2 * tx;
        const uint32_t* pk = sm.pk[q & 1] + half * (T / 2);
#pragma unroll 4
        for (int k = 0; k < T / 2; ++k) {
          const ulonglong2 a01 = *reinterpret_cast<const ulonglong2*>(A + k * T);
          const ulonglong2 a23 = *reinterpret_cast<const ulonglong2*>(A + k * T + 2);
          const ulonglong2 bv = *reinterpret_cast<const ulonglong2*>(B + k * T);
          const U64 av[4] = {a01.x, a01.y, a23.x, a23.y};
          const uint32_t p = pk[k];
#pragma unroll
          for (int r = 0; r < 4; ++r) {
            fold64(best[r][0], (U64)P[r][0] * p + av[r] + bv.x, a.one);
            fold64(best[r][1], (U64)P[r][1] * p + av[r] + bv.y, a.one);
          }
        }
        __syncthreads();
      }
      // the two halves' minima; a finisher reads them from sm.best
      ulonglong2* const mine = reinterpret_cast<ulonglong2*>(&sm.best[4 * ty * T + 2 * tx]);
      if (half == 1) {
#pragma unroll
        for (int r = 0; r < 4; ++r) mine[r * (T / 2)] = make_ulonglong2(best[r][0], best[r][1]);
      }
      __syncthreads();
      if (half == 0) {
#pragma unroll
        for (int r = 0; r < 4; ++r) {
          const ulonglong2 o = mine[r * (T / 2)];
          best[r][0] = umin64(best[r][0], o.x);
          best[r][1] = umin64(best[r][1], o.y);
          if (finisher) {
            mine[r * (T / 2)] = make_ulonglong2(best[r][0], best[r][1]);
          } else {
            U64* acc = a.acc + (int64_t)accslot * T * T + (4 * ty + r) * T + 2 * tx;
            atomicMin(acc, best[r][0]);
            atomicMin(acc + 1, best[r][1]);
          }
        }
      }
    }
    if (!finisher) {
      __syncthreads();
      // release (cumulative over the block's merges before the barrier)
      if (tid == 0) red_release_add(a.counters + tidx, 1);
      continue;
    }

    // ---------------- finisher ----------------
    const int64_t n = inst.n;
    U64 out[4];  // final shifted costs of row 4w + r, column = lane
    if (D >= 1) {
      // the two blocks of 8 x 8 cells this warp owns (mcm_tile.cuh)
      const int g = lane >> 3, cc = lane & 7;
      cp_async_wait<0>();  // U, L and the dims, on their way since the task began
      __syncthreads();
      const TileTabs tab{sm.u, sm.l, sm.x.xr, sm.x.xc, sm.pi, sm.pkj, a.one};
      int passed = 0;  // waves whose barrier this warp has passed
#pragma unroll 1
      for (int sl = 0; sl < 2; ++sl) {
        const int ba = tile_block_a(sl, w), bk = tile_block_c(sl, w);
        TileCells cell;
        cell.li = 8 * ba + g;
        cell.lj = 8 * bk + cc;
#pragma unroll
        for (int q = 0; q < 2; ++q) {  // splits known before: the boundary IT + 31 and the external ones
          const int li = cell.li + 4 * q, x = li * T + cell.lj;
          cell.w[q] = (sm.pi[li] >> 16) * (sm.pkj[cell.lj] >> 16);
          cell.m[q] = sm.u[swz(li, 0)] + (sl ? brow1 : brow0) + (U64)cell.w[q] * pI32;
          if (seg.count > 0) cell.m[q] = umin64(cell.m[q], sm.best[x]);
          cell.m[q] = umin64(cell.m[q], sl ? ext[1][q] : ext[0][q]);
        }
        U64 bc[2][8], br[2][8];
        cell.bases(tab, g, cc, bc, br);
        const int wave = 3 - ba + bk;
#pragma unroll 1
        for (int d = 0; d < wave; ++d) {
          if (d >= passed) {
            __syncthreads();
            ++passed;
          }
          if (d >= bk) cell.fold_col(tab, 3 - d + bk);
          if (d >= 3 - ba) cell.fold_row(tab, d - 3 + ba);
        }
        cell.solve(g, cc, bc, br);
#pragma unroll
        for (int q = 0; q < 2; ++q) {
          const int li = cell.li + 4 * q;
          sm.x.xr[swz(li, cell.lj)] = cell.m[q] & kValue;
          sm.x.xc[swz(cell.lj, li)] = cell.m[q] & kValue;
          sm.ks[li * T + cell.lj] = (int16_t)(cell.m[q] & 0xFFFF);
        }
        // arrive before the second block's folds: other warps wait for this one
        __syncthreads();
        ++passed;
      }
      for (; passed < kTileWaves; ++passed) __syncthreads();
#pragma unroll
      for (int r = 0; r < 4; ++r) out[r] = sm.x.xr[swz(4 * w + r, lane)];
    } else {
      // diagonal tile: an ordinary chain of 32 matrices, one cell diagonal per
      // step; warp w owns rows 4w .. 4w+3, lane = column
      U64 m[4];
      uint32_t wv[4];
      const uint32_t pj1 = (uint32_t)a.pp[inst.pp_base + JT + lane + 1];
      if (tid < T) sm.pkj[tid] = a.pk[inst.pk_base + JT + tid];
#pragma unroll
      for (int r = 0; r < 4; ++r) {
        m[r] = kInf;
        wv[r] = (uint32_t)a.pp[inst.pp_base + IT + 4 * w + r] * pj1;
      }
#pragma unroll 1
      for (int e = 0; e <= T - 2; ++e) {
#pragma unroll
        for (int r = 0; r < 4; ++r) {
          const int li = 4 * w + r;
          if (lane - li == e) sm.diag[li * T + lane] = e == 0 ? 0 : m[r] & kValue;
        }
        __syncthreads();
#pragma unroll
        for (int r = 0; r < 4; ++r) {
          const int li = 4 * w + r, f = lane - li;
          // split li + e (left operand on diagonal e) and split lane - 1 - e
          // (right operand on diagonal e), where the other operand is final too
          const bool v1 = f > e && f - e - 1 <= e, v2 = f > e && f - 1 - e < e;
          const int k1 = v1 ? li + e : 0, k2 = v2 ? lane - 1 - e : 0;
          const U64 c1 = sm.diag[li * T + k1] + sm.diag[(k1 + 1) * T + lane] + (U64)wv[r] * sm.pkj[k1] + (U64)(IT + k1);
          const U64 c2 = sm.diag[li * T + k2] + sm.diag[(k2 + 1) * T + lane] + (U64)wv[r] * sm.pkj[k2] + (U64)(IT + k2);
          if (v1) m[r] = umin64(m[r], c1);
          if (v2) m[r] = umin64(m[r], c2);
        }
      }
#pragma unroll
      for (int r = 0; r < 4; ++r) {
        const bool upper = 4 * w + r < lane;
        out[r] = upper ? m[r] & kValue : 0;
        sm.ks[(4 * w + r) * T + lane] = upper ? (int16_t)(m[r] & 0xFFFF) : (int16_t)-1;  // read by this thread only
      }
    }
    // ---------------- panels needed by other tiles, then publish ----------------
    {
      U64* pa = static_cast<U64*>(a.af) + tidx * T * T;
      U64* pb = static_cast<U64*>(a.bf) + tidx * T * T;
      const U64 k = (U64)(JT + lane);
      if (D >= 1) {
        *reinterpret_cast<ulonglong2*>(pa + lane * T + 4 * w) = make_ulonglong2(out[0] | k, out[1] | k);
        *reinterpret_cast<ulonglong2*>(pa + lane * T + 4 * w + 2) = make_ulonglong2(out[2] | k, out[3] | k);
      }
#pragma unroll
      for (int r = 0; r < 4; ++r) {
        const int li = 4 * w + r;
        if (D == 0) pa[swz(li, (lane + 1) & 31)] = out[r] | k;  // U and L of the tiles that read this one
        if (li >= 1) pb[D >= 1 ? (li - 1) * T + lane : swz(lane, li - 1)] = D >= 1 ? out[r] : out[r] | (U64)(JT + li - 1);
        else if (I >= 1) static_cast<U64*>(a.bf)[tile_index(inst, I - 1, J) * T * T + (T - 1) * T + lane] = out[r];
      }
    }
    __syncthreads();
    // release: the panel stores of every thread, ordered before this store by
    // the barrier, are visible to whoever acquires the flag
    if (tid == 0) st_release(a.flags + tidx, 1);
    // ---------------- the tables themselves (not read by other tiles) ----------------
    int64_t* mt = static_cast<int64_t*>(inst.m);
#pragma unroll
    for (int r = 0; r < 4; ++r) {
      const int li = 4 * w + r;
      const int64_t i = IT + li, j = JT + lane;
      if (i < n && j < n) {
        mt[i * n + j] = (int64_t)(out[r] >> 16);
        inst.s[i * n + j] = sm.ks[li * T + lane];
      }
      const int64_t i2 = JT + li, j2 = IT + lane;  // mirror tile (J, I)
      if (D >= 1 && i2 < n && j2 < n) {
        mt[i2 * n + j2] = 0;
        inst.s[i2 * n + j2] = -1;
      }
    }
  }
}

}  // namespace

size_t mcm64_smem_bytes() { return sizeof(Smem64); }

cudaError_t mcm64_configure() {
  return cudaFuncSetAttribute(mcm64_kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)sizeof(Smem64));
}

cudaError_t mcm64_occupancy(int* blocks_per_sm) {
  return cudaOccupancyMaxActiveBlocksPerMultiprocessor(blocks_per_sm, mcm64_kernel, kThreads, sizeof(Smem64));
}

cudaError_t mcm64_preload() {
  cudaFuncAttributes fa;
  return cudaFuncGetAttributes(&fa, mcm64_kernel);
}

cudaError_t launch_mcm64(const McmLaunchArgs& a, int grid, cudaStream_t st) {
  return launch_dependent(mcm64_kernel, grid, kThreads, sizeof(Smem64), st, a);
}

}  // namespace dpk
