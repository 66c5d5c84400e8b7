// mcm_tile.cuh -- the in-tile solve of an off-diagonal tile (I, J) with int64
// costs (keys (m << 16) | k).
//
// X is the 32 x 32 tile; its in-tile splits are
//   column splits k = IT + r - 1, li < r <= 31:  U[li][r] + X[r][lj] + w
//   row splits    k = JT + u,     0 <= u < lj:   X[li][u] + L[u][lj] + w
// with U[li][r] = m[IT+li][IT+r-1] from the diagonal tile (I, I), L[u][lj] =
// m[JT+u+1][JT+lj] from (J, J) and w = p[IT+li] p[k+1] p[JT+lj+1].  The
// external splits and the boundary split k = IT + 31 are known before.
//
// The paper fills a table by diagonals (Figs. 5-7); here that order is applied
// twice.  The tile is cut into 4 x 4 blocks of 8 x 8 cells; block (a, c) (rows
// 8a.., columns 8c..) belongs to wave 3 - a + c, and the blocks of a wave
// depend only on earlier waves.  A warp owns two blocks of different waves
// (lane = cells (g, cc) and (g + 4, cc), g = lane / 8, cc = lane % 8):
//   * after the barrier that ends wave d it folds into its cells the splits
//     whose operand lies in the wave-d block of its block column (8 column
//     splits) and of its block row (8 row splits), read as 16-byte vectors;
//   * in its block's own wave it finishes the 15 cell diagonals of the block
//     among its own lanes: a cell that became final is passed on by shuffles,
//     and what each of the 8 in-block splits adds to it (U + w or L + w) was
//     put into registers before.
// What bounds it: 64-bit minima.  A split evaluation is a multiply-add and six
// instructions on the half-rate ALU pipe, so it pays to evaluate each split
// once: a wavefront over the whole tile, which evaluates two candidates of
// every cell at each of its 62 steps, finished or not, does 2.7 times as many.
//
// Tables of 32 x 32 entries in shared memory hold entry (row, x) at
// swz(row, x): the 16-byte granule of a row is exchanged by the row number, so
// that the same granule of 8 rows lies in distinct banks.  U and L come from
// global memory in this form (the diagonal tile writes them so, U by row with
// r mod 32, L by column).
#pragma once

#include <cstdint>

#include "dp_common.cuh"
#include "mcm_kernels.cuh"

namespace dpk {

using U64 = unsigned long long;

__host__ __device__ constexpr int swz(int row, int x) { return row * kTile + (((x >> 1) ^ (row & 7)) << 1 | (x & 1)); }

// Entries x0 .. x0 + 7 of a row (x0 a multiple of 8).
__device__ __forceinline__ void tile_ld8(const U64* tab, int row, int x0, U64 (&v)[8]) {
#pragma unroll
  for (int i = 0; i < 4; ++i) {
    const ulonglong2 q = *reinterpret_cast<const ulonglong2*>(tab + row * kTile + (((x0 / 2 + i) ^ (row & 7)) << 1));
    v[2 * i] = q.x, v[2 * i + 1] = q.y;
  }
}

__device__ __forceinline__ void tile_ldp(const uint32_t* p, uint32_t (&v)[8]) {
  const uint4 a = *reinterpret_cast<const uint4*>(p), b = *reinterpret_cast<const uint4*>(p + 4);
  v[0] = a.x, v[1] = a.y, v[2] = a.z, v[3] = a.w, v[4] = b.x, v[5] = b.y, v[6] = b.z, v[7] = b.w;
}

// m = min(m, c).  A 64-bit minimum is a compare and a select in two halves
// each, all on the ALU pipe, which bounds these kernels.  Written as
// predicated multiply-adds by `one` (1), which the compiler cannot turn back
// into selects, the halves move on the less loaded FMA pipe: the segment loop
// of 4 x 2 cells per thread 9.74 -> 10.64 split evaluations per clock and SM
// (alu_probe.cu), batches of chains 4077 -> 3617 us.
__device__ __forceinline__ void fold64(U64& m, U64 c, uint32_t one) {
  uint32_t ml = (uint32_t)m, mh = (uint32_t)(m >> 32);
  asm("{\n\t.reg .pred p;\n\t.reg .b64 a, b;\n\t"
      "mov.b64 a, {%2, %3};\n\tmov.b64 b, {%0, %1};\n\tsetp.lt.u64 p, a, b;\n\t"
      "@p mad.lo.u32 %0, %2, %4, 0;\n\t@p mad.lo.u32 %1, %3, %4, 0;\n\t}"
      : "+r"(ml), "+r"(mh)
      : "r"((uint32_t)c), "r"((uint32_t)(c >> 32)), "r"(one));
  m = ((U64)mh << 32) | ml;
}
// m = min(m, c) where cond holds, in the fewest dependent steps.
__device__ __forceinline__ void fold64_if(U64& m, U64 c, bool cond) {
  if (cond && c < m) m = c;
}

// v[t] = old v[(t - by) mod 8] for a lane-dependent by in [0, 8)
__device__ __forceinline__ void tile_rotate(U64 (&v)[8], int by) {
#pragma unroll
  for (int b = 1; b < 8; b *= 2) {
    const bool on = (by & b) != 0;
    U64 o[8];
#pragma unroll
    for (int t = 0; t < 8; ++t) o[t] = on ? v[(t - b) & 7] : v[t];
#pragma unroll
    for (int t = 0; t < 8; ++t) v[t] = o[t];
  }
}

// v[t] = old v[(t + by) mod 8] for a lane-dependent by in [0, 4)
__device__ __forceinline__ void tile_rotate_back4(U64 (&v)[8], int by) {
#pragma unroll
  for (int b = 1; b < 4; b *= 2) {
    const bool on = (by & b) != 0;
    U64 o[8];
#pragma unroll
    for (int t = 0; t < 8; ++t) o[t] = on ? v[(t + b) & 7] : v[t];
#pragma unroll
    for (int t = 0; t < 8; ++t) v[t] = o[t];
  }
}

// What a tile's solve reads and writes in shared memory.
struct TileTabs {
  const U64* U;        // key of U[li][r] at swz(li, r & 31); slot 0: the boundary column r = 32
  const U64* L;        // L[u][lj] with the row split's k at swz(lj, u)
  U64* Xr;             // X[li][lj] << 16 at swz(li, lj)
  U64* Xc;             // the same at swz(lj, li)
  const uint32_t* pr;  // pr[r] = p[IT + r] << 16
  const uint32_t* pu;  // pu[u] = p[JT + u + 1] << 16
  uint32_t one;        // for fold64
};

// The cells of one block that a lane computes.
struct TileCells {
  int li, lj;     // cells (li, lj) and (li + 4, lj) of the tile
  uint32_t w[2];  // p[IT+li] p[JT+lj+1]
  U64 m[2];       // running minima

  // the 8 column splits whose operand lies in block row a
  __device__ __forceinline__ void fold_col(const TileTabs& t, int a) {
    U64 x[8], u[8];
    uint32_t p[8];
    tile_ld8(t.Xc, lj, 8 * a, x);
    tile_ldp(t.pr + 8 * a, p);
#pragma unroll
    for (int q = 0; q < 2; ++q) {
      tile_ld8(t.U, li + 4 * q, 8 * a, u);
#pragma unroll
      for (int r = 0; r < 8; ++r) fold64(m[q], (U64)w[q] * p[r] + u[r] + x[r], t.one);
    }
  }
  // the 8 row splits whose operand lies in block column c
  __device__ __forceinline__ void fold_row(const TileTabs& t, int c) {
    U64 x[8], l[8];
    uint32_t p[8];
    tile_ld8(t.L, lj, 8 * c, l);
    tile_ldp(t.pu + 8 * c, p);
#pragma unroll
    for (int q = 0; q < 2; ++q) {
      tile_ld8(t.Xr, li + 4 * q, 8 * c, x);
#pragma unroll
      for (int u = 0; u < 8; ++u) fold64(m[q], (U64)w[q] * p[u] + l[u] + x[u], t.one);
    }
  }

  // In-block splits: bc[q][e mod 8] is what the column split met at cell
  // diagonal e adds to its operand (r = cc - e inside the block), br[q][e mod
  // 8] the same for the row split (u = i + e).
  __device__ __forceinline__ void bases(const TileTabs& t, int g, int cc, U64 (&bc)[2][8], U64 (&br)[2][8]) const {
    uint32_t p[8];
    U64 v[8];
    tile_ldp(t.pr + (li & ~7), p);
#pragma unroll
    for (int q = 0; q < 2; ++q) {
      tile_ld8(t.U, li + 4 * q, li & ~7, v);
#pragma unroll
      for (int r = 0; r < 8; ++r) bc[q][(8 - r) & 7] = (U64)w[q] * p[r] + v[r];  // at -r: rotated by cc
      tile_rotate(bc[q], cc);
    }
    tile_ldp(t.pu + (lj & ~7), p);
    tile_ld8(t.L, lj, lj & ~7, v);
#pragma unroll
    for (int q = 0; q < 2; ++q) {
#pragma unroll
      for (int u = 0; u < 8; ++u) br[q][(u - 4 * q) & 7] = (U64)w[q] * p[u] + v[u];  // at u - 4q: rotated back by g
      tile_rotate_back4(br[q], g);
    }
  }

  // The 15 cell diagonals of the block.
  __device__ __forceinline__ void solve(int g, int cc, const U64 (&bc)[2][8], const U64 (&br)[2][8]) {
    const int d = cc - g;  // the lane's cells lie on the block's cell diagonals d and d - 4
#pragma unroll
    for (int e = -7; e <= 6; ++e) {
      // the lane passes on the one of its cells that lies on diagonal e, if any
      const U64 x = (d == e ? m[0] : m[1]) & ~0xFFFFull;
      const U64 xc = __shfl_sync(0xffffffffu, x, (((cc - e) & 3) << 3) | cc);
      const U64 x0 = __shfl_sync(0xffffffffu, x, (g << 3) | ((g + e) & 7));
      const U64 x1 = __shfl_sync(0xffffffffu, x, (g << 3) | ((g + 4 + e) & 7));
      const bool up = e >= 0 || cc - e <= 7;  // the column operand's row r = cc - e is inside the block
      const bool l0 = e >= 0 || g + e >= 0, l1 = e >= -4 || g + 4 + e >= 0;
      fold64_if(m[0], bc[0][e & 7] + xc, d > e && up);
      fold64_if(m[1], bc[1][e & 7] + xc, d - 4 > e && up);
      fold64_if(m[0], br[0][e & 7] + x0, d > e && l0);
      fold64_if(m[1], br[1][e & 7] + x1, d - 4 > e && l1);
    }
  }
};

// Blocks (a, c) of warp w, first and second: one nibble per warp.  The waves
// of the pairs are (0,3) (1,3) (1,4) (2,4) (2,4) (2,5) (3,5) (3,6): at least
// two apart, so that what the second block missed while the first was being
// solved is folded in while other blocks of the wave between are solved, and
// every block of a wave has a warp of its own.
__device__ __forceinline__ int tile_block_a(int which, int w) {
  return ((which ? 0x01021010u : 0x32321323u) >> (4 * w)) & 15;
}
__device__ __forceinline__ int tile_block_c(int which, int w) {
  return ((which ? 0x33232110u : 0x32210100u) >> (4 * w)) & 15;
}
constexpr int kTileWaves = 7;

}  // namespace dpk
