// traceback.cu -- mcm_traceback: the optimal parenthesisation from the split
// table, on the device.
//
// The split table s defines a full binary tree over the chain: node (i, j),
// i < j, multiplies the product of matrices i..k by that of k+1..j, k =
// s[i][j] (Cormen et al., cited by the paper for the MCM recurrence).  The
// output lists the n-1 products in post-order, so every product comes after
// the two it consumes.  In post-order the products of the subtree (i, j)
// occupy j - i consecutive slots: its left subtree (i, k) the first k - i, its
// right subtree (k+1, j) the next j - k - 1, and (i, j) itself the last.  So
// each node knows its slot from its parent.
//
// What bounds it is latency: a node's children are known only after its split
// has come from memory, and a tree is often much deeper than log n (dims with
// many equal smallest entries, or that grow or fall along the chain, make it a
// comb).  Subtrees are handled by kind:
//   * a node is expanded by a thread, a level per pass;
//   * after three lopsided nodes in a row a path is followed: the larger child,
//     that one's larger child and so on.  The splits the path is likely to meet are loaded around the
//     node in one round trip -- column j (the path keeps to the right), row i
//     (to the left) and the corner of s next to (i, j) (it changes sides in
//     small steps) -- and then a hop costs a shared-memory read.  The block
//     loads for more than kMid matrices, a warp for fewer;
//   * at most kSmall matrices: a warp loads the subtree's triangle of s at
//     once and expands it in shared memory.
// n = 4096, dims in [1, 32] (a comb of about 100 products over subtrees of
// about 32 matrices): 153 us level by level, a round trip and two block
// barriers each; 62 us here.  Combs of 4000 products: 1.9 and 2.4 ms -> 0.26 ms,
// a random tree of 4000 (no long path): 31 -> 26 us.
#include <cuda_runtime.h>

#include <algorithm>
#include <cstdint>

#include "api_internal.h"
#include "dp_common.cuh"

namespace {

constexpr int kThreads = 1024;
constexpr int kWarps = kThreads / 32;
constexpr int kSmall = 32;      // subtrees of at most this many matrices are expanded whole
constexpr int kMid = 1024;      // paths from nodes of more are followed by the whole block
constexpr int kLopsided = 16;   // lopsided: the smaller child has less than 1/16 of the node's matrices
constexpr int kStreak = 3;      // a path is followed from the larger child of this many lopsided nodes in a row
constexpr int kMaxN = 32767;
constexpr int kMaxFront = kMaxN / (kSmall + 1) + 1;  // disjoint subtrees of more than kSmall matrices
static_assert(kMaxFront <= kThreads, "a thread per node of a pass");

struct __align__(8) Node {
  int16_t i, j;    // subtree (i, j), i < j
  int16_t base;    // its products start at this slot
  int16_t streak;  // lopsided ancestors in a row whose larger child this is
};
__device__ __forceinline__ Node node(int i, int j, int base, int streak) {
  return Node{(int16_t)i, (int16_t)j, (int16_t)base, (int16_t)streak};
}

// The splits loaded around a node (i, j): s[i + x][j], s[i][j - x] and
// s[i + x][j - y].
template <int LINE, int CORNER>
struct Window {
  static constexpr int kLine = LINE, kCorner = CORNER;
  static constexpr int kHops = 2 * LINE + 2 * CORNER;  // a path leaves the window after fewer
  int16_t col[LINE], row[LINE], corner[CORNER][CORNER];
  Node path[kHops + 1];
};
using BlockWindow = Window<4096, 64>;
using WarpWindow = Window<128, 16>;

// Working space of a small subtree, of a path, and of either in one block
// (never in use together).
struct WarpTri {
  int16_t s[kSmall][kSmall + 1];
  Node queue[kSmall];
};
union Work {
  BlockWindow block;
  WarpWindow warp[kWarps];
  WarpTri tri[kWarps];
};
struct Smem {
  Node front[2][kMaxFront];  // nodes of this pass and of the next, to be expanded ...
  Node lop[2][kMaxFront];    // ... and where a path starts
  int32_t nfront[2], nlop[2], nsmall, hops;
  Work work;
};

// Files a subtree of at least two matrices for the next pass, or for the end.
__device__ __forceinline__ void push(Smem& sm, int to, Node* small, int i, int j, int base, int streak) {
  if (i >= j) return;
  const Node nd = node(i, j, base, streak);
  if (j - i + 1 <= kSmall) small[atomicAdd(&sm.nsmall, 1)] = nd;
  else if (streak >= kStreak) sm.lop[to][atomicAdd(&sm.nlop[to], 1)] = nd;
  else sm.front[to][atomicAdd(&sm.nfront[to], 1)] = nd;
}

__device__ __forceinline__ void emit(int32_t* steps, int slot, int i, int k, int j) {
  steps[3 * slot + 0] = i;
  steps[3 * slot + 1] = k;
  steps[3 * slot + 2] = j;
}

// Loads the window of nd, by the COUNT threads of number t.
template <int COUNT, typename WIN>
__device__ __forceinline__ void load_window(const int16_t* s, int n, const Node& nd, int t, WIN& w) {
  constexpr int L = WIN::kLine / COUNT, C = WIN::kCorner * WIN::kCorner / COUNT;
  const int len = nd.j - nd.i;
  int16_t c[L], r[L], q[C];
#pragma unroll
  for (int u = 0; u < L; ++u) {
    const int x = t + u * COUNT;
    if (x < len) {
      c[u] = s[(int64_t)(nd.i + x) * n + nd.j];
      r[u] = s[(int64_t)nd.i * n + (nd.j - x)];
    }
  }
#pragma unroll
  for (int u = 0; u < C; ++u) {
    const int x = (t + u * COUNT) / WIN::kCorner, y = (t + u * COUNT) % WIN::kCorner;
    if (x + y < len) q[u] = s[(int64_t)(nd.i + x) * n + (nd.j - y)];
  }
#pragma unroll
  for (int u = 0; u < L; ++u) {
    const int x = t + u * COUNT;
    if (x < len) w.col[x] = c[u], w.row[x] = r[u];
  }
#pragma unroll
  for (int u = 0; u < C; ++u) {
    const int x = (t + u * COUNT) / WIN::kCorner, y = (t + u * COUNT) % WIN::kCorner;
    if (x + y < len) w.corner[x][y] = q[u];
  }
}

// Follows the path of larger children from nd through the window (one thread):
// path[0 .. hops) are its nodes, path[hops] the one after the last (perhaps a
// single matrix).  A split outside its subtree ends the path before its node;
// at the root that gives 0.
template <typename WIN>
__device__ int follow(const Node& nd, WIN& w) {
  const int i0 = nd.i, j0 = nd.j;
  int i = i0, j = j0, base = nd.base, hops = 0;
  Node* out = w.path;
  out[0] = nd;
  // one hop with split k; false where the path ends
  auto hop = [&](int k) -> bool {
    if (k < i || k >= j) return false;
    if (2 * k + 1 >= i + j) {  // the left child has at least as many matrices
      j = k;
    } else {
      base += k - i;
      i = k + 1;
    }
    out[++hops] = node(i, j, base, kStreak);
    return true;
  };
  bool on = true;
  while (on && i < j) {
    if (j == j0 && i - i0 < WIN::kLine) {  // column j: as long as the path keeps to the right
      while (on && i < j && j == j0 && i - i0 < WIN::kLine) on = hop(w.col[i - i0]);
    } else if (i == i0 && j0 - j < WIN::kLine) {
      while (on && i < j && i == i0 && j0 - j < WIN::kLine) on = hop(w.row[j0 - j]);
    } else if (i - i0 < WIN::kCorner && j0 - j < WIN::kCorner) {
      while (on && i < j && i - i0 < WIN::kCorner && j0 - j < WIN::kCorner) on = hop(w.corner[i - i0][j0 - j]);
    } else {
      on = false;
    }
  }
  return hops;
}

// Writes the path's products and files its smaller children and its end, by
// the `count` threads of number t.
__device__ void emit_path(Smem& sm, int to, Node* small, int32_t* steps, const Node* path, int hops, int t, int count) {
  for (int h = t; h < hops; h += count) {
    const Node a = path[h], b = path[h + 1];
    const bool right = b.j == a.j;
    const int k = right ? b.i - 1 : b.j;
    emit(steps, a.base + (a.j - a.i) - 1, a.i, k, a.j);
    if (right) push(sm, to, small, a.i, k, a.base, 0);
    else push(sm, to, small, k + 1, a.j, a.base + (k - a.i), 0);
    if (h + 1 == hops) push(sm, to, small, b.i, b.j, b.base, kStreak);
  }
}

// A warp expands a subtree of at most kSmall matrices, a level at a time.
__device__ void expand_small(const int16_t* s, int n, const Node& root, WarpTri& w, int32_t* steps, int32_t* status,
                             int lane) {
  const int m = root.j - root.i + 1;
  const int16_t* p = s + (int64_t)root.i * n + root.i;
  int16_t v[kSmall - 1];
#pragma unroll
  for (int r = 0; r < kSmall - 1; ++r)
    if (lane > r && lane < m) v[r] = p[(int64_t)r * n + lane];
#pragma unroll
  for (int r = 0; r < kSmall - 1; ++r)
    if (lane > r && lane < m) w.s[r][lane] = v[r];
  if (lane == 0) w.queue[0] = root;
  __syncwarp();
  int head = 0, tail = 1;  // at most m - 1 <= 31 nodes in all
  while (head < tail) {
    const int here = head + lane;
    bool l = false, r = false, bad = false;
    Node nd = node(0, 0, 0, 0);
    int k = 0;
    if (here < tail) {
      nd = w.queue[here];
      k = w.s[nd.i - root.i][nd.j - root.i];
      bad = k < nd.i || k >= nd.j;
      if (!bad) {
        emit(steps, nd.base + (nd.j - nd.i) - 1, nd.i, k, nd.j);
        l = k > nd.i;
        r = k + 1 < nd.j;
      }
    }
    const unsigned bl = __ballot_sync(0xffffffffu, l), br = __ballot_sync(0xffffffffu, r);
    const bool stop = __any_sync(0xffffffffu, bad);
    const unsigned below = (1u << lane) - 1u;
    if (stop) {
      if (bad) dpk::set_status(status, DP_EINVAL);
      return;
    }
    if (l) w.queue[tail + __popc(bl & below)] = node(nd.i, k, nd.base, 0);
    if (r) w.queue[tail + __popc(bl) + __popc(br & below)] = node(k + 1, nd.j, nd.base + (k - nd.i), 0);
    __syncwarp();
    head = tail;
    tail += __popc(bl) + __popc(br);
  }
}

// Expands everything but the small subtrees, which it lists in small[0 ..
// *count) for the kernel below, or (count == nullptr) expands in turn.
__global__ void __launch_bounds__(kThreads) traceback_kernel(const int16_t* __restrict__ s, int32_t n,
                                                             int32_t* __restrict__ steps, Node* small, int32_t* count,
                                                             int32_t* status) {
  extern __shared__ __align__(16) uint8_t raw[];
  Smem& sm = *reinterpret_cast<Smem*>(raw);
  const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31;
  dpk::launch_dependents();  // the kernel for the small subtrees
  if (tid == 0) {
    sm.nfront[0] = sm.nfront[1] = sm.nlop[0] = sm.nlop[1] = sm.nsmall = 0;
    push(sm, 0, small, 0, n - 1, 0, 0);
  }
  __syncthreads();
  // every pass writes at least one product, or reports a node and drops it
  for (int pass = 0; pass < n; ++pass) {
    const int cur = pass & 1, nxt = cur ^ 1;
    const int nfront = sm.nfront[cur], nlop = sm.nlop[cur];
    if (nfront + nlop == 0) break;
    // the split of this thread's node is on its way while the paths are followed
    Node mine = node(0, 0, 0, 0);
    int k = 0;
    if (tid < nfront) {
      mine = sm.front[cur][tid];
      k = s[(int64_t)mine.i * n + mine.j];
    }
    for (int x = warp; x < nlop; x += kWarps) {
      const Node nd = sm.lop[cur][x];
      if (nd.j - nd.i + 1 > kMid) continue;
      WarpWindow& w = sm.work.warp[warp];
      load_window<32>(s, n, nd, lane, w);
      __syncwarp();
      int hops = 0;
      if (lane == 0) {
        hops = follow(nd, w);
        if (hops == 0) dpk::set_status(status, DP_EINVAL);
      }
      hops = __shfl_sync(0xffffffffu, hops, 0);
      __syncwarp();
      emit_path(sm, nxt, small, steps, w.path, hops, lane, 32);
      __syncwarp();
    }
    if (tid < nfront) {
      if (k < mine.i || k >= mine.j) {  // not a split table of a solved chain
        dpk::set_status(status, DP_EINVAL);
      } else {
        const int l = k - mine.i + 1, r = mine.j - k;
        const int streak = min(l, r) * kLopsided < l + r ? mine.streak + 1 : 0;
        emit(steps, mine.base + (mine.j - mine.i) - 1, mine.i, k, mine.j);
        push(sm, nxt, small, mine.i, k, mine.base, l >= r ? streak : 0);
        push(sm, nxt, small, k + 1, mine.j, mine.base + (k - mine.i), l >= r ? 0 : streak);
      }
    }
    for (int x = 0; x < nlop; ++x) {
      const Node nd = sm.lop[cur][x];
      if (nd.j - nd.i + 1 <= kMid) continue;
      BlockWindow& w = sm.work.block;
      __syncthreads();  // the warps' windows, or the previous path, are done with
      load_window<kThreads>(s, n, nd, tid, w);
      __syncthreads();
      if (tid == 0) {
        sm.hops = follow(nd, w);
        if (sm.hops == 0) dpk::set_status(status, DP_EINVAL);
      }
      __syncthreads();
      emit_path(sm, nxt, small, steps, w.path, sm.hops, tid, kThreads);
    }
    __syncthreads();
    if (tid == 0) sm.nfront[cur] = sm.nlop[cur] = 0;
    __syncthreads();
  }
  if (count) {
    if (tid == 0) *count = sm.nsmall;
    return;
  }
  const int nsmall = sm.nsmall;
  for (int x = warp; x < nsmall; x += kWarps) {
    expand_small(s, n, small[x], sm.work.tri[warp], steps, status, lane);
    __syncwarp();
  }
}

// A warp per small subtree.
constexpr int kTriWarps = 4;
__global__ void __launch_bounds__(32 * kTriWarps) traceback_small_kernel(const int16_t* __restrict__ s, int32_t n,
                                                                         int32_t* __restrict__ steps,
                                                                         const Node* small, const int32_t* count,
                                                                         int32_t* status) {
  __shared__ WarpTri tri[kTriWarps];
  const int warp = threadIdx.x >> 5;
  dpk::grid_dependency_wait();  // the list
  const int total = *count;
  for (int x = blockIdx.x * kTriWarps + warp; x < total; x += gridDim.x * kTriWarps) {
    expand_small(s, n, small[x], tri[warp], steps, status, threadIdx.x & 31);
    __syncwarp();
  }
}

}  // namespace

cudaError_t dph::traceback_configure() {
  return cudaFuncSetAttribute(traceback_kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)sizeof(Smem));
}

extern "C" dp_status mcm_traceback(const int16_t* s, int32_t n, int32_t* steps, int32_t* status_dev, void* stream) {
  if (n < 1 || n > kMaxN) return dph::fail(DP_EINVAL, "mcm_traceback: n = %d outside [1, 32767]", n);
  if (n == 1) return DP_OK;  // a single matrix: no products (steps may be NULL)
  if (!s || !steps) return dph::fail(DP_EINVAL, "mcm_traceback: NULL pointer argument");
  dph::DevState* ds = nullptr;
  dp_status rc = dph::current_dev(&ds);
  if (rc != DP_OK) return rc;
  cudaStream_t st = static_cast<cudaStream_t>(stream);
  // the small subtrees: disjoint, of at least two matrices each
  Node* small = nullptr;
  cudaError_t e = cudaMallocAsync(reinterpret_cast<void**>(&small), (size_t)(n / 2 + 2) * sizeof(Node), st);
  if (e != cudaSuccess) return dph::fail_cuda(e, "mcm_traceback: subtree list");
  int32_t* count = reinterpret_cast<int32_t*>(small + n / 2 + 1);
  int32_t* status = status_dev ? status_dev : ds->status;
  // Up to 512 matrices there are at most a few small subtrees for each of the
  // block's warps, and a second launch costs more than it saves.  Above, they
  // are shared out over the SMs, about a warp each (2 n / kSmall in a random
  // tree; n = 4000: 57 -> 23 us), by blocks that are resident before the list is
  // complete: launched after it, a balanced tree of 600 to 1000 took 14.3 us,
  // 10.7 like this (a level at a time in one block: 11.3 to 12.4), a random one
  // of 800 20.3 and 18.0 (19.1).
  const bool one = n <= 512;
  traceback_kernel<<<1, kThreads, sizeof(Smem), st>>>(s, n, steps, small, one ? nullptr : count, status);
  e = cudaGetLastError();
  if (!one && e == cudaSuccess) {
    const int blocks = std::min(2 * ds->sms, n / (8 * kTriWarps) + 1);
    e = dpk::launch_early(traceback_small_kernel, dim3((unsigned)blocks), 32 * kTriWarps, st, s, n, steps, small, count,
                          status);
  }
  cudaError_t e2 = cudaFreeAsync(small, st);
  if (e != cudaSuccess) return dph::fail_cuda(e, "mcm_traceback: launch");
  if (e2 != cudaSuccess) return dph::fail_cuda(e2, "mcm_traceback: release");
  return DP_OK;
}
