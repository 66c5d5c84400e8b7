// sdp.cu -- sm_103a kernels for the simplified DP problem (paper Definition 1,
// Eq. (1)).  One thread block per instance; see sdp_kernels.cuh.
#include <cstdint>

#include "dp_common.cuh"
#include "sdp_kernels.cuh"

namespace dpk {

namespace {

template <int OP>
__device__ __forceinline__ uint32_t combine(uint32_t x, uint32_t y) {
  if constexpr (OP == 0) return x < y ? x : y;
  return x + y;  // wraps modulo 2^32
}

template <int OP>
__device__ __forceinline__ uint32_t combine3(uint32_t x, uint32_t y, uint32_t z) {
  if constexpr (OP == 0) return __vimin3_u32(x, y, z);
  return x + y + z;
}

// Barrier over the threads that compute cells (`count`, a multiple of 32).
__device__ __forceinline__ void bar_step(int count) { asm volatile("bar.sync 1, %0;" ::"r"(count) : "memory"); }

// Writes st[lo .. hi) with the values cls[x mod g] of the residue classes,
// as the part-th of nparts blocks.  Stores are 16 bytes wide where the table
// allows (lo and hi need no alignment).  Bound by the memory's write rate: a
// table of 2^26 cells (268 MB) takes 49 us in all, 5.5 TB/s, with the cells
// before the tail computed beside the fill (in 152 chunks it took 404 us);
// 200 tables of 4096 to 65536 cells in one launch 19 us (325 us step by step).
__device__ void fill_classes(uint32_t* st, int64_t lo, int64_t hi, const uint32_t* cls, int g, int part, int nparts) {
  const int64_t mis = (int64_t)((reinterpret_cast<uintptr_t>(st) >> 2) & 3);  // words past a 16-byte boundary
  int64_t v0 = (lo + mis + 3) >> 2, v1 = (hi + mis) >> 2;                     // whole vectors: words 4v - mis ..
  if (v1 < v0) v1 = v0;
  const int64_t head = v0 * 4 - mis < hi ? v0 * 4 - mis : hi;
  if (part == 0) {
    for (int64_t x = lo + threadIdx.x; x < head; x += blockDim.x) st[x] = cls[x % g];
    for (int64_t x = (v1 * 4 - mis > head ? v1 * 4 - mis : head) + threadIdx.x; x < hi; x += blockDim.x)
      st[x] = cls[x % g];
  }
  const int64_t stride = (int64_t)nparts * blockDim.x;
  int64_t v = v0 + (int64_t)part * blockDim.x + threadIdx.x;
  uint4* out = reinterpret_cast<uint4*>(st - mis);
  if (g == 1) {
    const uint32_t c = cls[0];
    const uint4 q = make_uint4(c, c, c, c);
#pragma unroll 4
    for (; v < v1; v += stride) out[v] = q;
    return;
  }
  const int adv = (int)((4 * stride) % g);
  int r = v < v1 ? (int)((4 * v - mis) % g) : 0;
  for (; v < v1; v += stride) {
    uint32_t c[4];
    int x = r;
#pragma unroll
    for (int i = 0; i < 4; ++i) {
      c[i] = cls[x];
      if (++x == g) x = 0;
    }
    out[v] = make_uint4(c[0], c[1], c[2], c[3]);
    r += adv;
    if (r >= g) r -= g;
  }
}

__device__ __forceinline__ uint32_t lds_u32(uint32_t addr) {
  uint32_t v;
  asm volatile("ld.shared.u32 %0, [%1];" : "=r"(v) : "r"(addr));
  return v;
}
__device__ __forceinline__ void sts_u32(uint32_t addr, uint32_t v) {
  asm volatile("st.shared.u32 [%0], %1;" ::"r"(addr), "r"(v) : "memory");
}

// RING = 0: read the table in global memory (window too large for shared memory).
// RING = 1: a ring of R = 2^ring_log2 words indexed modulo R.
// RING = 2: the same ring stored twice (word x at x and at x + R), so that the
//           read of ST[i - a_j] is ring[(i mod R) + R - a_j] with no wrap:
//           an add, a load and the operator per offset.
// KP: offsets held in registers (k <= KP); 0: offsets read from shared memory
//     (k > kSdpMaxKRegs).  G: loads in flight together.  FULL: k == KP (no
//     per-offset predicate).
//
// What bounds a step of W cells.  With many warps, shared-memory wavefronts:
// k W / 32 of reads and W / 16 of the two stores, one per clock (k = 32, W =
// 1024: 1088 of the 1290 clocks a step takes, data pipe 84 % busy, no bank
// conflicts).  With few, the latency of loads, combination, store and
// barrier.  Ring positions and displacements are byte addresses, so that a
// read is an add and a load: as word indices, which the compiler scales again
// at every read, a step took 1470 clocks.  Fewer loads in flight (G = 8
// against 16 or 32) drain more evenly when the pipe is the limit, more of them
// hide latency when it is not: k = 32, W = 64: 339, 296 and 280 clocks a step.
// Reading the next step's far offsets (a_j >= 2 W) before the barrier was
// slower at every size (W = 1024: 1750 clocks, W = 64: 385 against 225).
template <int OP, int RING, int KP, int G, bool FULL>
__global__ void __launch_bounds__(1024) sdp_kernel(const __grid_constant__ SdpLaunchArgs args) {
  extern __shared__ __align__(16) uint32_t sm[];
  constexpr uint32_t kIdentity = OP == 0 ? 0xFFFFFFFFu : 0u;
  const int tid = threadIdx.x;

  if ((int)blockIdx.x >= args.ninst) {
    // single table whose cells from one.tail_from - g on depend on their
    // residue class modulo g alone: this block fills its share of them with
    // the minima of the preset's classes while block 0 computes the rest
    const SdpInstDev in = args.one;
    const int g = in.g, A = args.one_offs[0];
    for (int c = tid; c < g; c += blockDim.x) sm[c] = 0xFFFFFFFFu;
    __syncthreads();
    if (g == 1) {
      uint32_t v = 0xFFFFFFFFu;
      for (int s = tid; s < A; s += blockDim.x) v = min(v, in.st[s]);
      v = __reduce_min_sync(0xFFFFFFFFu, v);
      if ((tid & 31) == 0) atomicMin(sm, v);
    } else {  // a stride that is a multiple of g where one fits: a thread stays in one class
      const int stride = g < (int)blockDim.x ? (int)blockDim.x / g * g : (int)blockDim.x;
      if (g <= (int)blockDim.x) {
        uint32_t v = 0xFFFFFFFFu;
        for (int s = tid; tid < stride && s < A; s += stride) v = min(v, in.st[s]);
        if (tid < stride) atomicMin(sm + tid % g, v);
      } else {
        for (int s = tid; s < A; s += stride) atomicMin(sm + s % g, in.st[s]);
      }
    }
    __syncthreads();
    fill_classes(in.st, in.tail_from, in.n, sm, g, (int)blockIdx.x - args.ninst, (int)gridDim.x - args.ninst);
    return;
  }

  SdpInstDev in = args.insts ? args.insts[blockIdx.x] : args.one;
  uint32_t* st = args.st_off ? args.st_all + args.st_off[blockIdx.x] : in.st;
  const int64_t n = in.tail_from > 0 ? in.tail_from : in.n;  // cells computed by the recurrence
  const int k = in.k;
  const int ring_log2 = args.ring_log2;
  const uint32_t R = RING ? (1u << ring_log2) : 0u;
  const uint32_t mask = R - 1u;
  uint32_t* ring = sm;
  const int32_t* a = args.insts ? in.a : args.one_offs;
  const int32_t a1 = a[0];
  const int32_t ak = a[k - 1];
  if (in.n <= a1) return;
  const int W = ak < (int)blockDim.x ? ak : (int)blockDim.x;
  const int nstep = (W + 31) & ~31;  // threads that take part in the steps (blockDim is a multiple of 32)
  // per-offset read displacement: -a_j words (table), -4 a_j bytes (masked
  // ring), 4 (R - a_j) bytes + the ring's address (mirrored ring)
  const uint32_t rb = smem_u32(ring), maskb = 4 * R - 1u;
  int32_t* disp = reinterpret_cast<int32_t*>(sm + (RING == 2 ? 2 * R : R));
  for (int j = tid; j < k; j += blockDim.x) disp[j] = RING == 2 ? 4 * ((int32_t)R - a[j]) + (int32_t)rb : (RING == 1 ? -4 * a[j] : -a[j]);
  if constexpr (RING != 0) {
    for (int x = tid; x < a1; x += blockDim.x) {
      const uint32_t v = st[x];
      ring[(uint32_t)x & mask] = v;
      if constexpr (RING == 2) ring[((uint32_t)x & mask) + R] = v;
    }
  }
  __syncthreads();
  if (tid < nstep) {
    constexpr int NR = KP > 0 ? KP : 1;
    int32_t ro[NR];
    if constexpr (KP > 0) {
#pragma unroll
      for (int j = 0; j < KP; ++j) ro[j] = disp[j < k ? j : 0];  // (min: reading a_1's term again changes nothing)
    }
    uint32_t pos = RING ? 4 * (((uint32_t)a1 + (uint32_t)tid) & mask) : 0u;  // 4 (i mod R) of the cell being computed
    uint32_t* cur = st + a1 + tid;                                           // its place in the table
    auto rd = [&](int32_t d) -> uint32_t {
      if constexpr (RING == 2) return lds_u32(pos + (uint32_t)d);
      if constexpr (RING == 1) return lds_u32(rb + ((pos + (uint32_t)d) & maskb));
      return cur[d];
    };
    auto cell = [&]() -> uint32_t {
      uint32_t v = kIdentity;
      if constexpr (KP > 0) {
#pragma unroll
        for (int q = 0; q < KP; q += G) {
          if (FULL || q < k) {
            uint32_t x[G];
#pragma unroll
            for (int i = 0; i < G; ++i) x[i] = (FULL || OP == 0 || q + i < k) ? rd(ro[q + i]) : kIdentity;
#pragma unroll
            for (int i = 0; i < G; i += 2) v = combine3<OP>(x[i], x[i + 1], v);
          }
        }
      } else {
        int j = 0;
        for (; j + G <= k; j += G) {
          uint32_t x[G];
#pragma unroll
          for (int i = 0; i < G; i += 4) {
            const int4 d = *reinterpret_cast<const int4*>(disp + j + i);
            x[i] = rd(d.x), x[i + 1] = rd(d.y), x[i + 2] = rd(d.z), x[i + 3] = rd(d.w);
          }
#pragma unroll
          for (int i = 0; i < G; i += 2) v = combine3<OP>(x[i], x[i + 1], v);
        }
        for (; j < k; ++j) v = combine<OP>(v, rd(disp[j]));
      }
      return v;
    };
    auto put = [&](uint32_t v) {
      if constexpr (RING != 0) {
        sts_u32(rb + pos, v);
        if constexpr (RING == 2) sts_u32(rb + 4 * R + pos, v);
      }
      *cur = v;
    };
    // Whole steps: threads from W up read with the others (their reads stay
    // inside the ring; off the ring they are kept from the table) and write
    // nothing.
    const bool active = tid < W;
    const bool all = nstep == (int)blockDim.x;
    const int64_t whole = (n - a1) / W;
    for (int64_t s = 0; s < whole; ++s) {
      if (RING != 0 || active) {
        const uint32_t v = cell();
        if (active) put(v);
      }
      pos = (pos + 4 * (uint32_t)W) & maskb;
      cur += W;
      if (all) __syncthreads();
      else bar_step(nstep);
    }
    if (tid < n - a1 - whole * W) put(cell());
  }
  if (in.tail_from > 0 && (int)gridDim.x == args.ninst) {
    // the rest of the table repeats its last g computed cells
    const int g = in.g;
    __syncthreads();
    uint32_t* cls = sm;
    for (int64_t x = n - g + tid; x < n; x += blockDim.x) cls[x % g] = st[x];
    __syncthreads();
    fill_classes(st, n, in.n, cls, g, 0, 1);
  }
}

template <int OP, int RING, int KP, int G, bool FULL>
cudaError_t launch_variant(const SdpLaunchArgs& a, size_t smem, cudaStream_t stream) {
  auto kern = sdp_kernel<OP, RING, KP, G, FULL>;
  cudaError_t e = cudaFuncSetAttribute(kern, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem);
  if (e != cudaSuccess) return e;
  kern<<<a.ninst + a.fill_blocks, a.threads, smem, stream>>>(a);
  return cudaGetLastError();
}

// The smallest register-resident variant that holds kmax offsets: in one of
// twice the size half the reads are predicated off but still issued (k = 16,
// W = 600: 1106 clocks a step in the 32-offset variant, 522 in its own).
template <int OP, int RING>
cudaError_t launch_k(const SdpLaunchArgs& a, int kmax, bool same_k, size_t smem, cudaStream_t stream) {
  // off the ring a read waits for L2, and 64-bit addresses leave no registers
  // for more offsets
  if (kmax > (RING == 0 ? 8 : kSdpMaxKRegs)) return launch_variant<OP, RING, 0, 8, false>(a, smem, stream);
  if constexpr (RING != 0) {
    if (kmax > 16) {
      if (!same_k || kmax < 32) return launch_variant<OP, RING, 32, 8, false>(a, smem, stream);
      // up to 8 warps the latency of the loads counts, above the pipe does
      return a.threads <= 256 ? launch_variant<OP, RING, 32, 32, true>(a, smem, stream)
                              : launch_variant<OP, RING, 32, 8, true>(a, smem, stream);
    }
    if (kmax > 8)
      return same_k && kmax == 16 ? launch_variant<OP, RING, 16, 8, true>(a, smem, stream)
                                  : launch_variant<OP, RING, 16, 8, false>(a, smem, stream);
  }
  if (kmax > 4) return launch_variant<OP, RING, 8, 8, false>(a, smem, stream);
  return launch_variant<OP, RING, 4, 4, false>(a, smem, stream);
}

template <int OP>
cudaError_t launch_op(const SdpLaunchArgs& a, int kmax, bool same_k, size_t smem, cudaStream_t stream) {
  const int mode = sdp_ring_mode(a.ring_log2);
  if (mode == 2) return launch_k<OP, 2>(a, kmax, same_k, smem, stream);
  if (mode == 1) return launch_k<OP, 1>(a, kmax, same_k, smem, stream);
  return launch_k<OP, 0>(a, kmax, same_k, smem, stream);
}

}  // namespace

int sdp_ring_mode(int ring_log2) {
  if (ring_log2 <= 0) return 0;
  return ring_log2 <= kSdpMirrorMaxLog2 ? 2 : 1;
}

size_t sdp_smem_bytes(int ring_log2, int kmax) {
  const int mode = sdp_ring_mode(ring_log2);
  const size_t ring = mode == 0 ? 0 : ((size_t)1 << ring_log2) * 4 * (mode == 2 ? 2 : 1);
  return ring + ((size_t)kmax * 4 + 31) / 32 * 32;
}

cudaError_t launch_sdp(const SdpLaunchArgs& a, cudaStream_t stream) {
  if (a.ninst <= 0) return cudaSuccess;
  // kmax: largest k in the launch (the host passes it through one.k for both
  // paths); same_k: every instance has that many offsets
  const int kmax = a.one.k;
  const bool same_k = a.same_k != 0;
  const size_t smem = sdp_smem_bytes(a.ring_log2, kmax);
  if (a.op == 0) return launch_op<0>(a, kmax, same_k, smem, stream);
  return launch_op<1>(a, kmax, same_k, smem, stream);
}

}  // namespace dpk
