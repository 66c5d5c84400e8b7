// sdp_ntt.cu -- see sdp_ntt.cuh.
#include "sdp_ntt.cuh"

namespace dpk {
namespace {

constexpr int N = kNttN;
constexpr int kThreads = 1024;  // 16 words per thread
constexpr int kPrimes = 3;
// primes c 2^23 + 1 (and higher powers of 2) below 2^30, each with 3 as a primitive root
__host__ __device__ constexpr uint32_t prime(int i) { return i == 0 ? 998244353u : i == 1 ? 167772161u : 469762049u; }
__host__ __device__ constexpr uint32_t mul_mod(uint32_t a, uint32_t b, uint32_t p) {
  return (uint32_t)((uint64_t)a * b % p);
}
__host__ __device__ constexpr uint32_t pow_mod(uint32_t a, uint32_t e, uint32_t p) {
  uint32_t r = 1;
  for (; e; e >>= 1, a = mul_mod(a, a, p))
    if (e & 1) r = mul_mod(r, a, p);
  return r;
}
__host__ __device__ constexpr uint32_t inv_mod(uint32_t a, uint32_t p) { return pow_mod(a % p, p - 2, p); }
// -p^-1 mod 2^32 (Newton's iteration)
__host__ __device__ constexpr uint32_t neg_inv32(uint32_t p) {
  uint32_t x = p;
  for (int i = 0; i < 5; ++i) x *= 2u - p * x;
  return 0u - x;
}
__host__ __device__ constexpr uint32_t quotient(uint32_t w, uint32_t p) { return (uint32_t)(((uint64_t)w << 32) / p); }

struct PrimeConsts {
  uint32_t p, np;         // the prime, -p^-1 mod 2^32
  uint32_t one;           // quotient(1)
  uint32_t mont1, rootm;  // 2^32 and 2^32 times a root of order N
  uint32_t scale, scaleq; // 2^32 / N: undoes a Montgomery factor and two transforms
};
constexpr PrimeConsts consts(uint32_t p) {
  const uint32_t scale = mul_mod((uint32_t)((1ull << 32) % p), inv_mod(kNttN, p), p);
  return PrimeConsts{p, neg_inv32(p), quotient(1, p), (uint32_t)((1ull << 32) % p),
                     mul_mod((uint32_t)((1ull << 32) % p), pow_mod(3, (p - 1) / kNttN, p), p), scale, quotient(scale, p)};
}
__constant__ const PrimeConsts kConsts[kPrimes] = {consts(prime(0)), consts(prime(1)), consts(prime(2))};

// All values are kept below 2p < 2^31.
__device__ __forceinline__ uint32_t below(uint32_t x, uint32_t m) { return min(x, x - m); }  // x < 2m -> x mod m
// x w mod p, below 2p, for any 32-bit x; q = quotient(w, p)
__device__ __forceinline__ uint32_t mul_const(uint32_t x, uint32_t w, uint32_t q, uint32_t p) {
  return x * w - __umulhi(x, q) * p;
}
// a b 2^-32 mod p, below 2p (Montgomery), for a b < 2^32 p
__device__ __forceinline__ uint32_t mul_redc(uint32_t a, uint32_t b, uint32_t p, uint32_t np) {
  const uint64_t t = (uint64_t)a * b;
  return (uint32_t)((t + (uint64_t)((uint32_t)t * np) * p) >> 32);
}

// tables, per prime and direction (forward, inverse): N words 2^32 w, those of
// the level with butterflies at distance h at h + j, w = root_{2h}^j, j < h.
__global__ void __launch_bounds__(256) ntt_table_kernel(uint32_t* tables) {
  const int at = blockIdx.x * blockDim.x + threadIdx.x, pi = blockIdx.y >> 1, inverse = blockIdx.y & 1;
  if (at == 0) return;
  const PrimeConsts c = kConsts[pi];
  const int h = 1 << (31 - __clz(at));
  uint32_t e = (uint32_t)(at - h) * (uint32_t)(N / 2 / h);  // w = root_N^e
  if (inverse) e = N - e;
  // Montgomery powers: r = root^e 2^32
  uint32_t r = c.mont1, b = c.rootm;
  for (; e; e >>= 1, b = mul_redc(b, b, c.p, c.np))
    if (e & 1) r = mul_redc(r, b, c.p, c.np);
  tables[(size_t)(pi * 2 + inverse) * N + at] = below(r, c.p);
}

// Shared-memory place of word i: a word of padding every 16 keeps the passes
// of strides 16 and 1 free of bank conflicts.  In those of strides 4096 and 256
// a warp touches 32 neighbouring words, of which the first and the last then
// share a bank: two wavefronts for what could be one.
__device__ __forceinline__ int place(int i) { return i + (i >> 4); }
constexpr int kSmemWords = N + N / 16;
// Twiddles of the levels up to distance 2048 follow the words in shared memory
// (those of the two larger ones are used once, and read from global memory
// along with the data): read through L1 at every butterfly they made a
// transform 24 us, 15 like this (13 of them multiplications and exchanges).
constexpr int kSmemTwiddles = 4096;
constexpr int kSmemBytes = (kSmemWords + kSmemTwiddles) * 4;

static_assert(kSmemTwiddles == 4 * kThreads, "16 bytes per thread");
__device__ __forceinline__ const uint32_t* stage_twiddles(uint32_t* sm, const uint32_t* tw) {
  reinterpret_cast<uint4*>(sm + kSmemWords)[threadIdx.x] = __ldg(reinterpret_cast<const uint4*>(tw) + threadIdx.x);
  return sm + kSmemWords;
}

// The butterflies of 2^LOGR words at distance `stride`, offset j < stride;
// forward: from the largest distance down (decimation in frequency), inverse:
// from the smallest up (decimation in time).
template <int LOGR, bool INVERSE>
__device__ __forceinline__ void butterflies(uint32_t (&v)[1 << LOGR], int j, int stride, const uint32_t* tw,
                                            uint32_t p, uint32_t np) {
  constexpr int R = 1 << LOGR;
  const uint32_t p2 = 2 * p;
#pragma unroll
  for (int l = 0; l < LOGR; ++l) {
    const int half = INVERSE ? 1 << l : R >> (l + 1);
#pragma unroll
    for (int k = 0; k < R; ++k) {
      if (k & half) continue;
      const uint32_t w = tw[stride * half + j + stride * (k & (half - 1))];
      uint32_t& a = v[k];
      uint32_t& b = v[k + half];
      if constexpr (INVERSE) {
        const uint32_t t = mul_redc(b, w, p, np), s = a + t, d = a + (p2 - t);
        a = below(s, p2);
        b = below(d, p2);
      } else {
        const uint32_t s = a + b, d = a + (p2 - b);
        a = below(s, p2);
        b = mul_redc(d, w, p, np);
      }
    }
  }
}

// Words (first + k stride), k < 16, from / to shared memory around their butterflies.
template <bool INVERSE>
__device__ __forceinline__ void pass16(uint32_t* sm, int first, int j, int stride, const uint32_t* tw, uint32_t p,
                                       uint32_t np) {
  uint32_t v[16];
#pragma unroll
  for (int k = 0; k < 16; ++k) v[k] = sm[place(first + k * stride)];
  butterflies<4, INVERSE>(v, j, stride, tw, p, np);
#pragma unroll
  for (int k = 0; k < 16; ++k) sm[place(first + k * stride)] = v[k];
}

// One row modulo one prime per block.  A transform is three round trips
// through shared memory; 14 N / 2 butterflies of about 7 instructions bound it
// (about 13 us per block of 1024 threads).
__global__ void __launch_bounds__(kThreads) ntt_forward_kernel(const uint32_t* tables, const NttRows u, uint32_t* spec_u,
                                                               const NttRows z, uint32_t* spec_z) {
  extern __shared__ __align__(16) uint32_t sm[];
  const bool is_u = (int)blockIdx.x < u.rows;
  const NttRows in = is_u ? u : z;
  const int tid = threadIdx.x, row = is_u ? blockIdx.x : blockIdx.x - u.rows, pi = blockIdx.y;
  const uint32_t p = kConsts[pi].p, np = kConsts[pi].np, one = kConsts[pi].one;
  const uint32_t* tw = tables + (size_t)(pi * 2) * N;
  const uint32_t* tws = stage_twiddles(sm, tw);
  const int64_t at = (int64_t)row * in.pitch;
  const int64_t len = in.len < in.limit - at ? in.len : in.limit - at;
  const uint32_t* src = in.src + at;
#pragma unroll
  for (int m = 0; m < 4; ++m) {
    const int j = tid + kThreads * m;
    uint32_t v[4];
#pragma unroll
    for (int k = 0; k < 4; ++k) {
      const int64_t i = in.reverse ? in.len - 1 - (j + 4096 * k) : j + 4096 * k;
      v[k] = mul_const(i >= 0 && i < len ? src[i] : 0u, 1u, one, p);
    }
    butterflies<2, false>(v, j, 4096, tw, p, np);
#pragma unroll
    for (int k = 0; k < 4; ++k) sm[place(j + 4096 * k)] = v[k];
  }
  __syncthreads();
  pass16<false>(sm, (tid >> 8) * 4096 + (tid & 255), tid & 255, 256, tws, p, np);
  __syncthreads();
  pass16<false>(sm, (tid >> 4) * 256 + (tid & 15), tid & 15, 16, tws, p, np);
  __syncthreads();
  uint32_t v[16];
#pragma unroll
  for (int k = 0; k < 16; ++k) v[k] = sm[place(16 * tid + k)];
  butterflies<4, false>(v, 0, 1, tws, p, np);
  uint4* out = reinterpret_cast<uint4*>((is_u ? spec_u : spec_z) + ((int64_t)pi * in.rows + row) * N + 16 * tid);
#pragma unroll
  for (int k = 0; k < 4; ++k) out[k] = make_uint4(v[4 * k], v[4 * k + 1], v[4 * k + 2], v[4 * k + 3]);
}

// Point-wise product of spectra u[lo] and z[hi] and its inverse transform: the
// residues of outputs A - 1 + t, t < A.
__global__ void __launch_bounds__(kThreads) ntt_window_kernel(const uint32_t* tables, const uint32_t* u, int nlo,
                                                              const uint32_t* z, int nhi, int A, uint32_t* residues) {
  extern __shared__ __align__(16) uint32_t sm[];
  const int tid = threadIdx.x, pair = blockIdx.x, pi = blockIdx.y;
  const uint32_t p = kConsts[pi].p, np = kConsts[pi].np;
  const uint32_t* tw = tables + (size_t)(pi * 2 + 1) * N;
  const uint32_t* tws = stage_twiddles(sm, tw);
  const int hi = pair / nlo, lo = pair % nlo;
  const uint4* us = reinterpret_cast<const uint4*>(u + ((int64_t)pi * nlo + lo) * N + 16 * tid);
  const uint4* zs = reinterpret_cast<const uint4*>(z + ((int64_t)pi * nhi + hi) * N + 16 * tid);
  uint32_t v[16];
#pragma unroll
  for (int k = 0; k < 4; ++k) {
    const uint4 a = us[k], b = zs[k];
    v[4 * k] = mul_redc(a.x, b.x, p, np);
    v[4 * k + 1] = mul_redc(a.y, b.y, p, np);
    v[4 * k + 2] = mul_redc(a.z, b.z, p, np);
    v[4 * k + 3] = mul_redc(a.w, b.w, p, np);
  }
  __syncthreads();
  butterflies<4, true>(v, 0, 1, tws, p, np);
#pragma unroll
  for (int k = 0; k < 16; ++k) sm[place(16 * tid + k)] = v[k];
  __syncthreads();
  pass16<true>(sm, (tid >> 4) * 256 + (tid & 15), tid & 15, 16, tws, p, np);
  __syncthreads();
  pass16<true>(sm, (tid >> 8) * 4096 + (tid & 255), tid & 255, 256, tws, p, np);
  __syncthreads();
  const uint32_t scale = kConsts[pi].scale, sq = kConsts[pi].scaleq;
  uint32_t* out = residues + ((int64_t)pi * gridDim.x + pair) * A;
#pragma unroll
  for (int m = 0; m < 4; ++m) {
    const int j = tid + kThreads * m;
    uint32_t c[4];
#pragma unroll
    for (int k = 0; k < 4; ++k) c[k] = sm[place(j + 4096 * k)];
    butterflies<2, true>(c, j, 4096, tw, p, np);
#pragma unroll
    for (int k = 0; k < 4; ++k) {
      const int t = j + 4096 * k - (A - 1);
      if (t >= 0 && t < A) out[t] = below(mul_const(c[k], scale, sq, p), p);
    }
  }
}

// The outputs from their residues (Garner), modulo 2^32.
__global__ void __launch_bounds__(256) ntt_place_kernel(const uint32_t* residues, int nlo, int A, int64_t pairs,
                                                        uint32_t* out, int64_t pitch_hi, int64_t pitch_lo,
                                                        int64_t limit) {
  const int t = blockIdx.x * blockDim.x + threadIdx.x, pair = blockIdx.y;
  if (t >= A) return;
  constexpr uint32_t p0 = prime(0), p1 = prime(1), p2 = prime(2);
  constexpr uint32_t i01 = inv_mod(p0 % p1, p1), q01 = quotient(i01, p1);
  constexpr uint32_t i012 = inv_mod(mul_mod(p0 % p2, p1 % p2, p2), p2), q012 = quotient(i012, p2);
  constexpr uint32_t p0in2 = p0 % p2, qp0in2 = quotient(p0in2, p2);
  const uint32_t r0 = residues[(int64_t)pair * A + t], r1 = residues[(pairs + pair) * A + t],
                 r2 = residues[(2 * pairs + pair) * A + t];
  // value = r0 + p0 k1 + p0 p1 k2
  const uint32_t k1 = below(mul_const(r1 + (p0 / p1 + 1) * p1 - r0, i01, q01, p1), p1);
  const uint32_t v = below(mul_const(k1, p0in2, qp0in2, p2), p2);  // p0 k1 mod p2
  const uint32_t k2 = below(mul_const(r2 + (p0 / p2 + 1) * p2 - r0 + (p2 - v), i012, q012, p2), p2);
  const int64_t at = (int64_t)(pair / nlo) * pitch_hi + (int64_t)(pair % nlo) * pitch_lo + t;
  if (at < limit) out[at] = r0 + p0 * k1 + p0 * p1 * k2;
}

}  // namespace

size_t ntt_table_words() { return (size_t)kPrimes * 2 * N; }

cudaError_t ntt_configure() {
  const cudaError_t e = cudaFuncSetAttribute(ntt_forward_kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, kSmemBytes);
  return e != cudaSuccess
             ? e
             : cudaFuncSetAttribute(ntt_window_kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, kSmemBytes);
}

cudaError_t launch_ntt_tables(uint32_t* tables, cudaStream_t st) {
  ntt_table_kernel<<<dim3(N / 256, 2 * kPrimes), 256, 0, st>>>(tables);
  return cudaGetLastError();
}

cudaError_t launch_ntt_forward(const uint32_t* tables, const NttRows& u, uint32_t* spec_u, const NttRows& z,
                               uint32_t* spec_z, cudaStream_t st) {
  if (u.rows + z.rows <= 0) return cudaSuccess;
  ntt_forward_kernel<<<dim3((unsigned)(u.rows + z.rows), kPrimes), kThreads, kSmemBytes, st>>>(tables, u, spec_u, z,
                                                                                              spec_z);
  return cudaGetLastError();
}

cudaError_t launch_ntt_windows(const uint32_t* tables, const uint32_t* u, int nlo, const uint32_t* z, int nhi, int A,
                               uint32_t* residues, uint32_t* out, int64_t pitch_hi, int64_t pitch_lo, int64_t limit,
                               cudaStream_t st) {
  const int pairs = nlo * nhi;
  if (pairs <= 0) return cudaSuccess;
  ntt_window_kernel<<<dim3((unsigned)pairs, kPrimes), kThreads, kSmemBytes, st>>>(
      tables, u, nlo, z, nhi, A, residues);
  cudaError_t e = cudaGetLastError();
  if (e != cudaSuccess) return e;
  ntt_place_kernel<<<dim3((unsigned)((A + 255) / 256), (unsigned)pairs), 256, 0, st>>>(residues, nlo, A, pairs, out,
                                                                                       pitch_hi, pitch_lo, limit);
  return cudaGetLastError();
}

}  // namespace dpk
