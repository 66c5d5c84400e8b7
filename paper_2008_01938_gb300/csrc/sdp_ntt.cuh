// sdp_ntt.cuh -- middle products over Z/2^32 by number-theoretic transforms.
//
// The windows of sdp_jump.cu are middle products
//     out[t] = sum_{s < A} u[s] z[t + s],   0 <= t < A,
// of rows u (A words) and z (2A - 1 words), one for every pair of a u and a z.
// Directly that is A^2 multiply-adds each; as cyclic convolutions of length N =
// 2^14 >= 2A - 1 of the reversed u with z (the outputs wanted, at A - 1 + t, are
// the ones no wrapped term reaches) it is a transform per row, a point-wise
// product and an inverse transform per pair, modulo three primes of 30, 28 and 29 bits.
// The exact integer sums are below A 2^64 <= 2^77, less than the primes' product
// (above 2^86), so Garner's form of the Chinese remainder theorem gives them modulo
// 2^32 exactly.  (D. E. Knuth, The Art of Computer Programming 2, 4.3.2 and
// 4.3.3; products by constants as in V. Shoup's NTL.)
#pragma once

#include <cstdint>
#include <cuda_runtime.h>

namespace dpk {

constexpr int kNttLog2 = 14;
constexpr int kNttN = 1 << kNttLog2;
constexpr int kNttMaxA = kNttN / 2;

struct NttRows {          // rows (words) of a forward transform
  const uint32_t* src;
  int64_t pitch;          // row r starts at src + r * pitch
  int64_t len;            // words of a row ...
  int64_t limit;          // ... of which those at src + x, x < limit, are read; the others are 0
  int32_t reverse;        // 1: word i of the transform's input is word len - 1 - i of the row
  int32_t rows;
};

// Words of workspace: twiddle tables, and a spectrum per row and prime.
size_t ntt_table_words();
inline size_t ntt_spectrum_words(int64_t rows) { return (size_t)3 * rows * kNttN; }
cudaError_t ntt_configure();
cudaError_t launch_ntt_tables(uint32_t* tables, cudaStream_t st);
// The spectra of the rows u and z (side by side in one launch).
cudaError_t launch_ntt_forward(const uint32_t* tables, const NttRows& u, uint32_t* spec_u, const NttRows& z,
                               uint32_t* spec_z, cudaStream_t st);
// Outputs t < A of every pair (hi, lo) of nhi spectra z and nlo spectra u:
// word t goes to out + hi * pitch_hi + lo * pitch_lo + t where that offset
// is below limit.  residues: 3 nhi nlo A words.
cudaError_t launch_ntt_windows(const uint32_t* tables, const uint32_t* u, int nlo, const uint32_t* z, int nhi, int A,
                               uint32_t* residues, uint32_t* out, int64_t pitch_hi, int64_t pitch_lo, int64_t limit,
                               cudaStream_t st);

}  // namespace dpk
