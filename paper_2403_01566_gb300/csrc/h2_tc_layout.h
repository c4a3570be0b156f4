// Shared-memory layout of the sliced tensor-core GEMM (h2_gemm_tc.cu): the S
// slices of op(A), those of op(B), the FP64 outputs, the maxima, and the middle
// product of three-factor terms.  Plain functions of the shape, so that the
// host can check them.
#pragma once
#include <cuda_runtime.h>
#include <stdint.h>

namespace h2 {

// Bytes of a slice tile: 64 rows of TK = 32 FP16 whatever the job's size, so
// that the slices of an element and of a fragment lie at constant offsets.
constexpr int TC_SLICE = 64 * 64;

// Slice tiles: rows of TK FP16 (64 bytes), the 16-byte pieces of a row
// exchanged by its row pair, so that the eight rows of an ldmatrix and the
// row pairs of a slice store meet in distinct banks without padding.
__host__ __device__ constexpr uint32_t tc_piece(int row, int c) {
  return (uint32_t)(row * 64 + ((c ^ ((row >> 1) & 3)) << 4));
}

// Ints of a set of maxima: rows of op(A) and columns of op(B) (64 each), the
// same after balancing, k of op(A) and op(B) (32 each); two sets (alternating
// chunks).
constexpr int TC_SET = 320;

// Row length of the FP64 tiles in shared memory: eight rows' pairs of outputs
// meet in distinct banks (a multiple of 128 bytes plus 64).
__host__ __device__ constexpr int tc_ldo(int nb) { return ((nb + 15) & ~15) + 8; }

// Fragments of op(B): one ldmatrix takes slices 2q and 2q + 1 of column tile ct
// and k step ks.  Offset of a lane's row, at q = 0; load q is 2 q slices on.
__host__ __device__ constexpr uint32_t tc_b_lane(int lane, int ct, int ks) {
  return (uint32_t)((lane >> 4) * TC_SLICE) + tc_piece(ct * 8 + (lane & 7), 2 * ks + ((lane >> 3) & 1));
}
// Lanes whose rows load q reads: the last slice of an odd number is loaded
// alone (the rows behind it are not op(B)'s, and for the smallest tiles not in
// the launch's shared memory).
__host__ __device__ constexpr int tc_b_lanes(int S, int q) { return 2 * q + 1 < S ? 32 : 16; }

__host__ __device__ constexpr int tc_smem_bytes(int S, int mmax, int nb, bool t3) {
  return 2 * S * TC_SLICE + 2 * TC_SET * 4 + (t3 ? 2 : 1) * 8 * mmax * tc_ldo(nb);
}

}  // namespace h2
