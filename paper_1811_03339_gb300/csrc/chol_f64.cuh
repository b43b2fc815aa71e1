// Interface of the FP64 tile factorisation (chol_f64.cu).
#pragma once

#include "fem3_impl.cuh"

namespace fem3 {

constexpr int kChol64Tile = 32;

// flag words of a factorisation of order n (zeroed by the call)
inline int64_t chol_f64_flags(int64_t n) {
    const int64_t nblk = (n + kChol64Tile - 1) / kChol64Tile;
    return nblk * (nblk + 1) + 3;
}

// A = L L^T (row-major n x n, lower triangle read) in place below the diagonal tiles, and the
// inverses of the 64 x 64 diagonal blocks of L into dinv ([ceil(n / 64)][64][64], padded with
// the identity).  first_col: per block of kChol64Tile rows the first tile column with a nonzero
// of A (device, [ceil(n / kChol64Tile)]), or null for a full matrix.  flags: chol_f64_flags(n) words; err: ERR_COUNT error words (ERR_NOT_SPD
// gets 1 + the first column with a non-positive pivot).  Adds its launches to *launches.
int chol_f64(double *A, int64_t n, double *dinv, const int *first_col, int *flags, int32_t *err,
             cudaStream_t s, int *launches);

}  // namespace fem3
