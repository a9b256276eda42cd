// Cholesky factor of one block's R x R Hadamard-of-Grams matrix by one warp, shared by
// the update kernels.
#pragma once

#include <cuda_runtime.h>

namespace jk {

// H = L L^T in place in shared memory (lower triangle; R <= 32, row stride LD): L below
// the diagonal and on it, invd[j] = 1 / L_jj from the reciprocal square root (both
// substitutions multiply by it: no FP64 division on the serial paths).  A non-positive
// or non-finite pivot clears *spd_ok and counts as 1.

// Left-looking, for ranks known at compile time (up to 8): the short unrolled sums of a
// column's terms cost less than a pass over the trailing matrix per column (rank 5, 100
// rows: 17.6 us an update against 19.4 us with the form below; rank 3: 10.6, 11.2).
template <int LD>
__device__ __forceinline__ void warp_cholesky_left(double (*H)[LD], double* invd, int R, int lane, int* spd_ok) {
  for (int j = 0; j < R; ++j) {
    if (lane == 0) {
      double d = H[j][j];
      for (int k = 0; k < j; ++k) d -= H[j][k] * H[j][k];
      if (!(d > 0.0) || !isfinite(d)) {
        *spd_ok = 0;
        d = 1.0;
      }
      const double rs = rsqrt(d);
      H[j][j] = d * rs;
      invd[j] = rs;
    }
    __syncwarp();
    const int i = j + 1 + lane;
    if (i < R) {
      double v = H[i][j];
      for (int k = 0; k < j; ++k) v -= H[i][k] * H[j][k];
      H[i][j] = v * invd[j];
    }
    __syncwarp();
  }
}

// Right-looking, for ranks known at run time: once column j is scaled, lane i subtracts
// its products from row i of the trailing matrix, so a step's chain is one reciprocal
// square root, one product and one multiply-add, where the left-looking sums put j
// dependent multiply-adds behind shared-memory loads before every pivot and again after
// it.  The terms of every element are subtracted in the same order, one by one.  (With
// the pivot formed by every lane instead of one, all updates were 1 to 2 us longer.)
template <int LD>
__device__ __forceinline__ void warp_cholesky(double (*H)[LD], double* invd, int R, int lane, int* spd_ok) {
#pragma unroll 1
  for (int j = 0; j < R; ++j) {
    if (lane == 0) {
      double d = H[j][j];
      if (!(d > 0.0) || !isfinite(d)) {
        *spd_ok = 0;
        d = 1.0;
      }
      const double rs = rsqrt(d);
      H[j][j] = d * rs;
      invd[j] = rs;
    }
    __syncwarp();
    double l = 0.0;
    if (lane > j && lane < R) {
      l = H[lane][j] * invd[j];
      H[lane][j] = l;
    }
    __syncwarp();
    if (lane < R) {
#pragma unroll 2
      for (int k = j + 1; k <= lane; ++k) H[lane][k] -= l * H[k][j];
    }
    __syncwarp();
  }
}

// The same as a call: for kernels whose registers are full.
template <int LD>
__device__ __noinline__ void warp_cholesky_call(double (*H)[LD], double* invd, int R, int lane, int* spd_ok) {
  warp_cholesky(H, invd, R, lane, spd_ok);
}

}  // namespace jk
