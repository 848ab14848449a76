// FP64 32x32 tile helpers for the setup factorizations (CTA of 256 threads; tiles
// live in shared memory with a row pitch of 33 to spread banks).
#pragma once
#include "common.cuh"

namespace lsq {

// S = / += / -= op(P) op(Q) with op(P)[i][l] = tP ? P[l][i] : P[i][l] and
// op(Q)[l][j] = tQ ? Q[j][l] : Q[l][j]; mode 0 assigns, +1 adds, -1 subtracts.
// Each thread owns row t/8 and four consecutive columns.
template <bool tP, bool tQ>
__device__ __forceinline__ void tile_mm(double* S, const double* P, const double* Q, int mode) {
  const int t = threadIdx.x;
  const int i = t >> 3, j0 = (t & 7) * 4;
  double a0 = 0, a1 = 0, a2 = 0, a3 = 0;
#pragma unroll 8
  for (int l = 0; l < kT; ++l) {
    const double p = tP ? P[l * 33 + i] : P[i * 33 + l];
    a0 += p * (tQ ? Q[(j0 + 0) * 33 + l] : Q[l * 33 + j0 + 0]);
    a1 += p * (tQ ? Q[(j0 + 1) * 33 + l] : Q[l * 33 + j0 + 1]);
    a2 += p * (tQ ? Q[(j0 + 2) * 33 + l] : Q[l * 33 + j0 + 2]);
    a3 += p * (tQ ? Q[(j0 + 3) * 33 + l] : Q[l * 33 + j0 + 3]);
  }
  double* s = S + i * 33 + j0;
  if (mode == 0) { s[0] = a0; s[1] = a1; s[2] = a2; s[3] = a3; }
  else if (mode > 0) { s[0] += a0; s[1] += a1; s[2] += a2; s[3] += a3; }
  else { s[0] -= a0; s[1] -= a1; s[2] -= a2; s[3] -= a3; }
}

__device__ __forceinline__ void load_tile(double* dst, const double* src, int64_t ld, int64_t col0) {
  for (int e = threadIdx.x; e < kT * kT; e += blockDim.x) {
    const int rr = e >> 5, cc = e & 31;
    dst[rr * 33 + cc] = src[(int64_t)rr * ld + col0 + cc];
  }
}

__device__ __forceinline__ void store_tile(const double* src, double* dst, int64_t ld, int64_t col0) {
  for (int e = threadIdx.x; e < kT * kT; e += blockDim.x) {
    const int rr = e >> 5, cc = e & 31;
    dst[(int64_t)rr * ld + col0 + cc] = src[rr * 33 + cc];
  }
}

// Cholesky of the 32x32 tile in S (lower triangle used); on a pivot that is not positive and
// finite records 1 + (row0 + row) in *fail (first failure only) and continues with pivot
// 1.  Then Q = L^{-1} (lower), S's strict upper part is zeroed.  Every thread of the CTA
// calls it; the first warp does the work, lane r holding row r (then column r of the
// inverse) in registers: with the tile in shared memory and three CTA barriers a column it
// took 76 us, nearly all of it barriers.
__device__ __forceinline__ void tile_potrf_inv(double* S, double* Q, int* fail, int row0) {
  __syncthreads();
  if (threadIdx.x < 32) {
    const int lane = threadIdx.x;
    double a[kT];
#pragma unroll
    for (int c = 0; c < kT; ++c) a[c] = S[lane * 33 + c];
#pragma unroll
    for (int j = 0; j < kT; ++j) {
      double d = __shfl_sync(0xffffffffu, a[j], j);
      if (!(d > 0.0) || !isfinite(d)) {
        if (lane == 0 && *fail == 0) *fail = row0 + j + 1;
        d = 1.0;
      }
      const double root = sqrt(d);
      a[j] = lane == j ? root : lane > j ? a[j] / root : 0.0;
#pragma unroll
      for (int c = j + 1; c < kT; ++c) a[c] -= a[j] * __shfl_sync(0xffffffffu, a[j], c);
    }
#pragma unroll
    for (int c = 0; c < kT; ++c) S[lane * 33 + c] = c <= lane ? a[c] : 0.0;
    __syncwarp();
    // column `lane` of the inverse, top down
#pragma unroll
    for (int r = 0; r < kT; ++r) {
      double acc = 0.0;
#pragma unroll
      for (int l = 0; l < r; ++l) acc += S[r * 33 + l] * a[l];
      a[r] = r < lane ? 0.0 : (r == lane ? 1.0 : -acc) / S[r * 33 + r];
    }
#pragma unroll
    for (int r = 0; r < kT; ++r) Q[r * 33 + lane] = a[r];
  }
  __syncthreads();
}

}  // namespace lsq
