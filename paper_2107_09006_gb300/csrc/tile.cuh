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
// 1.  Then Q = L^{-1} (lower), S's strict upper part is zeroed.  All 256 threads of the CTA
// call it.
//
// A sub-partition of the SM issues one FP64 warp instruction per 64 cycles, so the work is
// spread over four warps, one in each: warp w holds the columns c = w mod 4 (lane = row) in
// registers, column j goes through shared memory to the others, and the owner of column j +
// 1 updates and scales it before the rest of its columns, so the chain per column is one
// reciprocal square root, one product and one barrier of four warps.  The inverse is taken
// in halves of 16 (both diagonal blocks at once, one column a lane, then X21 = -X22 (L21
// X11) with one entry a thread).  It took 76 us with three CTA barriers a column, 81 us on one
// warp (992 FMAs and 64 divisions at 64 cycles each), now about 20.
__device__ __forceinline__ void tile_potrf_inv(double* S, double* Q, int* fail, int row0) {
  const int lane = threadIdx.x & 31, w = threadIdx.x >> 5;
  __syncthreads();
  if (w < 4) {
    double a[kT / 4];  // a[m]: column 4 m + w of this lane's row
#pragma unroll
    for (int m = 0; m < kT / 4; ++m) a[m] = S[lane * 33 + 4 * m + w];
    auto scale = [&](int m, int j) {  // column j (= 4 m + w) of L into S; its reciprocal pivot into Q's diagonal
      double d = __shfl_sync(0xffffffffu, a[m], j);
      if (!(d > 0.0) || !isfinite(d)) {
        if (lane == 0 && *fail == 0) *fail = row0 + j + 1;
        d = 1.0;
      }
      const double ri = rsqrt(d);
      a[m] = lane == j ? d * ri : lane > j ? a[m] * ri : 0.0;
      S[lane * 33 + j] = a[m];
      if (lane == j) Q[j * 33 + j] = ri;
    };
    if (w == 0) scale(0, 0);
#pragma unroll
    for (int j = 0; j < kT - 1; ++j) {
      asm volatile("bar.sync 1, 128;" ::: "memory");
      const double lr = S[lane * 33 + j];
      const int own = (j + 1) & 3, mo = (j + 1) >> 2;
      if (w == own) {
        a[mo] -= lr * S[(j + 1) * 33 + j];
        scale(mo, j + 1);
      }
#pragma unroll
      for (int m = (j + 1) / 4; m < kT / 4; ++m) {
        const int c = 4 * m + w;
        if (c > j + 1 || (c == j + 1 && w != own)) a[m] -= lr * S[c * 33 + j];
      }
    }
  }
  __syncthreads();
  // Q: the inverses of the two 16 x 16 diagonal blocks (the diagonal holds 1 / L_rr)
  if (w == 0) {
    const int o = lane & 16, col = lane & 15;
    double x[16];
#pragma unroll
    for (int r = 0; r < 16; ++r) {
      double acc = 0.0;
#pragma unroll
      for (int l = 0; l < r; ++l) acc += S[(o + r) * 33 + o + l] * x[l];
      const double ri = Q[(o + r) * 33 + o + r];
      x[r] = r < col ? 0.0 : r == col ? ri : -acc * ri;
    }
    __syncwarp();
#pragma unroll
    for (int r = 0; r < 16; ++r) {
      Q[(o + r) * 33 + o + col] = x[r];
      if (o == 0) Q[r * 33 + 16 + col] = 0.0;
    }
  }
  __syncthreads();
  // T = L21 X11 (kept in S's strict upper block, which is free), then Q21 = -X22 T
  const int r = threadIdx.x >> 4, c = threadIdx.x & 15;
  double acc = 0.0;
#pragma unroll
  for (int l = 0; l < 16; ++l) acc += S[(16 + r) * 33 + l] * Q[l * 33 + c];
  S[r * 33 + 16 + c] = acc;
  __syncthreads();
  acc = 0.0;
#pragma unroll
  for (int l = 0; l < 16; ++l) acc += Q[(16 + r) * 33 + 16 + l] * S[l * 33 + 16 + c];
  Q[(16 + r) * 33 + c] = -acc;
  __syncthreads();
  S[r * 33 + 16 + c] = 0.0;
  __syncthreads();
}

}  // namespace lsq
