// Local matrices in block-envelope storage: assembly of C_ii and C~_ii, the shifts of
// Section 4.1.2 and the batched Cholesky (right-looking over 32x32 tiles).
#include "band.cuh"
#include "tile.cuh"
#include "kernels.h"

namespace lsq {

namespace {

__device__ __forceinline__ int lower_bound_i32(const int32_t* a, int n, int32_t key) {
  int lo = 0, hi = n;
  while (lo < hi) {
    const int mid = (lo + hi) >> 1;
    if (a[mid] < key) lo = mid + 1; else hi = mid;
  }
  return lo;
}

// One thread per local row k of subdomain i: row k of C_ii = sum over the rows r of A
// that touch column Omega_i[k] of a_{r,k} a_{r,q} (q in Omega_i, q <= k); the rows
// of Xi_i (those touching an interior column) also go to C~_ii (eq. (3.2)).
__global__ void __launch_bounds__(kThreads) k_assemble(BandPlan P, CsrDev A, CscDev At,
                                                       const int32_t* __restrict__ part, int64_t total,
                                                       double* __restrict__ C, double* __restrict__ Ct) {
  for (int64_t e = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; e < total; e += (int64_t)gridDim.x * blockDim.x) {
    const int i = P.row_sub[e];
    const int64_t o0 = P.om_off[i];
    const int ni = (int)(P.om_off[i + 1] - o0);
    const int k = (int)(e - o0);
    const int32_t* om = P.om_glob + o0;
    const int b = k >> 5, rr = k & 31;
    const int64_t bi = P.blk_off[i] + b;
    const int t0 = P.blk_tf[bi];
    const int width = (b - t0 + 1) * kT;
    const int64_t rowoff = P.blk_poff[bi] + (int64_t)rr * width - (int64_t)t0 * kT;
    const int32_t g = om[k];
    for (int64_t e2 = At.col_ptr[g]; e2 < At.col_ptr[g + 1]; ++e2) {
      const int32_t r = At.row[e2];
      const double arg = At.val[e2];
      const int64_t s0 = A.row_ptr[r], s1 = A.row_ptr[r + 1];
      bool inxi = false;
      for (int64_t s = s0; s < s1; ++s)
        if (part[A.col[s]] == i) { inxi = true; break; }
      for (int64_t s = s0; s < s1; ++s) {
        const int32_t c = A.col[s];
        const int q = lower_bound_i32(om, ni, c);
        if (q < ni && om[q] == c && q <= k) {
          const double v = arg * A.val[s];
          C[rowoff + q] += v;
          if (inxi) Ct[rowoff + q] += v;
        }
      }
    }
  }
}

// One CTA per block row (blockIdx.y) of a subdomain (blockIdx.x): the row's part of the two sums,
// added per subdomain in row order by k_norms_sum.  (16 subdomains of 1,900 columns: one CTA
// per subdomain took 1.42 ms, 0.10 so; the same split of k_prep 1.46 ms, 0.07.)
__global__ void __launch_bounds__(kThreads) k_norms(BandPlan P, const double* __restrict__ C,
                                                    const double* __restrict__ Ct, double* __restrict__ parts) {
  __shared__ double red[kWarps];
  const int i = blockIdx.x, b = blockIdx.y;
  const int64_t o0 = P.om_off[i];
  const int ni = (int)(P.om_off[i + 1] - o0);
  const int64_t b0 = P.blk_off[i];
  if (b >= (int)(P.blk_off[i + 1] - b0)) return;
  const uint8_t* isint = P.om_int + o0;
  double sc = 0.0, st = 0.0;
  const int t0 = P.blk_tf[b0 + b];
  const int width = (b - t0 + 1) * kT;
  const int64_t po = P.blk_poff[b0 + b];
  for (int e = threadIdx.x; e < kT * width; e += blockDim.x) {
    const int rr = e / width, cc = e - rr * width;
    const int p = b * kT + rr, q = t0 * kT + cc;
    if (p >= ni || q > p) continue;
    const double v = C[po + e], w = Ct[po + e];
    sc += v * v * (double)(isint[p] + (q < p ? isint[q] : 0));
    st += w * w * (q == p ? 1.0 : 2.0);
  }
  const double s1 = block_sum(sc, red);
  const double s2 = block_sum(st, red);
  if (threadIdx.x == 0) { parts[2 * (b0 + b)] = s1; parts[2 * (b0 + b) + 1] = s2; }
}

__global__ void k_norms_sum(BandPlan P, const double* __restrict__ parts, double* __restrict__ cn2,
                            double* __restrict__ ctn2) {
  const int i = blockIdx.x * blockDim.x + threadIdx.x;
  if (i >= P.N) return;
  double sc = 0.0, st = 0.0;
  for (int64_t b = P.blk_off[i]; b < P.blk_off[i + 1]; ++b) { sc += parts[2 * b]; st += parts[2 * b + 1]; }
  cn2[i] = sc;
  ctn2[i] = st;
}

// C_ii += delta I; eqs = diag^{-1/2}.
__global__ void __launch_bounds__(kThreads) k_prep_diag(BandPlan P, const double* __restrict__ dsub,
                                                        double* __restrict__ C, double* __restrict__ eqs) {
  const int i = blockIdx.x, k = blockIdx.y * kThreads + threadIdx.x;
  const int64_t o0 = P.om_off[i];
  const int ni = (int)(P.om_off[i + 1] - o0);
  const int64_t b0 = P.blk_off[i];
  if (k >= (int)(P.blk_off[i + 1] - b0) * kT) return;
  const int b = k >> 5, rr = k & 31;
  const int width = (b - P.blk_tf[b0 + b] + 1) * kT;
  const int64_t d = P.blk_poff[b0 + b] + (int64_t)rr * width + (width - kT) + rr;
  if (k < ni) {
    const double c = C[d] + dsub[i];
    C[d] = c;
    eqs[o0 + k] = c > 0.0 ? 1.0 / sqrt(c) : 1.0;
  } else {
    C[d] = 1.0;
  }
}

// C_ii <- diag(eqs) C_ii diag(eqs); B = C~_ii + s_i I, one CTA per block row.  Padding rows
// (k >= n_i) become identity rows in both storages.
__global__ void __launch_bounds__(kThreads) k_prep(BandPlan P, const double* __restrict__ s, double* __restrict__ C,
                                                   const double* __restrict__ eqs, const double* __restrict__ Ct,
                                                   double* __restrict__ B) {
  const int i = blockIdx.x, b = blockIdx.y;
  const int64_t o0 = P.om_off[i];
  const int ni = (int)(P.om_off[i + 1] - o0);
  const int64_t b0 = P.blk_off[i];
  if (b >= (int)(P.blk_off[i + 1] - b0)) return;
  const double si = s[i];
  const int t0 = P.blk_tf[b0 + b];
  const int width = (b - t0 + 1) * kT;
  const int64_t po = P.blk_poff[b0 + b];
  for (int e = threadIdx.x; e < kT * width; e += blockDim.x) {
    const int rr = e / width, cc = e - rr * width;
    const int p = b * kT + rr, q = t0 * kT + cc;
    double bv = Ct[po + e];
    if (p < ni && q < ni) {
      C[po + e] *= eqs[o0 + p] * eqs[o0 + q];
      if (p == q) bv += si;
    } else if (p == q) {
      bv = 1.0;
    } else {
      bv = 0.0;
      C[po + e] = 0.0;
    }
    B[po + e] = bv;
  }
}

// Right-looking tiled Cholesky of every subdomain's block-envelope matrix, in place, block
// column by block column for all subdomains at once: the diagonal tile (and its inverse, kept
// in dinv, 1024 doubles per block row), the tiles below it, the update of the window's
// tiles, one CTA per tile.  FP64-bound: a tile update is 32,768 FMAs, 8 us of one SM's two
// per cycle; one CTA per subdomain ran the whole factor on as many SMs as there were
// subdomains (16 of 1,936 columns: 33 ms).
__global__ void __launch_bounds__(kThreads) k_chol_diag(BandPlan P, double* __restrict__ F, double* __restrict__ idiag,
                                                        double* __restrict__ dinv, int* __restrict__ status,
                                                        const int32_t* __restrict__ order, int k) {
  __shared__ double S[kT * 33], Q[kT * 33];
  __shared__ int fail;
  const int i = order ? order[blockIdx.x] : blockIdx.x;
  const int64_t b0 = P.blk_off[i];
  if (k >= (int)(P.blk_off[i + 1] - b0)) return;
  const int t0 = P.blk_tf[b0 + k];
  const int width = (k - t0 + 1) * kT;
  double* pan = F + P.blk_poff[b0 + k];
  if (threadIdx.x == 0) fail = 0;
  load_tile(S, pan, width, width - kT);
  tile_potrf_inv(S, Q, &fail, k * kT);
  store_tile(S, pan, width, width - kT);
  double* dv = dinv + (b0 + k) * (int64_t)(kT * kT);
  for (int e = threadIdx.x; e < kT * kT; e += blockDim.x) dv[e] = Q[(e >> 5) * 33 + (e & 31)];
  if (threadIdx.x < kT) idiag[b0 * kT + k * kT + threadIdx.x] = Q[threadIdx.x * 33 + threadIdx.x];
  if (threadIdx.x == 0 && fail && status[i] == 0) status[i] = fail;
}

// L(b, k) = A(b, k) L(k, k)^{-T} for the block rows b > k that reach column k.
__global__ void __launch_bounds__(kThreads) k_chol_col(BandPlan P, double* __restrict__ F,
                                                       const double* __restrict__ dinv,
                                                       const int32_t* __restrict__ order, int k) {
  __shared__ double S[kT * 33], A[kT * 33], Q[kT * 33];
  const int i = order ? order[blockIdx.x] : blockIdx.x, b = k + 1 + blockIdx.y;
  const int64_t b0 = P.blk_off[i];
  if (b >= (int)(P.blk_off[i + 1] - b0)) return;
  const int t0 = P.blk_tf[b0 + b];
  if (t0 > k) return;
  const int width = (b - t0 + 1) * kT;
  double* pan = F + P.blk_poff[b0 + b];
  load_tile(A, pan, width, (k - t0) * kT);
  const double* dv = dinv + (b0 + k) * (int64_t)(kT * kT);
  for (int e = threadIdx.x; e < kT * kT; e += blockDim.x) Q[(e >> 5) * 33 + (e & 31)] = dv[e];
  __syncthreads();
  tile_mm<false, true>(S, A, Q, 0);
  __syncthreads();
  store_tile(S, pan, width, (k - t0) * kT);
}

// A(b, c) -= L(b, k) L(c, k)^T for k < c <= b, both reaching column k (the CTAs in y stride over
// the pairs of the window below k).
__global__ void __launch_bounds__(kThreads) k_chol_update(BandPlan P, double* __restrict__ F,
                                                          const int32_t* __restrict__ order, int k, int below) {
  __shared__ double S[kT * 33], A[kT * 33], Q[kT * 33];
  const int i = order ? order[blockIdx.x] : blockIdx.x;
  const int64_t b0 = P.blk_off[i];
  const int nb = (int)(P.blk_off[i + 1] - b0);
  const int64_t pairs = chol_pairs(below);
  for (int64_t e = blockIdx.y; e < pairs; e += gridDim.y) {
    int b, c;
    chol_pair(e, b, c);
    b += k + 1;
    c += k + 1;
    if (b >= nb) return;
    const int tb = P.blk_tf[b0 + b], tc = P.blk_tf[b0 + c];
    if (tb > k || tc > k) continue;
    const int wb = (b - tb + 1) * kT, wc = (c - tc + 1) * kT;
    double* panb = F + P.blk_poff[b0 + b];
    const double* panc = F + P.blk_poff[b0 + c];
    load_tile(S, panb, wb, (c - tb) * kT);
    load_tile(A, panb, wb, (k - tb) * kT);
    load_tile(Q, panc, wc, (k - tc) * kT);
    __syncthreads();
    tile_mm<false, true>(S, A, Q, -1);
    __syncthreads();
    store_tile(S, panb, wb, (c - tb) * kT);
    __syncthreads();
  }
}

int grid_for(int64_t work, int cap) {
  int64_t g = (work + kThreads - 1) / kThreads;
  return (int)(g < 1 ? 1 : (g > cap ? cap : g));
}

}  // namespace

void launch_assemble(const BandPlan& P, const CsrDev& A, const CscDev& At, const int32_t* part,
                     int64_t total_local, double* Cst, double* Ctst, cudaStream_t st) {
  k_assemble<<<grid_for(total_local, 1 << 15), kThreads, 0, st>>>(P, A, At, part, total_local, Cst, Ctst);
}

void launch_norms(const BandPlan& P, int max_nb, const double* Cst, const double* Ctst, double* parts, double* cn2,
                  double* ctn2, cudaStream_t st) {
  k_norms<<<dim3(P.N, max_nb), kThreads, 0, st>>>(P, Cst, Ctst, parts);
  k_norms_sum<<<(P.N + 63) / 64, 64, 0, st>>>(P, parts, cn2, ctn2);
}

void launch_prep(const BandPlan& P, int max_nb, const double* dsub, const double* s, double* Cst, double* eqs,
                 const double* Ctst, double* Bst, cudaStream_t st) {
  k_prep_diag<<<dim3(P.N, (max_nb * kT + kThreads - 1) / kThreads), kThreads, 0, st>>>(P, dsub, Cst, eqs);
  k_prep<<<dim3(P.N, max_nb), kThreads, 0, st>>>(P, s, Cst, eqs, Ctst, Bst);
}

void launch_band_cholesky(const BandPlan& P, const std::vector<CholGroup>& groups, const int32_t* order, double* F,
                          double* idiag, double* dinv, int* status, cudaStream_t st) {
  cudaMemsetAsync(status, 0, sizeof(int) * P.N, st);
  for (const CholGroup& g : groups) {
    const int32_t* ord = groups.size() > 1 ? order + g.first : nullptr;  // (one group: all, in any order)
    for (int k = 0; k < g.max_nb; ++k) {
      k_chol_diag<<<g.count, kThreads, 0, st>>>(P, F, idiag, dinv, status, ord, k);
      const int below = std::min(g.below, g.max_nb - 1 - k);  // block rows that can reach column k
      if (below > 0) {
        k_chol_col<<<dim3(g.count, below), kThreads, 0, st>>>(P, F, dinv, ord, k);
        k_chol_update<<<dim3(g.count, chol_grid_y(below)), kThreads, 0, st>>>(P, F, ord, k, below);
      }
    }
  }
}

}  // namespace lsq
