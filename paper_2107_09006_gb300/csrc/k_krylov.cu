// Sparse products with A and A^T, the CG vector updates, the overlap scatter-add with
// coarse prolongation, the coarse GEMV and the adjoint-gradient kernel.  All FP64.
//
// Reductions: a kernel that produces a dot product writes one partial sum per block;
// the last block to finish (an atomic ticket after a memory fence, no waiting) sums
// the partials in block order and stores the scalar into a slot of the device CG
// state.  The result does not depend on scheduling, so CUDA-graph replays are
// bit-reproducible, and consumers read one scalar.
#include "common.cuh"
#include "kernels.h"
#include "normal_tiles.h"

namespace lsq {

namespace {

__device__ __forceinline__ unsigned seg_mask(int V) {
  const int lane = threadIdx.x & 31;
  return V == 32 ? 0xffffffffu : (((1u << V) - 1u) << (lane / V * V));
}

// Block sums of one or two values in thread 0: the warps' sums meet in shared memory and eight
// lanes add them (a sub-partition issues one FP64 warp instruction per 64 cycles, so the sum
// of block_sum, formed by every warp, costs more than everything else in a small kernel: the
// vector update of 37 thousand columns takes 5.7 us, 6.6 with block_sum; 102 thousand 8.2 and 10.3).
__device__ __forceinline__ void block_sums(double& s1, double& s2, bool two, double* red) {
  const int lane = threadIdx.x & 31, w = threadIdx.x >> 5;
  s1 = warp_sum(s1);
  if (two) s2 = warp_sum(s2);
  if (lane == 0) {
    red[w] = s1;
    if (two) red[kWarps + w] = s2;
  }
  __syncthreads();
  if (w == 0) {  // lanes 0-7: the first value, 8-15: the second
    double s = lane < (two ? 2 * kWarps : kWarps) ? red[lane] : 0.0;
#pragma unroll
    for (int o = kWarps / 2; o > 0; o >>= 1) s += __shfl_xor_sync(0xffffffffu, s, o);
    s1 = s;
    s2 = __shfl_sync(0xffffffffu, s, kWarps);
  }
}

// Block partials -> last block sums them in order -> *out (and a second sum if two).
__device__ __forceinline__ void finish_dots(double s1, double s2, bool two, const DotSite& d) {
  __shared__ double red[2 * kWarps];
  __shared__ bool last;
  block_sums(s1, s2, two, red);
  if (threadIdx.x == 0) {
    d.parts[blockIdx.x] = s1;
    if (two) d.parts[d.stride + blockIdx.x] = s2;
    __threadfence();
    const unsigned t = atomicAdd(d.counter, 1u);
    last = (t == gridDim.x - 1);
  }
  __syncthreads();
  if (last) {
    __threadfence();
    double a1 = 0.0, a2 = 0.0;
    for (int k = threadIdx.x; k < (int)gridDim.x; k += blockDim.x) {
      a1 += __ldcg(d.parts + k);
      if (two) a2 += __ldcg(d.parts + d.stride + k);
    }
    block_sums(a1, a2, two, red);
    if (threadIdx.x == 0) {
      d.out[0] = a1;
      if (two) d.out[d.out2] = a2;
      *d.counter = 0u;
    }
  }
}

// y = A x, V lanes per row.  Each lane group walks its row with stride V; rows of a
// few entries use small V so more rows are in flight per warp.
template <int V>
__global__ void __launch_bounds__(kThreads) k_spmv_csr(CsrDev A, const double* __restrict__ x,
                                                       double* __restrict__ y) {
  const int64_t gt = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
  const int sub = threadIdx.x % V;
  const int64_t stride = (int64_t)gridDim.x * blockDim.x / V;
  const unsigned mask = seg_mask(V);
  for (int64_t r = gt / V; r < A.m; r += stride) {
    double acc = 0.0;
    const int64_t e0 = __ldg(A.row_ptr + r), e1 = __ldg(A.row_ptr + r + 1);
#pragma unroll 4
    for (int64_t e = e0 + sub; e < e1; e += V) acc += __ldg(A.val + e) * __ldg(x + __ldg(A.col + e));
#pragma unroll
    for (int o = V / 2; o > 0; o >>= 1) acc += __shfl_xor_sync(mask, acc, o);
    if (sub == 0) y[r] = acc;
  }
}

// w = A^T q through the CSC copy; optionally d.w into the dot site (d = w if null).
template <int V>
__global__ void __launch_bounds__(kThreads) k_spmv_csc(CscDev At, const double* __restrict__ q,
                                                       double* __restrict__ w, const double* __restrict__ d,
                                                       DotSite ds) {
  const int64_t gt = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
  const int sub = threadIdx.x % V;
  const int64_t stride = (int64_t)gridDim.x * blockDim.x / V;
  const unsigned mask = seg_mask(V);
  double dacc = 0.0;
  for (int64_t j = gt / V; j < At.n; j += stride) {
    double acc = 0.0;
    const int64_t e0 = __ldg(At.col_ptr + j), e1 = __ldg(At.col_ptr + j + 1);
#pragma unroll 4
    for (int64_t e = e0 + sub; e < e1; e += V) acc += __ldg(At.val + e) * __ldg(q + __ldg(At.row + e));
#pragma unroll
    for (int o = V / 2; o > 0; o >>= 1) acc += __shfl_xor_sync(mask, acc, o);
    if (sub == 0) {
      w[j] = acc;
      dacc += (d ? d[j] : acc) * acc;
    }
  }
  if (ds.parts) finish_dots(dacc, 0.0, false, ds);
}

// y = B x for a CSR matrix B (A, or A^T through the CSC copy) of unknown row lengths: V lanes
// per row as in k_spmv_csr, but a row of more than kLongRow entries per lane is left to its
// whole warp.  V goes by the mean length, and a few lanes on one long row are a chain that
// the rest of the matrix does not hide (400,000 rows of six entries, 25 us, and one of
// 100,000: 6.6 ms with two lanes on it, 2.2 with eight, 0.56 so; a column of 100,000 among
// columns of 24: 3.6 ms with four lanes, 0.40 so; Pareto row lengths: 8, 16 and 32 entries per
// lane 104, 84 and 86 us).  The bound on the blocks keeps 32 registers where rows are short.
constexpr int kLongRow = 16;
template <int V>
__global__ void __launch_bounds__(kThreads, V <= 2 ? 8 : 6) k_product(int64_t rows, const int64_t* __restrict__ ptr,
                                                      const int32_t* __restrict__ idx, const double* __restrict__ val,
                                                      const double* __restrict__ x, double* __restrict__ y) {
  const int lane = threadIdx.x & 31, sub = lane % V;
  const int64_t stride = (int64_t)gridDim.x * blockDim.x / V;
  for (int64_t r0 = ((int64_t)blockIdx.x * blockDim.x + threadIdx.x - lane) / V; r0 < rows; r0 += stride) {
    const int64_t r = r0 + lane / V;  // (the loop is the warp's)
    double acc = 0.0;
    bool longrow = false;
    if (r < rows) {
      const int64_t e0 = __ldg(ptr + r), e1 = __ldg(ptr + r + 1);
      longrow = V < 32 && e1 - e0 > kLongRow * V;
      if (!longrow) {
#pragma unroll 4
        for (int64_t e = e0 + sub; e < e1; e += V) acc += __ldg(val + e) * __ldg(x + __ldg(idx + e));
      }
    }
#pragma unroll
    for (int o = V / 2; o > 0; o >>= 1) acc += __shfl_xor_sync(0xffffffffu, acc, o);
    if (r < rows && sub == 0 && !longrow) y[r] = acc;
    if constexpr (V < 32) {
      for (unsigned todo = __ballot_sync(0xffffffffu, longrow && sub == 0); todo; todo &= todo - 1) {
        const int64_t rl = r0 + (__ffs(todo) - 1) / V, e1 = __ldg(ptr + rl + 1);
        double s = 0.0;
#pragma unroll 4
        for (int64_t e = __ldg(ptr + rl) + lane; e < e1; e += 32) s += __ldg(val + e) * __ldg(x + __ldg(idx + e));
        s = warp_sum(s);
        if (lane == 0) y[rl] = s;
      }
    }
  }
}

// Warp-stream product y = B x for a CSR matrix B (A itself, or A^T through the CSC copy):
// each warp takes R consecutive rows, loads all their entries coalesced (lanes stride the
// entry range, all loads independent), keeps the products in shared memory, then lane k
// sums row k in storage order.  Row blocks whose entries exceed CAP fall back to one
// warp per row.  Optional fused d . y as in k_spmv_csc.
template <int R, int CAP>
__global__ void __launch_bounds__(kThreads) k_spmv_stream(int64_t nrows, const int64_t* __restrict__ ptr,
                                                          const int32_t* __restrict__ idx,
                                                          const double* __restrict__ val,
                                                          const double* __restrict__ x, double* __restrict__ y,
                                                          const double* __restrict__ d, DotSite ds) {
  __shared__ double prod[kWarps][CAP];
  const int lane = threadIdx.x & 31, w = threadIdx.x >> 5;
  double* sm = prod[w];
  double dacc = 0.0;
  const int64_t nblk = (nrows + R - 1) / R;
  for (int64_t rb = (int64_t)blockIdx.x * kWarps + w; rb < nblk; rb += (int64_t)gridDim.x * kWarps) {
    const int64_t r0 = rb * R;
    const int64_t r = r0 + lane;
    const bool mine = lane < R && r < nrows;
    const int64_t plo = __ldg(ptr + (mine ? r : min(r0 + R, nrows)));
    const int64_t rend = min(r0 + R, nrows);
    const int64_t e1 = __ldg(ptr + rend);
    const int64_t e0 = __shfl_sync(0xffffffffu, plo, 0);
    const int64_t phi = __shfl_down_sync(0xffffffffu, plo, 1);
    const int64_t my_hi = (lane == R - 1 || r + 1 >= rend) ? e1 : phi;
    if (e1 - e0 <= CAP) {
#pragma unroll 4
      for (int64_t e = e0 + lane; e < e1; e += 32) sm[e - e0] = __ldg(val + e) * __ldg(x + __ldg(idx + e));
      __syncwarp();
      if (mine) {
        double s = 0.0;
        for (int64_t e = plo; e < my_hi; ++e) s += sm[e - e0];
        y[r] = s;
        dacc += (d ? d[r] : s) * s;
      }
      __syncwarp();
    } else {
      for (int64_t rr = r0; rr < rend; ++rr) {
        const int64_t a0 = __ldg(ptr + rr), a1 = __ldg(ptr + rr + 1);
        double s = 0.0;
        for (int64_t e = a0 + lane; e < a1; e += 32) s += __ldg(val + e) * __ldg(x + __ldg(idx + e));
        s = warp_sum(s);
        if (lane == 0) {
          y[rr] = s;
          dacc += (d ? d[rr] : s) * s;
        }
      }
    }
  }
  if (ds.parts) finish_dots(dacc, 0.0, false, ds);
}

// Sliced-ELL product: one warp per slice of 32 rows, lane l owns slice row l; every
// step k loads 32 consecutive (column, value) pairs, so there is no per-row pointer
// chase and the gathers of successive k are independent.
__global__ void __launch_bounds__(kThreads) k_spmv_sell(SellDev S, const double* __restrict__ x,
                                                        double* __restrict__ y, const double* __restrict__ d,
                                                        DotSite ds) {
  const int lane = threadIdx.x & 31;
  double dacc = 0.0;
  for (int64_t s = ((int64_t)blockIdx.x * blockDim.x + threadIdx.x) >> 5; s < S.nslices;
       s += ((int64_t)gridDim.x * blockDim.x) >> 5) {
    const int64_t o = __ldg(S.off + s);
    const int W = (int)((__ldg(S.off + s + 1) - o) >> 5);
    const int r = __ldg(S.perm + s * 32 + lane);
    const int32_t* cp = S.col + o + lane;
    const double* vp = S.val + o + lane;
    double acc = 0.0;
#pragma unroll 8
    for (int k = 0; k < W; ++k) acc += __ldg(vp + 32 * k) * __ldg(x + __ldg(cp + 32 * k));
    if (r >= 0) {
      y[r] = acc;
      dacc += (d ? d[r] : acc) * acc;
    }
  }
  if (ds.parts) finish_dots(dacc, 0.0, false, ds);
}

// alpha = rz / pw; x += alpha p; r_old = r; r -= alpha w; rr = r.r.  One thread of a block
// divides (a division in every thread is FP64 issue of the same order as the update) while
// the others' loads, four entries each, are in flight; the same in k_p_update (102 thousand
// columns: 8.1 -> 6.9 and 5.5 -> 4.1 us; a million: 21.8 -> 20.2 and 9.9 -> 6.9).
constexpr int kVecUnroll = 4;
__global__ void __launch_bounds__(kThreads) k_cg_update(int64_t n, double* scal, const double* __restrict__ p,
                                                        const double* __restrict__ w, double* __restrict__ x,
                                                        double* __restrict__ r, double* __restrict__ r_old,
                                                        DotSite rr, int* ctr, double* alpha_hist, int cap) {
  __shared__ double sh;
  if (threadIdx.x == 0) {
    const double rz = scal[S_RZ], pw = scal[S_PW];
    const double al = rz / pw;
    sh = al;
    if (blockIdx.x == 0) {
      scal[S_RZOLD] = rz;
      scal[S_ALPHA] = al;
      const int it = *ctr;
      if (it >= 0 && it < cap) alpha_hist[it] = al;
      if (!(pw > 0.0) || !isfinite(al)) scal[S_FLAG] = 1.0;
    }
  }
  const int64_t step = (int64_t)gridDim.x * blockDim.x;
  double acc = 0.0, alpha = 0.0;
  bool first = true;
  for (int64_t k0 = (int64_t)blockIdx.x * blockDim.x; k0 < n; k0 += kVecUnroll * step) {
    double pk[kVecUnroll], wk[kVecUnroll], xk[kVecUnroll], rk[kVecUnroll];
#pragma unroll
    for (int u = 0; u < kVecUnroll; ++u) {
      const int64_t k = k0 + u * step + threadIdx.x;
      const bool in = k < n;
      pk[u] = in ? p[k] : 0.0;
      wk[u] = in ? w[k] : 0.0;
      xk[u] = in ? x[k] : 0.0;
      rk[u] = in ? r[k] : 0.0;
    }
    if (first) {  // (the whole block)
      __syncthreads();
      alpha = sh;
      first = false;
    }
#pragma unroll
    for (int u = 0; u < kVecUnroll; ++u) {
      const int64_t k = k0 + u * step + threadIdx.x;
      if (k >= n) continue;
      x[k] = xk[u] + alpha * pk[u];
      if (r_old) r_old[k] = rk[u];
      const double rn = rk[u] - alpha * wk[u];
      r[k] = rn;
      acc += rn * rn;
    }
  }
  finish_dots(acc, 0.0, false, rr);
}

// beta = rz_new / rz_old (or (rz_new - rzo_new) / rz_old, flexible); p = z + beta p.
__global__ void __launch_bounds__(kThreads) k_p_update(int64_t n, double* scal, int* ctr, double* beta_hist,
                                                       int cap, const double* __restrict__ z, double* __restrict__ p,
                                                       int init, int flex, LoopTest loop) {
  __shared__ double sh;
  if (!init && threadIdx.x == 0) {
    const double num = flex ? scal[S_RZ] - scal[S_RZO] : scal[S_RZ];
    const double beta = num / scal[S_RZOLD];
    sh = beta;
    if (blockIdx.x == 0) {
      scal[S_BETA] = beta;
      const int it = *ctr;
      if (it >= 0 && it < cap) beta_hist[it] = beta;
      *ctr = it + 1;
      scal[S_ITS] = (double)(it + 1);
      if (!isfinite(beta)) scal[S_FLAG] = 1.0;
      if (loop.limit > 0) {
        const double rr = scal[S_RR], thr = scal[S_THR];
        bool go = isfinite(beta) && scal[S_FLAG] == 0.0 && scal[S_ERR] == 0.0 && isfinite(rr) && it + 1 < loop.limit;
        if (thr > 0.0 && rr <= thr) go = false;
        cudaGraphSetConditional(loop.handle, go ? 1u : 0u);
      }
    }
  }
  const int64_t step = (int64_t)gridDim.x * blockDim.x;
  double beta = 0.0;
  bool first = !init;
  for (int64_t k0 = (int64_t)blockIdx.x * blockDim.x; k0 < n; k0 += kVecUnroll * step) {
    double zk[kVecUnroll], pk[kVecUnroll];
#pragma unroll
    for (int u = 0; u < kVecUnroll; ++u) {
      const int64_t k = k0 + u * step + threadIdx.x;
      zk[u] = k < n ? z[k] : 0.0;
      pk[u] = k < n && !init ? p[k] : 0.0;
    }
    if (first) {  // (the whole block)
      __syncthreads();
      beta = sh;
      first = false;
    }
#pragma unroll
    for (int u = 0; u < kVecUnroll; ++u) {
      const int64_t k = k0 + u * step + threadIdx.x;
      if (k < n) p[k] = init ? zk[u] : zk[u] + beta * pk[u];
    }
  }
}

__global__ void k_stamp(unsigned long long* stamps, const int* ctr, int cap, int k, int after) {
  unsigned long long t;
  asm volatile("mov.u64 %0, %%globaltimer;" : "=l"(t));
  const int slot = *ctr - after;
  if (slot >= 0 && slot < cap) stamps[(int64_t)slot * 8 + k] = t;
}

__global__ void __launch_bounds__(kThreads) k_dot(int64_t n, const double* __restrict__ a,
                                                  const double* __restrict__ b, DotSite ds) {
  double acc = 0.0;
  for (int64_t k = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; k < n; k += (int64_t)gridDim.x * blockDim.x)
    acc += a[k] * b[k];
  finish_dots(acc, 0.0, false, ds);
}

__global__ void k_axpby(int64_t n, double alpha, const double* __restrict__ a, double beta,
                        const double* __restrict__ b, double* __restrict__ out) {
  for (int64_t k = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; k < n; k += (int64_t)gridDim.x * blockDim.x)
    out[k] = alpha * a[k] + (b ? beta * b[k] : 0.0);
}

__global__ void k_gather(int64_t n, const int32_t* __restrict__ idx, const double* __restrict__ src,
                         double* __restrict__ dst) {
  for (int64_t k = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; k < n; k += (int64_t)gridDim.x * blockDim.x)
    dst[k] = src[idx[k]];
}

__global__ void k_gather64(int64_t n, const int64_t* __restrict__ idx, const double* __restrict__ src,
                           double* __restrict__ dst) {
  for (int64_t k = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; k < n; k += (int64_t)gridDim.x * blockDim.x) {
    const int64_t t = idx[k];
    dst[k] = t >= 0 ? src[t] : 0.0;
  }
}

__global__ void k_scatter_idx(int64_t n, const int32_t* __restrict__ i32, const int64_t* __restrict__ i64,
                              const double* __restrict__ src, double* __restrict__ dst, int accumulate) {
  for (int64_t k = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; k < n; k += (int64_t)gridDim.x * blockDim.x) {
    const int64_t t = i32 ? (int64_t)i32[k] : i64[k];
    dst[t] = accumulate ? dst[t] + src[k] : src[k];
  }
}

__global__ void k_fill(int64_t n, double v, double* __restrict__ out) {
  for (int64_t k = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; k < n; k += (int64_t)gridDim.x * blockDim.x)
    out[k] = v;
}

// z_j = sum over the copies of column j in the subdomains (ascending subdomain order)
//     + sum_t Zbar_{part[j]}[t, jj(j)] y0[coff + t]          (coarse prolongation)
__global__ void __launch_bounds__(kThreads) k_scatter(ScatterArgs a) {
  double acc_rz = 0.0, acc_rzo = 0.0;
  for (int64_t j = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; j < a.n; j += (int64_t)gridDim.x * blockDim.x) {
    double z = 0.0;
    if (a.add_coarse_only != 1) {
      for (int64_t e = a.map_ptr[j]; e < a.map_ptr[j + 1]; ++e)
        if (in_range(a.map_idx[e], a.total_local, a.err)) z += a.y[a.map_idx[e]];
    }
    if (a.coarse && a.add_coarse_only != 2) {
      const int i = a.part[j];
      const int c0 = a.coff[i], k = a.coff[i + 1] - c0;
      const int64_t nIi = a.nI[i];
      const double* Zi = a.Z + a.zoff[i] + a.jj_of[j];
      int t = 0;
      // Four basis entries loaded ahead of their products: one chain of dependent loads per
      // entry bound the launch (37k columns, basis of 464: 12.7 us, 17.0 one at a time; 102k
      // columns: 15.1 against 21.4; a million columns: 67.6 against 77).
      for (; t + 3 < k; t += 4) {
        double v[4], y[4];
#pragma unroll
        for (int u = 0; u < 4; ++u) {
          v[u] = __ldg(Zi + (t + u) * nIi);
          y[u] = __ldg(a.y0 + c0 + t + u);
        }
#pragma unroll
        for (int u = 0; u < 4; ++u) z += v[u] * y[u];
      }
      for (; t < k; ++t) z += __ldg(Zi + t * nIi) * __ldg(a.y0 + c0 + t);
    }
    a.z[j] = z;
    if (a.dots.parts) {
      acc_rz += a.r[j] * z;
      if (a.r_old) acc_rzo += a.r_old[j] * z;
    }
  }
  if (a.dots.parts) finish_dots(acc_rz, acc_rzo, a.r_old != nullptr, a.dots);
}

// r0[c0 + t] = sum_jj Zbar_i[t, jj] v[Omega_I,i[jj]]: the coarse restriction R_0 v.  A block
// takes four vectors of one subdomain (blockIdx.y), its threads stride the columns: each
// gathered v entry is used four times and five loads per step are independent.  (One block
// per subdomain with a warp per vector, its gathers on one dependent chain, took 25-68 us
// for 25-64 subdomains of 1,600-2,304 columns, where this is a few.)
constexpr int kRestrictVecs = 4;
__global__ void __launch_bounds__(kThreads) k_restrict(const int64_t* __restrict__ int_off,
                                                       const int32_t* __restrict__ int_glob,
                                                       const int64_t* __restrict__ zoff,
                                                       const int32_t* __restrict__ coff, const double* __restrict__ Z,
                                                       const double* __restrict__ v, double* __restrict__ r0) {
  __shared__ double red[kWarps][kRestrictVecs];
  const int i = blockIdx.x, t0 = blockIdx.y * kRestrictVecs;
  const int c0 = coff[i], kk = coff[i + 1] - c0;
  if (t0 >= kk) return;
  const int64_t io = int_off[i];
  const int nIi = (int)(int_off[i + 1] - io);
  const double* Zi = Z + zoff[i];
  const double* row[kRestrictVecs];
#pragma unroll
  for (int u = 0; u < kRestrictVecs; ++u) row[u] = Zi + (int64_t)min(t0 + u, kk - 1) * nIi;
  double acc[kRestrictVecs] = {0.0, 0.0, 0.0, 0.0};
#pragma unroll 2
  for (int jj = threadIdx.x; jj < nIi; jj += kThreads) {
    const double g = v[__ldg(int_glob + io + jj)];
#pragma unroll
    for (int u = 0; u < kRestrictVecs; ++u) acc[u] += __ldg(row[u] + jj) * g;
  }
  const int lane = threadIdx.x & 31, w = threadIdx.x >> 5;
#pragma unroll
  for (int u = 0; u < kRestrictVecs; ++u) {
    const double sum = warp_sum(acc[u]);
    if (lane == 0) red[w][u] = sum;
  }
  __syncthreads();
  if (threadIdx.x < kRestrictVecs && t0 + (int)threadIdx.x < kk) {
    double sum = 0.0;
#pragma unroll
    for (int k = 0; k < kWarps; ++k) sum += red[k][threadIdx.x];
    r0[c0 + t0 + threadIdx.x] = sum;
  }
}

// z = a + b - c with the fused dots r.z (and r_old.z) of the preconditioned residual.
__global__ void __launch_bounds__(kThreads) k_combine3(int64_t n, const double* __restrict__ a,
                                                       const double* __restrict__ b, const double* __restrict__ c,
                                                       double* __restrict__ z, const double* __restrict__ r,
                                                       const double* __restrict__ r_old, DotSite ds) {
  double d1 = 0.0, d2 = 0.0;
  for (int64_t k = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; k < n; k += (int64_t)gridDim.x * blockDim.x) {
    const double v = a[k] + b[k] - c[k];
    z[k] = v;
    if (ds.parts) {
      d1 += r[k] * v;
      if (r_old) d2 += r_old[k] * v;
    }
  }
  if (ds.parts) finish_dots(d1, d2, r_old != nullptr, ds);
}

// The three vector kernels of a preconditioned LSQR step.  The scalars stay on the device, so
// that a step is one fixed sequence of launches (a graph) and the host waits once, for the
// report; square roots and quotients are one thread's work (formed by every thread they took
// 3-6 us of FP64 issue per launch).  40 thousand columns, 17 steps: 4.08 ms a solve; 5.43 with
// the rotation on the host, two waits and three pageable reads a step.
__global__ void __launch_bounds__(kThreads) k_lsqr_u(int64_t m, const double* __restrict__ state,
                                                     const double* __restrict__ q, double* __restrict__ u, DotSite ds) {
  const double inv_beta = state[L_INVBETA], alpha = state[L_ALPHA];
  double acc = 0.0;
  for (int64_t k = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; k < m; k += (int64_t)gridDim.x * blockDim.x) {
    const double un = q[k] - alpha * (inv_beta * u[k]);
    u[k] = un;
    acc += un * un;
  }
  finish_dots(acc, 0.0, false, ds);
}

__global__ void __launch_bounds__(kThreads) k_lsqr_s(int64_t n, double* __restrict__ state,
                                                     const double* __restrict__ q, double* __restrict__ s) {
  __shared__ double sc[2];
  if (threadIdx.x == 0) {
    const double beta = sqrt(state[L_BETA2]);
    sc[0] = beta > 0.0 ? 1.0 / beta : 0.0;
    sc[1] = beta;
  }
  if (blockIdx.x == 0 && threadIdx.x >= 32 && threadIdx.x < 32 + L_PREV)
    state[L_PREV + threadIdx.x - 32] = state[threadIdx.x - 32];
  __syncthreads();
  const double inv = sc[0], beta = sc[1];
  for (int64_t k = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; k < n; k += (int64_t)gridDim.x * blockDim.x)
    s[k] = q ? s[k] * inv - beta * q[k] : s[k] * inv;
}

__global__ void __launch_bounds__(kThreads) k_lsqr_step(int64_t n, int first, double* __restrict__ state,
                                                        const double* __restrict__ scal, const double* __restrict__ t,
                                                        const double* __restrict__ s, double* __restrict__ v,
                                                        double* __restrict__ q, double* __restrict__ x,
                                                        double* __restrict__ w) {
  __shared__ double sc[3];
  if (threadIdx.x == 0) {
    const double* prev = state + L_PREV;
    const double beta = sqrt(state[L_BETA2]), alpha = sqrt(scal[S_RZ]);
    double phibar = beta, rhobar = alpha, c1 = 0.0, c2 = 0.0;
    if (!first) {  // plane rotation
      const double inv_rho = 1.0 / hypot(prev[L_RHOBAR], beta), c = prev[L_RHOBAR] * inv_rho, sn = beta * inv_rho;
      rhobar = -c * alpha;
      phibar = sn * prev[L_PHIBAR];
      c1 = c * prev[L_PHIBAR] * inv_rho;
      c2 = sn * alpha * inv_rho;
    }
    const bool ok = first || (beta > 0.0 && isfinite(beta) && alpha > 0.0 && isfinite(alpha));
    sc[0] = ok ? 1.0 / alpha : 0.0;
    sc[1] = c1;
    sc[2] = c2;
    if (blockIdx.x == 0) {
      state[L_INVBETA] = 1.0 / beta;
      state[L_ALPHA] = alpha;
      state[L_PHIBAR] = phibar;
      state[L_RHOBAR] = rhobar;
      double* rep = state + L_REP;
      rep[L_REP_ALPHA] = alpha;
      rep[L_REP_BETA] = beta;
      rep[L_REP_ERR] = scal[S_ERR];
      if (first) rep[L_REP_ALPHA0] = alpha;
    }
  }
  __syncthreads();
  const double inv_alpha = sc[0], c1 = sc[1], c2 = sc[2];
  if (inv_alpha == 0.0) return;  // breakdown: the host reads it from the report, x stays
  for (int64_t k = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; k < n; k += (int64_t)gridDim.x * blockDim.x) {
    const double vk = t[k] * inv_alpha;
    v[k] = vk;
    q[k] = s[k] * inv_alpha;
    if (!first) {
      const double wk = w[k];
      x[k] += c1 * wk;
      w[k] = vk - c2 * wk;
    } else {
      w[k] = vk;
    }
  }
}

// RAS prolongation: z_j = a_j + y[own[j]] (a may be null), the local solution of the
// subdomain that owns column j only.
__global__ void __launch_bounds__(kThreads) k_ras_combine(int64_t n, const int64_t* __restrict__ own,
                                                          const double* __restrict__ y, const double* __restrict__ a,
                                                          double* __restrict__ z) {
  for (int64_t j = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; j < n; j += (int64_t)gridDim.x * blockDim.x)
    z[j] = (a ? a[j] : 0.0) + y[own[j]];
}

// One Gram-Schmidt pass (see launch_gs_pass).  A thread keeps its rows: it updates them with
// all columns (eight loads in flight), and the sums that the next pass needs are taken of the
// new values at once.  The sums of eight columns over a warp are formed together, each step
// halving the values a lane holds: nine FP64 adds for eight columns instead of forty (a
// sub-partition issues one FP64 warp instruction per 64 cycles).  A step of the Arnoldi
// process takes three passes and a scaling, eight launches with separate products, sums,
// updates and norm (147 thousand columns, seven steps: 310 us before, 234 now).
constexpr int kGsCols = 8;
__device__ __forceinline__ double warp_sum8(double (&v)[kGsCols]) {  // sum of v[(lane >> 2) & 7] on each lane
  const int lane = threadIdx.x & 31;
#pragma unroll
  for (int h = 4; h > 0; h >>= 1) {
    const bool up = lane & (4 * h);
#pragma unroll
    for (int u = 0; u < h; ++u) {
      const double other = __shfl_xor_sync(0xffffffffu, up ? v[u] : v[u + h], 4 * h);
      v[u] = (up ? v[u + h] : v[u]) + other;
    }
  }
  double s = v[0];
  s += __shfl_xor_sync(0xffffffffu, s, 2);
  s += __shfl_xor_sync(0xffffffffu, s, 1);
  return s;
}

__global__ void __launch_bounds__(kThreads) k_gs_pass(int64_t n, const double* __restrict__ V, int64_t ld, int k,
                                                      const double* __restrict__ coef, double sign, double* w, int next,
                                                      double* part, unsigned* counter, double* __restrict__ out) {
  __shared__ double red[2][kWarps][kGsCols];
  __shared__ bool last;
  const int64_t r0 = (int64_t)blockIdx.x * blockDim.x + threadIdx.x, step = (int64_t)gridDim.x * blockDim.x;
  const int lane = threadIdx.x & 31, wp = threadIdx.x >> 5;
  double nrm = 0.0;
  if (coef) {
    for (int64_t r = r0; r < n; r += step) {
      double acc = 0.0;
      for (int c = 0; c < k; c += kGsCols) {
        double v[kGsCols];
#pragma unroll
        for (int u = 0; u < kGsCols; ++u) v[u] = c + u < k ? __ldg(V + (int64_t)(c + u) * ld + r) : 0.0;
#pragma unroll
        for (int u = 0; u < kGsCols; ++u)
          if (c + u < k) acc += v[u] * __ldg(coef + c + u);
      }
      const double wn = w[r] + sign * acc;
      w[r] = wn;
      if (next == 2) nrm += wn * wn;
    }
  }
  if (next == 0) return;
  const int ncol = next == 2 ? 1 : k;
  for (int c = 0; c < ncol; c += kGsCols) {
    double acc[kGsCols];
#pragma unroll
    for (int u = 0; u < kGsCols; ++u) acc[u] = 0.0;
    if (next == 2) {
      acc[0] = nrm;
    } else {
      for (int64_t r = r0; r < n; r += step) {
        const double wr = w[r];
#pragma unroll
        for (int u = 0; u < kGsCols; ++u)
          if (c + u < k) acc[u] += __ldg(V + (int64_t)(c + u) * ld + r) * wr;
      }
    }
    const double s = warp_sum8(acc);
    double(&rd)[kWarps][kGsCols] = red[(c / kGsCols) & 1];
    if ((lane & 3) == 0) rd[wp][lane >> 2] = s;
    __syncthreads();  // the buffer is written again two chunks on, behind the next barrier
    if (threadIdx.x < kGsCols && c + (int)threadIdx.x < ncol) {
      double t = 0.0;
#pragma unroll
      for (int q = 0; q < kWarps; ++q) t += rd[q][threadIdx.x];
      part[(int64_t)(c + threadIdx.x) * gridDim.x + blockIdx.x] = t;
    }
  }
  __syncthreads();
  if (threadIdx.x == 0) {
    __threadfence();
    last = atomicAdd(counter, 1u) == gridDim.x - 1;
  }
  __syncthreads();
  if (!last) return;
  __threadfence();
  for (int c = wp; c < ncol; c += kWarps) {
    double t = 0.0;
    for (int b = lane; b < (int)gridDim.x; b += 32) t += __ldcg(part + (int64_t)c * gridDim.x + b);
    t = warp_sum(t);
    if (lane == 0) out[c] = t;
  }
  if (threadIdx.x == 0) *counter = 0u;
}

__global__ void __launch_bounds__(kThreads) k_gs_scale(int64_t n, const double* __restrict__ norm2,
                                                       const double* __restrict__ err, double* __restrict__ err_out,
                                                       double* __restrict__ w) {
  __shared__ double sc;  // one thread's square root and quotient (see k_lsqr_s)
  if (threadIdx.x == 0) {
    const double hn = sqrt(*norm2);
    sc = hn > 0.0 && isfinite(hn) ? 1.0 / hn : 0.0;
    if (blockIdx.x == 0) *err_out = *err;
  }
  __syncthreads();
  const double inv = sc;
  if (inv == 0.0) return;
  for (int64_t k = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; k < n; k += (int64_t)gridDim.x * blockDim.x)
    w[k] *= inv;
}

// y0 = X r0 for the dense n0 x n0 coarse inverse (one warp per row).
__global__ void __launch_bounds__(kThreads) k_gemv(int64_t n0, const double* __restrict__ X,
                                                   const double* __restrict__ r0, double* __restrict__ y0) {
  const int lane = threadIdx.x & 31;
  const int64_t wg = ((int64_t)blockIdx.x * blockDim.x + threadIdx.x) >> 5;
  const int64_t nw = ((int64_t)gridDim.x * blockDim.x) >> 5;
  for (int64_t row = wg; row < n0; row += nw) {
    const double* xr = X + row * n0;
    double acc = 0.0;
    for (int64_t c = lane; c < n0; c += 32) acc += __ldg(xr + c) * __ldg(r0 + c);
    acc = warp_sum(acc);
    if (lane == 0) y0[row] = acc;
  }
}

// g[e] (+)= rho_r lam_c - mu_r x_c for every stored entry e = (r, c) of A.
__global__ void __launch_bounds__(kThreads) k_grad_vals(CsrDev A, const double* __restrict__ rho,
                                                        const double* __restrict__ lam,
                                                        const double* __restrict__ mu,
                                                        const double* __restrict__ x, double* __restrict__ g,
                                                        int accumulate) {
  for (int64_t r = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; r < A.m; r += (int64_t)gridDim.x * blockDim.x) {
    const double rr = rho[r], mr = mu[r];
    for (int64_t e = A.row_ptr[r]; e < A.row_ptr[r + 1]; ++e) {
      const int32_t c = A.col[e];
      const double v = rr * lam[c] - mr * x[c];
      g[e] = accumulate ? g[e] + v : v;
    }
  }
}

// One-pass normal product, part 1: one block per row tile (layout in normal_tiles.h).
// The tile's window of p is loaded into shared memory; each warp then takes row slices
// (32 rows, lane l row l, entry k of every lane in one coalesced load) and leaves
// s_j = a_j . p in shared memory; after a barrier each warp takes column slices (32
// window columns) and forms u_c = sum_j a_jc s_j over the tile's rows, written over the p
// window; the window goes to the tile's partial buffer.  Both sums run in storage
// order.  The two sweeps read each stored entry once and gather only from shared memory.
//
// The sweeps are bound by the latency of the entry loads: a warp takes P adjacent slices
// at a time and issues up to 8 entry loads of each before the first FMA, and it loads the
// slice offsets of its next group while the current group's entries are in flight.
// Configurations (option normal_kernel): 512 threads with P = 1, 2, 3, or 1,024 threads
// with P = 1.  Slices are stored heaviest first; each warp starts on the group of its
// index and then claims the next unclaimed group from a shared counter, so the warps
// of a sweep finish close together.

// One sweep over slices [s_begin, s_end): acc = sum_k val[.] * src[idx[.]] per lane; the
// result of slice s goes to dst[(s - s_begin) * 32 + lane] (cid == nullptr) or to
// dst[cid[s * 32 + lane]] (lanes with cid 0xFFFF write nothing).
template <int P, int NT>
__device__ __forceinline__ void normal_sweep(const int64_t* __restrict__ off, const uint16_t* __restrict__ idx,
                                             const double* __restrict__ val, const uint16_t* __restrict__ cid,
                                             int s_begin, int s_end, const double* src, int src_n, double* dst,
                                             int dst_n, int* claim, double* err) {
  const int lane = threadIdx.x & 31;
  const int ng = (s_end - s_begin + P - 1) / P;
  int64_t o[P + 1], no[P + 1];
  auto load_off = [&](int g, int64_t(&oo)[P + 1]) {
#pragma unroll
    for (int q = 0; q <= P; ++q) oo[q] = __ldg(off + min(s_begin + g * P + q, s_end));
  };
  int g = threadIdx.x >> 5;
  if (g < ng) load_off(g, o);
  while (g < ng) {
    int nxt = 0;
    if (lane == 0) nxt = atomicAdd(claim, 1);
    nxt = __shfl_sync(0xffffffffu, nxt, 0);
    int K[P], Kmax = 0;
#pragma unroll
    for (int q = 0; q < P; ++q) {
      K[q] = (int)((o[q + 1] - o[q]) >> 5);
      Kmax = max(Kmax, K[q]);
    }
    double acc[P];
#pragma unroll
    for (int q = 0; q < P; ++q) acc[q] = 0.0;
    const bool more = nxt < ng;
    for (int k0 = 0; k0 < Kmax || k0 == 0; k0 += 8) {
      int c[P][8];
      double v[P][8];
#pragma unroll
      for (int q = 0; q < P; ++q)
#pragma unroll
        for (int u = 0; u < 8; ++u) {
          const bool ok = k0 + u < K[q];
          const int64_t e = o[q] + lane + 32 * (k0 + u);
          c[q][u] = ok ? (int)__ldg(idx + e) : 0;
          v[q][u] = ok ? __ldg(val + e) : 0.0;
        }
      if (k0 == 0 && more) load_off(nxt, no);
#pragma unroll
      for (int q = 0; q < P; ++q)
#pragma unroll
        for (int u = 0; u < 8; ++u)
          if (k0 + u < K[q] && in_range(c[q][u], src_n, err)) acc[q] = fma(v[q][u], src[c[q][u]], acc[q]);
    }
#pragma unroll
    for (int q = 0; q < P; ++q) {
      const int s = s_begin + g * P + q;
      if (s >= s_end) break;
      if (!cid) {
        dst[(s - s_begin) * 32 + lane] = acc[q];
      } else {
        const int c = __ldg(cid + (int64_t)s * 32 + lane);
        if (c != 0xFFFF && in_range(c, dst_n, err)) dst[c] = acc[q];
      }
    }
    if (more) {
#pragma unroll
      for (int q = 0; q <= P; ++q) o[q] = no[q];
    }
    g = nxt;
  }
}

template <int P, int NT>
__global__ void __launch_bounds__(NT, 1) k_normal_tile(NormalTilesDev T, const double* __restrict__ p) {
  extern __shared__ __align__(16) double nsm[];
  __shared__ int claim[2];
  const int t = blockIdx.x;
  if (threadIdx.x == 0) claim[0] = claim[1] = NT / 32;
  const int64_t lo = __ldg(T.lo + t);
  const int W = __ldg(T.wid + t);
  const int a0 = __ldg(T.as0 + t), a1 = __ldg(T.as0 + t + 1);
  const int b0 = __ldg(T.bs0 + t), b1 = __ldg(T.bs0 + t + 1);
  double* pw = nsm;
  double* sv = nsm + ((W + 1) & ~1);
  for (int i = threadIdx.x; i < W; i += NT) pw[i] = __ldg(p + lo + i);
  __syncthreads();
  normal_sweep<P, NT>(T.aoff, T.acol, T.aval, nullptr, a0, a1, pw, W, sv, (a1 - a0) * 32, claim, T.err);
  __syncthreads();
  normal_sweep<P, NT>(T.boff, T.brow, T.bval, T.bcid, b0, b1, sv, (a1 - a0) * 32, pw, W, claim + 1, T.err);
  __syncthreads();
  double* out = T.part + __ldg(T.poff + t);
  for (int i = threadIdx.x; i < W; i += NT) out[i] = pw[i];
}

// Part 2: w_c = sum of the partial windows that hold column c, in tile order (the tiles
// to look at come from the table of each block of kNormalColBlock columns), with the
// fused d . w.
__global__ void __launch_bounds__(kThreads) k_normal_reduce(NormalTilesDev T, double* __restrict__ w,
                                                            const double* __restrict__ d, DotSite ds) {
  double dacc = 0.0;
  for (int64_t c = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; c < T.n; c += (int64_t)gridDim.x * blockDim.x) {
    const int64_t b = c / kNormalColBlock;
    const int t0 = __ldg(T.cb_t0 + b), t1 = __ldg(T.cb_t1 + b);
    double acc = 0.0;
    for (int t = t0; t <= t1; ++t) {
      const int64_t off = c - __ldg(T.lo + t);
      if (off >= 0 && off < __ldg(T.wid + t)) acc += T.part[__ldg(T.poff + t) + off];
    }
    w[c] = acc;
    dacc += (d ? d[c] : acc) * acc;
  }
  if (ds.parts) finish_dots(dacc, 0.0, false, ds);
}

int grid_for(int64_t work, int per_block, int cap) {
  int64_t g = (work + per_block - 1) / per_block;
  if (g < 1) g = 1;
  if (g > cap) g = cap;
  return (int)g;
}

}  // namespace

void launch_spmv_csr(const CsrDev& A, const double* x, double* y, int lanes, int grid, cudaStream_t st) {
  if (lanes == -2) {
    if (grid <= 0) grid = grid_for(A.sell.nslices, kWarps, kMaxGrid);
    k_spmv_sell<<<grid, kThreads, 0, st>>>(A.sell, x, y, nullptr, DotSite{});
    return;
  }
  if (lanes < 0) {
    const int R = lanes == -3 ? 32 : 16;
    if (grid <= 0) grid = grid_for((A.m + R - 1) / R, kWarps, kMaxGrid);
    if (lanes == -3) k_spmv_stream<32, 512><<<grid, kThreads, 0, st>>>(A.m, A.row_ptr, A.col, A.val, x, y, nullptr, DotSite{});
    else k_spmv_stream<16, 768><<<grid, kThreads, 0, st>>>(A.m, A.row_ptr, A.col, A.val, x, y, nullptr, DotSite{});
    return;
  }
  if (grid <= 0) grid = grid_for(A.m * lanes, kThreads, kMaxGrid);
  switch (lanes) {
    case 1: k_spmv_csr<1><<<grid, kThreads, 0, st>>>(A, x, y); break;
    case 2: k_spmv_csr<2><<<grid, kThreads, 0, st>>>(A, x, y); break;
    case 4: k_spmv_csr<4><<<grid, kThreads, 0, st>>>(A, x, y); break;
    case 8: k_spmv_csr<8><<<grid, kThreads, 0, st>>>(A, x, y); break;
    case 16: k_spmv_csr<16><<<grid, kThreads, 0, st>>>(A, x, y); break;
    default: k_spmv_csr<32><<<grid, kThreads, 0, st>>>(A, x, y); break;
  }
}

void launch_product(int64_t rows, const int64_t* ptr, const int32_t* idx, const double* val, const double* x, double* y,
                    int lanes, cudaStream_t st) {
  const int grid = grid_for(rows * lanes, kThreads, kMaxGrid);
  switch (lanes) {
    case 1: k_product<1><<<grid, kThreads, 0, st>>>(rows, ptr, idx, val, x, y); break;
    case 2: k_product<2><<<grid, kThreads, 0, st>>>(rows, ptr, idx, val, x, y); break;
    case 4: k_product<4><<<grid, kThreads, 0, st>>>(rows, ptr, idx, val, x, y); break;
    case 8: k_product<8><<<grid, kThreads, 0, st>>>(rows, ptr, idx, val, x, y); break;
    case 16: k_product<16><<<grid, kThreads, 0, st>>>(rows, ptr, idx, val, x, y); break;
    default: k_product<32><<<grid, kThreads, 0, st>>>(rows, ptr, idx, val, x, y); break;
  }
}

void launch_spmv_csc(const CscDev& At, const double* q, double* w, const double* d, const DotSite& ds, int lanes,
                     int grid, cudaStream_t st) {
  if (lanes == -2) {
    if (grid <= 0) grid = grid_for(At.sell.nslices, kWarps, kMaxGrid);
    k_spmv_sell<<<grid, kThreads, 0, st>>>(At.sell, q, w, d, ds);
    return;
  }
  if (lanes < 0) {
    const int R = lanes == -3 ? 32 : 16;
    if (grid <= 0) grid = grid_for((At.n + R - 1) / R, kWarps, kMaxGrid);
    if (lanes == -3) k_spmv_stream<32, 512><<<grid, kThreads, 0, st>>>(At.n, At.col_ptr, At.row, At.val, q, w, d, ds);
    else k_spmv_stream<16, 768><<<grid, kThreads, 0, st>>>(At.n, At.col_ptr, At.row, At.val, q, w, d, ds);
    return;
  }
  if (grid <= 0) grid = grid_for(At.n * lanes, kThreads, kMaxGrid);
  switch (lanes) {
    case 1: k_spmv_csc<1><<<grid, kThreads, 0, st>>>(At, q, w, d, ds); break;
    case 2: k_spmv_csc<2><<<grid, kThreads, 0, st>>>(At, q, w, d, ds); break;
    case 4: k_spmv_csc<4><<<grid, kThreads, 0, st>>>(At, q, w, d, ds); break;
    case 8: k_spmv_csc<8><<<grid, kThreads, 0, st>>>(At, q, w, d, ds); break;
    case 16: k_spmv_csc<16><<<grid, kThreads, 0, st>>>(At, q, w, d, ds); break;
    default: k_spmv_csc<32><<<grid, kThreads, 0, st>>>(At, q, w, d, ds); break;
  }
}

bool normal_tiles_prepare(const NormalTilesDev& T) {
  const size_t bytes = (size_t)T.smem_doubles * sizeof(double);
  int dev = 0, cap = 0;
  if (cudaGetDevice(&dev) != cudaSuccess) return false;
  if (cudaDeviceGetAttribute(&cap, cudaDevAttrMaxSharedMemoryPerBlockOptin, dev) != cudaSuccess) return false;
  // Each configuration's limit is the device's (less its static shared memory), not this
  // matrix's need: handles of other matrices share the kernels.
  auto allow = [&](const void* fn) {
    cudaFuncAttributes fa{};
    if (cudaFuncGetAttributes(&fa, fn) != cudaSuccess) return false;
    const int dyn = cap - (int)fa.sharedSizeBytes;
    if (bytes > (size_t)dyn) return false;
    return cudaFuncSetAttribute(fn, cudaFuncAttributeMaxDynamicSharedMemorySize, dyn) == cudaSuccess;
  };
  const bool ok = allow((const void*)k_normal_tile<1, 512>) && allow((const void*)k_normal_tile<2, 512>) &&
                  allow((const void*)k_normal_tile<3, 512>) && allow((const void*)k_normal_tile<1, 1024>);
  if (!ok) cudaGetLastError();  // a refused setting leaves no error behind: the two products run instead
  return ok;
}

void launch_normal_tiles(const NormalTilesDev& T, const double* v, double* w, const double* d, const DotSite& ds,
                         cudaStream_t st) {
  const size_t smem = (size_t)T.smem_doubles * sizeof(double);
  if (T.ntiles > 0) {
    switch (T.config) {
      case 2: k_normal_tile<2, 512><<<T.ntiles, 512, smem, st>>>(T, v); break;
      case 3: k_normal_tile<3, 512><<<T.ntiles, 512, smem, st>>>(T, v); break;
      case 4: k_normal_tile<1, 1024><<<T.ntiles, 1024, smem, st>>>(T, v); break;
      default: k_normal_tile<1, 512><<<T.ntiles, 512, smem, st>>>(T, v); break;
    }
  }
  k_normal_reduce<<<grid_for(T.n, kThreads, kVecGrid), kThreads, 0, st>>>(T, w, d, ds);
}

void launch_cg_update(int64_t n, double* scal, const double* p, const double* w, double* x, double* r, double* r_old,
                      const DotSite& rr, int* ctr, double* alpha_hist, int hist_cap, cudaStream_t st) {
  k_cg_update<<<grid_for(n, kThreads, kVecGrid), kThreads, 0, st>>>(n, scal, p, w, x, r, r_old, rr, ctr, alpha_hist,
                                                                    hist_cap);
}

void launch_p_update(int64_t n, double* scal, int* ctr, double* beta_hist, int hist_cap, const double* z, double* p,
                     int init, int flex, const LoopTest* loop, cudaStream_t st) {
  k_p_update<<<grid_for(n, kThreads, kVecGrid), kThreads, 0, st>>>(n, scal, ctr, beta_hist, hist_cap, z, p, init,
                                                                   flex, loop ? *loop : LoopTest{});
}

void launch_stamp(unsigned long long* stamps, const int* ctr, int cap, int k, int after, cudaStream_t st) {
  k_stamp<<<1, 1, 0, st>>>(stamps, ctr, cap, k, after);
}

void launch_dot(int64_t n, const double* a, const double* b, const DotSite& ds, cudaStream_t st) {
  k_dot<<<grid_for(n, kThreads, kVecGrid), kThreads, 0, st>>>(n, a, b, ds);
}

void launch_axpby(int64_t n, double alpha, const double* a, double beta, const double* b, double* out,
                  cudaStream_t st) {
  k_axpby<<<grid_for(n, kThreads, kVecGrid), kThreads, 0, st>>>(n, alpha, a, beta, b, out);
}

void launch_fill(int64_t n, double v, double* out, cudaStream_t st) {
  k_fill<<<grid_for(n, kThreads, kVecGrid), kThreads, 0, st>>>(n, v, out);
}

void launch_gather(int64_t n, const int32_t* idx, const double* src, double* dst, cudaStream_t st) {
  k_gather<<<grid_for(n, kThreads, kVecGrid), kThreads, 0, st>>>(n, idx, src, dst);
}

void launch_gather64(int64_t n, const int64_t* idx, const double* src, double* dst, cudaStream_t st) {
  if (n <= 0) return;
  k_gather64<<<grid_for(n, kThreads, kVecGrid), kThreads, 0, st>>>(n, idx, src, dst);
}

void launch_scatter_idx(int64_t n, const int32_t* idx32, const int64_t* idx64, const double* src, double* dst,
                        int accumulate, cudaStream_t st) {
  k_scatter_idx<<<grid_for(n, kThreads, kVecGrid), kThreads, 0, st>>>(n, idx32, idx64, src, dst, accumulate);
}

void launch_lsqr_u(int64_t m, const double* state, const double* q, double* u, const DotSite& ds, cudaStream_t st) {
  k_lsqr_u<<<grid_for(m, kThreads, kVecGrid), kThreads, 0, st>>>(m, state, q, u, ds);
}

void launch_lsqr_s(int64_t n, double* state, const double* q, double* s, cudaStream_t st) {
  k_lsqr_s<<<grid_for(n, kThreads, kVecGrid), kThreads, 0, st>>>(n, state, q, s);
}

void launch_lsqr_step(int64_t n, int first, double* state, const double* scal, const double* t, const double* s,
                      double* v, double* q, double* x, double* w, cudaStream_t st) {
  k_lsqr_step<<<grid_for(n, kThreads, kVecGrid), kThreads, 0, st>>>(n, first, state, scal, t, s, v, q, x, w);
}

void launch_ras_combine(int64_t n, const int64_t* own, const double* y, const double* a, double* z, cudaStream_t st) {
  k_ras_combine<<<grid_for(n, kThreads, kVecGrid), kThreads, 0, st>>>(n, own, y, a, z);
}

// two rows a thread, up to two blocks per SM of the last block's sums
int multi_dot_grid(int64_t n) { return grid_for(n, kThreads * 2, 304); }

void launch_gs_pass(int64_t n, const double* V, int64_t ld, int k, const double* coef, double sign, double* w, int next,
                    double* part, unsigned* counter, double* out, cudaStream_t st) {
  const int g = next ? multi_dot_grid(n) : grid_for(n, kThreads, kVecGrid);
  k_gs_pass<<<g, kThreads, 0, st>>>(n, V, ld, k, coef, sign, w, next, part, counter, out);
}

void launch_gs_scale(int64_t n, const double* norm2, const double* err, double* err_out, double* w, cudaStream_t st) {
  k_gs_scale<<<grid_for(n, kThreads, kVecGrid), kThreads, 0, st>>>(n, norm2, err, err_out, w);
}

void launch_restrict(int N, int kmax, const int64_t* int_off, const int32_t* int_glob, const int64_t* zoff,
                     const int32_t* coff, const double* Z, const double* v, double* r0, cudaStream_t st) {
  const dim3 grid((unsigned)N, (unsigned)((kmax + kRestrictVecs - 1) / kRestrictVecs));
  if (kmax > 0) k_restrict<<<grid, kThreads, 0, st>>>(int_off, int_glob, zoff, coff, Z, v, r0);
}

void launch_combine3(int64_t n, const double* a, const double* b, const double* c, double* z, const double* r,
                     const double* r_old, const DotSite& ds, cudaStream_t st) {
  k_combine3<<<grid_for(n, kThreads, kVecGrid), kThreads, 0, st>>>(n, a, b, c, z, r, r_old, ds);
}

void launch_scatter(const ScatterArgs& a, cudaStream_t st) {
  k_scatter<<<grid_for(a.n, kThreads, kVecGrid), kThreads, 0, st>>>(a);
}

void launch_gemv(int64_t n0, const double* X, const double* r0, double* y0, cudaStream_t st) {
  if (n0 <= 0) return;
  k_gemv<<<grid_for(n0 * 32, kThreads, 8192), kThreads, 0, st>>>(n0, X, r0, y0);
}

void launch_grad_vals(const CsrDev& A, const double* rho, const double* lam, const double* mu,
                      const double* x, double* g, int accumulate, cudaStream_t st) {
  k_grad_vals<<<grid_for(A.m, kThreads, 8192), kThreads, 0, st>>>(A, rho, lam, mu, x, g, accumulate);
}

}  // namespace lsq
