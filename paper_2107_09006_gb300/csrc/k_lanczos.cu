// Device eigen setup: for every subdomain, the largest eigenpairs of the shifted
// local pencil  D_i C_ii D_i v = lambda (C~_ii + s I) v  (eq. (3.4)).
//
// With C~_ii + s I = L L^T, the pencil is the symmetric standard problem
// T u = lambda u, T = L^{-1} D_i C_ii D_i L^{-T}, v = L^{-T} u (so v is
// (C~_ii + s I)-normalised).  Each subdomain runs a thick-restart Lanczos (Krylov-Schur
// form): full re-orthogonalisation in two Gram-Schmidt passes,
// Rayleigh-Ritz on the projected matrix by parallel cyclic Jacobi, restart on the
// best `keep` Ritz vectors.  Only products and solves are needed (Remark 3.2):
// D C_ii D x = D (C~_ii (D x)) + delta D x, since the interior block of C~_ii equals
// that of C_ii = A(:,Omega)^T A(:,Omega) + delta I.  Every loop is bounded by
// maxit; a subdomain that does not converge reports status 2.
//
// Two forms with the same recurrences: run_lanczos_grid, every stage of a step a kernel over
// all subdomains, where a subdomain's FP64 vector fits the superblock kernel; k_lanczos, one
// CTA per subdomain for the whole iteration, where it does not or memory is short.
#include <algorithm>
#include <vector>

#include "band.cuh"
#include "kernels.h"

namespace lsq {

namespace {

constexpr int kMaxK = 160;  // largest Lanczos basis handled

__device__ __forceinline__ double hash_unit(uint32_t a, uint32_t b) {
  // splitmix-style integer hash of (a, b) mapped to [-1, 1)
  uint64_t z = ((uint64_t)a << 32) ^ (uint64_t)b ^ 0x9E3779B97F4A7C15ull;
  z = (z ^ (z >> 30)) * 0xBF58476D1CE4E5B9ull;
  z = (z ^ (z >> 27)) * 0x94D049BB133111EBull;
  z ^= z >> 31;
  return (double)(z >> 11) * (2.0 / 9007199254740992.0) - 1.0;
}

struct Shared {
  double* x1;  // operator work vector (nb*32)
  double* x2;  // operator output / new Lanczos vector (nb*32)
  double* dt;  // 32*33
  double* tmp; // 32
  double* hs;  // kMaxK projection coefficients
  double* h2;  // kMaxK
  double* cs;  // kMaxK/2 Jacobi cosines
  double* sn;  // kMaxK/2 Jacobi sines
  int* pp; int* qq; int* ord;
  double* red; // kWarps
};

// x2 = T x1, destroying x1: x1 <- L^{-T} x1; x2 = D (C~ (D x1)) + delta D x1; x2 <- L^{-1} x2.
__device__ void apply_T(const EigArgs& a, BandRef B, const uint8_t* isint, int ni, int npad, Shared& s) {
  band_backward<double, double>(a.Bfac, nullptr, a.Bidiag + (int64_t)(B.poff - a.P.blk_poff) * kT, B,
                                s.x1, s.dt, s.tmp);
  for (int k = threadIdx.x; k < npad; k += blockDim.x) {
    const double d = (k < ni && isint[k]) ? 1.0 : 0.0;
    s.x1[k] *= d;
    s.x2[k] = 0.0;
  }
  __syncthreads();
  band_symv<double>(a.Ct, B, s.x1, s.x2);
  for (int k = threadIdx.x; k < npad; k += blockDim.x) {
    const double d = (k < ni && isint[k]) ? 1.0 : 0.0;
    s.x2[k] = d * (s.x2[k] + a.delta[blockIdx.x] * s.x1[k]);
  }
  __syncthreads();
  band_forward<double, double>(a.Bfac, nullptr, a.Bidiag + (int64_t)(B.poff - a.P.blk_poff) * kT, B,
                               s.x2, s.dt, s.tmp);
}

// h[t] = V_t . x for t < nv (one warp per t, two vectors per warp at a time for more
// loads in flight; each sum keeps its order).
__device__ void project(const double* V, int64_t vs, int nv, const double* x, int npad, double* h) {
  const int lane = threadIdx.x & 31, w = threadIdx.x >> 5;
  for (int t = w; t < nv; t += 2 * kWarps) {
    const int t2 = t + kWarps;
    const double* vt = V + t * vs;
    const double* vu = V + (int64_t)min(t2, nv - 1) * vs;
    double acc = 0.0, acc2 = 0.0;
#pragma unroll 4
    for (int k = lane; k < npad; k += 32) {
      const double xk = x[k];
      acc += vt[k] * xk;
      acc2 += vu[k] * xk;
    }
    acc = warp_sum(acc);
    acc2 = warp_sum(acc2);
    if (lane == 0) {
      h[t] = acc;
      if (t2 < nv) h[t2] = acc2;
    }
  }
  __syncthreads();
}

// x -= sum_t V_t h[t]
__device__ void subtract(const double* V, int64_t vs, int nv, const double* h, double* x, int npad) {
  for (int k = threadIdx.x; k < npad; k += blockDim.x) {
    double acc = 0.0;
#pragma unroll 8
    for (int t = 0; t < nv; ++t) acc += V[t * vs + k] * h[t];
    x[k] -= acc;
  }
  __syncthreads();
}

__device__ double norm2(const double* x, int npad, double* red) {
  double acc = 0.0;
  for (int k = threadIdx.x; k < npad; k += blockDim.x) acc += x[k] * x[k];
  return sqrt(block_sum(acc, red));
}

// Eigen-decomposition of the symmetric n x n matrix H (leading block of a K x K
// buffer, upper triangle valid on entry) by parallel cyclic Jacobi (round-robin
// pairs).  On exit diag(H) holds the eigenvalues, S (K x K) the eigenvectors as
// columns, and s.ord the indices sorted by descending eigenvalue.
__device__ void jacobi(double* H, double* S, int K, int n, Shared& s) {
  const int np = n + (n & 1);  // even size; the extra index is an isolated zero
  for (int e = threadIdx.x; e < np * np; e += blockDim.x) {
    const int r = e / np, c = e % np;
    if (r > c && r < n) H[r * K + c] = H[c * K + r];
    if (r >= n || c >= n) H[r * K + c] = 0.0;
    S[r * K + c] = (r == c) ? 1.0 : 0.0;
  }
  __syncthreads();
  const int half = np / 2;
  for (int sweep = 0; sweep < 40; ++sweep) {
    double off = 0.0, dia = 0.0;
    for (int e = threadIdx.x; e < np * np; e += blockDim.x) {
      const int r = e / np, c = e % np;
      const double v = H[r * K + c];
      if (r != c) off += v * v; else dia += v * v;
    }
    off = block_sum(off, s.red);
    dia = block_sum(dia, s.red);
    if (off <= 1e-30 * (dia + off) || off == 0.0) break;
    for (int round = 0; round < np - 1; ++round) {
      for (int k = threadIdx.x; k < half; k += blockDim.x) {
        int p, q;
        if (k == 0) { p = round; q = np - 1; }
        else { p = (round + k) % (np - 1); q = (round - k + np - 1) % (np - 1); }
        if (p > q) { const int t = p; p = q; q = t; }
        const double apq = H[p * K + q];
        double c = 1.0, sn = 0.0;
        if (apq != 0.0) {
          const double app = H[p * K + p], aqq = H[q * K + q];
          const double th = (aqq - app) / (2.0 * apq);
          const double t = (th >= 0 ? 1.0 : -1.0) / (fabs(th) + sqrt(1.0 + th * th));
          c = 1.0 / sqrt(1.0 + t * t);
          sn = t * c;
        }
        s.pp[k] = p; s.qq[k] = q; s.cs[k] = c; s.sn[k] = sn;
      }
      __syncthreads();
      for (int e = threadIdx.x; e < half * np; e += blockDim.x) {
        const int k = e / np, col = e % np;
        const int p = s.pp[k], q = s.qq[k];
        const double c = s.cs[k], sn = s.sn[k];
        const double hp = H[p * K + col], hq = H[q * K + col];
        H[p * K + col] = c * hp - sn * hq;
        H[q * K + col] = sn * hp + c * hq;
      }
      __syncthreads();
      for (int e = threadIdx.x; e < half * np; e += blockDim.x) {
        const int k = e / np, row = e % np;
        const int p = s.pp[k], q = s.qq[k];
        const double c = s.cs[k], sn = s.sn[k];
        const double hp = H[row * K + p], hq = H[row * K + q];
        H[row * K + p] = c * hp - sn * hq;
        H[row * K + q] = sn * hp + c * hq;
        const double sp = S[row * K + p], sq = S[row * K + q];
        S[row * K + p] = c * sp - sn * sq;
        S[row * K + q] = sn * sp + c * sq;
      }
      __syncthreads();
    }
  }
  for (int t = threadIdx.x; t < n; t += blockDim.x) {
    const double th = H[t * K + t];
    int rank = 0;
    for (int u = 0; u < n; ++u) {
      const double tu = H[u * K + u];
      if (tu > th || (tu == th && u < t)) ++rank;
    }
    s.ord[rank] = t;
  }
  __syncthreads();
}

// Vout_t = sum_s Vin_s S[s][ord[t]] for t < cnt.
__device__ void rotate(const double* Vin, double* Vout, int64_t vs, int nv, const double* S, int K,
                       const int* ord, int cnt, int npad) {
  for (int k = threadIdx.x; k < npad; k += blockDim.x) {
    for (int t = 0; t < cnt; ++t) {
      const int col = ord[t];
      double acc = 0.0;
      for (int s2 = 0; s2 < nv; ++s2) acc += Vin[s2 * vs + k] * S[s2 * K + col];
      Vout[t * vs + k] = acc;
    }
  }
  __syncthreads();
}

__global__ void __launch_bounds__(kThreads) k_lanczos(EigArgs a, int use_smem) {
  extern __shared__ __align__(16) unsigned char smem_raw[];
  const int i = blockIdx.x;
  const int64_t o0 = a.P.om_off[i];
  const int ni = (int)(a.P.om_off[i + 1] - o0);
  const int64_t b0 = a.P.blk_off[i];
  const int nb = (int)(a.P.blk_off[i + 1] - b0);
  const int npad = nb * kT;
  const uint8_t* isint = a.P.om_int + o0;
  BandRef B{a.P.blk_tf + b0, a.P.blk_poff + b0, nb};
  const int K = a.Kmax;
  const int64_t vs = a.vstride;

  Shared s;
  double* base = reinterpret_cast<double*>(smem_raw);
  int off = 0;
  if (use_smem) {
    s.x1 = base; s.x2 = base + npad; off = 2 * (int)a.vstride;
  } else {
    s.x1 = a.vec + (int64_t)i * 2 * vs; s.x2 = s.x1 + vs;
  }
  s.dt = base + off; off += kT * 33;
  s.tmp = base + off; off += kT;
  s.hs = base + off; off += kMaxK;
  s.h2 = base + off; off += kMaxK;
  s.cs = base + off; off += kMaxK / 2;
  s.sn = base + off; off += kMaxK / 2;
  s.red = base + off; off += kWarps;
  int* ib = reinterpret_cast<int*>(base + off);
  s.pp = ib; s.qq = ib + kMaxK / 2; s.ord = ib + kMaxK;

  double* V = a.V + (int64_t)i * K * vs;
  double* W = a.V2 + (int64_t)i * K * vs;
  double* H = a.H + (int64_t)i * K * K;
  double* S = a.S + (int64_t)i * K * K;
  const int kw = min(a.kwant_cap, ni);
  const int Keff = min(K, ni);
  const int keep = max(kw, min(a.keep, Keff - 1));

  // deterministic start vector
  for (int k = threadIdx.x; k < npad; k += blockDim.x) V[k] = k < ni ? hash_unit(i, k) + 0.5 : 0.0;
  __syncthreads();
  {
    const double nv0 = norm2(V, npad, s.red);
    for (int k = threadIdx.x; k < npad; k += blockDim.x) V[k] /= nv0;
    __syncthreads();
  }
  int nV = 1, steps = 0, status = 0, nconv = 0, fresh = 1;
  double beta = 0.0;
  for (;;) {
    // expand the newest vector: x2 = T V[nV-1], orthogonalised against V[0..nV)
    const double* vj = V + (int64_t)(nV - 1) * vs;
    for (int k = threadIdx.x; k < npad; k += blockDim.x) s.x1[k] = vj[k];
    __syncthreads();
    apply_T(a, B, isint, ni, npad, s);
    ++steps;
    project(V, vs, nV, s.x2, npad, s.hs);
    subtract(V, vs, nV, s.hs, s.x2, npad);
    project(V, vs, nV, s.x2, npad, s.h2);
    subtract(V, vs, nV, s.h2, s.x2, npad);
    for (int t = threadIdx.x; t < nV; t += blockDim.x) H[t * K + (nV - 1)] = s.hs[t] + s.h2[t];
    double hn = 0.0;
    for (int t = 0; t < nV; ++t) hn += (s.hs[t] + s.h2[t]) * (s.hs[t] + s.h2[t]);
    beta = norm2(s.x2, npad, s.red);
    const bool breakdown = !(beta > 1e-12 * sqrt(hn + beta * beta));
    if (nV < Keff && steps < a.maxit) {
      double* vn = V + (int64_t)nV * vs;
      if (!breakdown) {
        for (int k = threadIdx.x; k < npad; k += blockDim.x) vn[k] = s.x2[k] / beta;
      } else {
        // invariant subspace: continue with a fresh vector orthogonal to V
        for (int k = threadIdx.x; k < npad; k += blockDim.x)
          s.x2[k] = k < ni ? hash_unit(i + 7919u * (uint32_t)(fresh + 1), k) : 0.0;
        ++fresh;
        __syncthreads();
        project(V, vs, nV, s.x2, npad, s.hs);
        subtract(V, vs, nV, s.hs, s.x2, npad);
        project(V, vs, nV, s.x2, npad, s.h2);
        subtract(V, vs, nV, s.h2, s.x2, npad);
        const double nn = norm2(s.x2, npad, s.red);
        for (int k = threadIdx.x; k < npad; k += blockDim.x) vn[k] = s.x2[k] / nn;
        beta = 0.0;
      }
      __syncthreads();
      ++nV;
      continue;
    }
    if (breakdown) beta = 0.0;
    // Rayleigh-Ritz on the nV x nV projected matrix
    __syncthreads();
    jacobi(H, S, K, nV, s);
    nconv = 0;
    const int kk = min(kw, nV);
    {
      const double th0 = fabs(H[s.ord[0] * K + s.ord[0]]);
      for (int t = 0; t < kk; ++t) {
        const double res = beta * fabs(S[(nV - 1) * K + s.ord[t]]);
        if (res <= a.tol * fmax(th0, 1e-300)) ++nconv; else break;
      }
    }
    const bool done = (nconv >= kk) || (nV >= ni) || (steps >= a.maxit);
    const int cnt = done ? kk : keep;
    rotate(V, W, vs, nV, S, K, s.ord, cnt, npad);
    for (int t = threadIdx.x; t < cnt; t += blockDim.x) s.hs[t] = H[s.ord[t] * K + s.ord[t]];
    __syncthreads();
    { double* tsw = V; V = W; W = tsw; }
    if (done) {
      if (nconv < kk && nV < ni) status = 2;
      for (int t = threadIdx.x; t < kk; t += blockDim.x) a.lam[(int64_t)i * a.kwant_cap + t] = s.hs[t];
      // the caller expects the Ritz vectors in its V region
      if (V != a.V + (int64_t)i * K * vs) {
        double* dst = a.V + (int64_t)i * K * vs;
        for (int64_t e = threadIdx.x; e < (int64_t)kk * vs; e += blockDim.x) dst[e] = V[e];
      }
      break;
    }
    // restart: H = diag(theta_0..theta_{keep-1}); the residual direction becomes V[keep]
    for (int e = threadIdx.x; e < K * K; e += blockDim.x) H[e] = 0.0;
    __syncthreads();
    for (int t = threadIdx.x; t < cnt; t += blockDim.x) H[t * K + t] = s.hs[t];
    double* vn = V + (int64_t)cnt * vs;
    if (beta > 0.0) {
      for (int k = threadIdx.x; k < npad; k += blockDim.x) vn[k] = s.x2[k] / beta;
      __syncthreads();
    } else {
      for (int k = threadIdx.x; k < npad; k += blockDim.x)
        s.x2[k] = k < ni ? hash_unit(i + 7919u * (uint32_t)(fresh + 1), k) : 0.0;
      ++fresh;
      __syncthreads();
      project(V, vs, cnt, s.x2, npad, s.hs);
      subtract(V, vs, cnt, s.hs, s.x2, npad);
      project(V, vs, cnt, s.x2, npad, s.h2);
      subtract(V, vs, cnt, s.h2, s.x2, npad);
      const double nn = norm2(s.x2, npad, s.red);
      for (int k = threadIdx.x; k < npad; k += blockDim.x) vn[k] = s.x2[k] / nn;
      __syncthreads();
    }
    nV = cnt + 1;
  }
  if (threadIdx.x == 0) {
    a.nconv[i] = nconv;
    a.steps[i] = steps;
    a.status[i] = status;
  }
}

// ---- the same iteration over the whole GPU ----------------------------------------------------
// k_lanczos keeps a subdomain on one CTA: with 16 subdomains of 1,900 columns, 16 SMs, each
// bound by its two FP64 FMAs per cycle (2 ms a step, 226 ms in all).  Here every stage of a
// step is a kernel over all subdomains: the triangular solves on the clusters of the
// superblock kernel, the product with D C~ D as two sparse products with the subdomain's
// part of A (about 90 multiplications per interior column instead of the 1,088 entries its
// row of the band holds), the re-orthogonalisation on a cluster of eight CTAs per subdomain.
// The recurrences, tolerances, restarts and start vectors are those of k_lanczos.

// Phases of a subdomain: 0 expanding, 1 expansion complete (Rayleigh-Ritz next), 2 done, 3
// restarting (its kept vectors are rotated, the residual direction is to be appended).
struct LzState {
  int* nV; int* steps; int* phase; int* buf; int* fresh;
};
__device__ __forceinline__ LzState lz_state(const LanczosGrid& g, int N) {
  return LzState{g.state, g.state + N, g.state + 2 * N, g.state + 3 * N, g.state + 4 * N};
}
__device__ __forceinline__ double* lz_basis(const EigArgs& a, int i, int buf) {
  return (buf ? a.V2 : a.V) + (int64_t)i * a.Kmax * a.vstride;
}

__global__ void __launch_bounds__(kThreads) k_lz_start(EigArgs a, LanczosGrid g) {
  __shared__ double red[kWarps];
  const int i = blockIdx.x;
  const int ni = (int)(a.P.om_off[i + 1] - a.P.om_off[i]);
  const int npad = (int)(a.P.blk_off[i + 1] - a.P.blk_off[i]) * kT;
  double* V = a.V + (int64_t)i * a.Kmax * a.vstride;
  double* x1 = a.vec + (int64_t)i * 2 * a.vstride;
  double s = 0.0;
  for (int k = threadIdx.x; k < ni; k += kThreads) {
    const double h = hash_unit(i, k) + 0.5;
    s += h * h;
  }
  s = sqrt(block_sum(s, red));
  for (int k = threadIdx.x; k < npad; k += kThreads) {
    V[k] = x1[k] = k < ni ? (hash_unit(i, k) + 0.5) / s : 0.0;
    x1[a.vstride + k] = 0.0;  // (the operator writes entries below n_i only)
  }
  if (threadIdx.x == 0) {
    const LzState t = lz_state(g, a.P.N);
    t.nV[i] = 1; t.steps[i] = 0; t.phase[i] = 0; t.buf[i] = 0; t.fresh[i] = 1;
    a.nconv[i] = 0; a.status[i] = 0;
  }
}

// x2 = D (A_i^T (A_i (D x1))) + delta D x1, A_i the rows of A that touch the subdomain's
// interior columns, restricted to them (= D C~_ii D x1 + delta D x1), in two launches: the
// products of the rows, one thread each, in the order of the rows' lists, and the sums of the
// columns, eight lanes each, through xpos.  Bound by the gathers' latency; one pass that forms
// every row's product once per column that needs it was bound by the FP64 units (16 thousand
// columns of 33 rows of nine entries: 34.6 us, 6.0 and 7.0 so).
__global__ void __launch_bounds__(kThreads) k_lz_rows(EigArgs a, LanczosGrid g) {
  const int* phase = g.state + 2 * a.P.N;
  for (int64_t e = (int64_t)blockIdx.x * kThreads + threadIdx.x; e < g.total_xi; e += (int64_t)gridDim.x * kThreads) {
    const int i = g.xi_sub[e];
    if (phase[i] != 0) continue;
    const double* x1 = a.vec + (int64_t)i * 2 * a.vstride;
    const int32_t r = g.xi[e];
    double s = 0.0;
    const int64_t q1 = g.A.row_ptr[r + 1];
#pragma unroll 4
    for (int64_t q = g.A.row_ptr[r]; q < q1; ++q) {
      const int32_t c = __ldg(g.A.col + q);
      if (__ldg(g.part + c) == i) s += __ldg(g.A.val + q) * x1[__ldg(g.locpos + c)];
    }
    g.rows[e] = s;
  }
}

constexpr int kLzLanes = 8;
__global__ void __launch_bounds__(kThreads) k_lz_cols(EigArgs a, LanczosGrid g) {
  const int sub = threadIdx.x % kLzLanes;
  const int* phase = g.state + 2 * a.P.N;
  const int64_t step = (int64_t)gridDim.x * (kThreads / kLzLanes);
  for (int64_t e0 = (int64_t)blockIdx.x * (kThreads / kLzLanes); e0 < g.total_local; e0 += step) {
    const int64_t e = e0 + threadIdx.x / kLzLanes;
    const bool in = e < g.total_local;
    const int i = in ? a.P.row_sub[e] : 0;
    const bool run = in && phase[i] == 0, inside = run && a.P.om_int[e];
    double y = 0.0;
    if (inside) {
      const int32_t j = a.P.om_glob[e];
      const int64_t t1 = g.At.col_ptr[j + 1];
#pragma unroll 4
      for (int64_t t = g.At.col_ptr[j] + sub; t < t1; t += kLzLanes) y += __ldg(g.At.val + t) * g.rows[__ldg(g.xpos + t)];
    }
#pragma unroll
    for (int o = kLzLanes / 2; o > 0; o >>= 1) y += __shfl_xor_sync(0xffffffffu, y, o);
    if (run && sub == 0) {
      double* x1 = a.vec + (int64_t)i * 2 * a.vstride;
      const int k = (int)(e - a.P.om_off[i]);
      x1[a.vstride + k] = inside ? y + a.delta[i] * x1[k] : 0.0;
    }
  }
}

// xpos: a binary search per entry of A^T.
__global__ void __launch_bounds__(kThreads) k_lz_xpos(EigArgs a, LanczosGrid g) {
  const int lane = threadIdx.x & 31;
  for (int64_t e = ((int64_t)blockIdx.x * kThreads + threadIdx.x) >> 5; e < g.total_local;
       e += ((int64_t)gridDim.x * kThreads) >> 5) {
    if (!a.P.om_int[e]) continue;
    const int i = a.P.row_sub[e];
    const int32_t j = a.P.om_glob[e];
    for (int64_t t = g.At.col_ptr[j] + lane; t < g.At.col_ptr[j + 1]; t += 32) {
      const int32_t r = g.At.row[t];
      int64_t lo = g.xi_off[i], hi = g.xi_off[i + 1] - 1;
      while (lo < hi) {
        const int64_t mid = (lo + hi) >> 1;
        if (g.xi[mid] < r) lo = mid + 1; else hi = mid;
      }
      g.xpos[t] = (int32_t)lo;
    }
  }
}

constexpr int kOrthCluster = 8;
__device__ __forceinline__ void lz_cluster_sync() {
  asm volatile("barrier.cluster.arrive.release.aligned;\n\tbarrier.cluster.wait.acquire.aligned;" ::: "memory");
}
__device__ __forceinline__ double lz_peer(const double* p, int rank) {
  uint32_t r;
  double v;
  asm volatile("mapa.shared::cluster.u32 %0, %1, %2;" : "=r"(r) : "r"((uint32_t)__cvta_generic_to_shared(p)), "r"(rank));
  asm volatile("ld.shared::cluster.f64 %0, [%1];" : "=d"(v) : "r"(r) : "memory");
  return v;
}

// One cluster per subdomain, each CTA an eighth of the entries: x2 orthogonalised twice
// against the basis (h = V^T x2, x2 -= V h), the column of H, the new basis vector (or, at
// the end of an expansion, the residual left in x2); phase 3: the residual direction (or a
// fresh one) appended to the kept vectors.  The ranks' partial sums are read through
// distributed shared memory and added in rank order.
__global__ void __cluster_dims__(kOrthCluster, 1, 1) __launch_bounds__(kThreads) k_lz_orth(EigArgs a, LanczosGrid g) {
  extern __shared__ __align__(16) double lsm[];
  __shared__ double hp[3][kMaxK + 1];  // this rank's partial sums (three places in turn: read by peers after a barrier)
  __shared__ double h1[kMaxK], h2[kMaxK], red[kWarps], bc[2];
  const int i = blockIdx.x / kOrthCluster, rank = blockIdx.x % kOrthCluster;
  const LzState st = lz_state(g, a.P.N);
  const int ph = st.phase[i];
  const bool gave_up = *g.err != 0.0;  // a wait of the sweeps before this launch: every subdomain stops
  if (ph == 1 || ph == 2 || gave_up) {  // (the whole cluster)
    if (gave_up) {
      lz_cluster_sync();  // (every rank has read the phase)
      if (rank == 0 && threadIdx.x == 0) st.phase[i] = 2;
    }
    return;
  }
  const int ni = (int)(a.P.om_off[i + 1] - a.P.om_off[i]);
  const int npad = (int)(a.P.blk_off[i + 1] - a.P.blk_off[i]) * kT;
  const int K = a.Kmax, Keff = min(K, ni);
  const int nV = st.nV[i], steps = st.steps[i] + (ph == 0 ? 1 : 0);
  int fresh = st.fresh[i];
  const int64_t vs = a.vstride;
  double* V = lz_basis(a, i, st.buf[i]);
  double* x1g = a.vec + (int64_t)i * 2 * vs;
  const int sl = (npad / kT + kOrthCluster - 1) / kOrthCluster * kT;
  const int k0 = min(npad, rank * sl), len = min(npad, k0 + sl) - k0;
  double* x = lsm;  // this rank's slice
  const int lane = threadIdx.x & 31, w = threadIdx.x >> 5;
  int turn = 0;
  auto project = [&](double* h) {
    double* mine = hp[turn];
    for (int t = w; t < nV; t += kWarps) {
      const double* vt = V + t * vs + k0;
      double acc = 0.0;
#pragma unroll 4
      for (int k = lane; k < len; k += 32) acc += vt[k] * x[k];
      acc = warp_sum(acc);
      if (lane == 0) mine[t] = acc;
    }
    lz_cluster_sync();
    for (int t = threadIdx.x; t < nV; t += kThreads) {
      double s = 0.0;
#pragma unroll
      for (int r = 0; r < kOrthCluster; ++r) s += lz_peer(&mine[t], r);
      h[t] = s;
    }
    turn = turn == 2 ? 0 : turn + 1;
    __syncthreads();
  };
  auto subtract = [&](const double* h) {
    for (int k = threadIdx.x; k < len; k += kThreads) {
      double acc = 0.0;
      const double* vk = V + k0 + k;
#pragma unroll 8
      for (int t = 0; t < nV; ++t) acc += vk[t * vs] * h[t];
      x[k] -= acc;
    }
    __syncthreads();
  };
  auto norm = [&]() -> double {
    double acc = 0.0;
    for (int k = threadIdx.x; k < len; k += kThreads) acc += x[k] * x[k];
    acc = block_sum(acc, red);
    if (threadIdx.x == 0) hp[turn][kMaxK] = acc;
    lz_cluster_sync();
    double s = 0.0;
#pragma unroll
    for (int r = 0; r < kOrthCluster; ++r) s += lz_peer(&hp[turn][kMaxK], r);
    turn = turn == 2 ? 0 : turn + 1;
    return sqrt(s);
  };
  auto orthogonalise = [&]() {
    project(h1);
    subtract(h1);
    project(h2);
    subtract(h2);
  };
  auto fresh_start = [&]() -> double {  // a new direction orthogonal to the basis: its norm
    for (int k = threadIdx.x; k < len; k += kThreads)
      x[k] = k0 + k < ni ? hash_unit(i + 7919u * (uint32_t)(fresh + 1), k0 + k) : 0.0;
    ++fresh;
    __syncthreads();
    orthogonalise();
    return norm();
  };
  auto append = [&](double scale) {
    double* vn = V + (int64_t)nV * vs + k0;
    for (int k = threadIdx.x; k < len; k += kThreads) vn[k] = x1g[k0 + k] = x[k] / scale;
  };
  for (int k = threadIdx.x; k < len; k += kThreads) x[k] = x1g[vs + k0 + k];
  __syncthreads();
  double beta = 0.0;
  int next = 0;
  if (ph == 0) {
    orthogonalise();
    double* H = a.H + (int64_t)i * K * K;
    if (rank == 0)
      for (int t = threadIdx.x; t < nV; t += kThreads) H[t * K + (nV - 1)] = h1[t] + h2[t];
    if (w == 0) {
      double hn = 0.0;
      for (int t = lane; t < nV; t += 32) hn += (h1[t] + h2[t]) * (h1[t] + h2[t]);
      hn = warp_sum(hn);
      if (lane == 0) bc[0] = hn;
    }
    beta = norm();
    __syncthreads();
    const bool breakdown = !(beta > 1e-12 * sqrt(bc[0] + beta * beta));
    if (nV < Keff && steps < a.maxit) {
      if (!breakdown) append(beta);
      else append(fresh_start());
    } else {
      next = 1;
      if (breakdown) beta = 0.0;
      for (int k = threadIdx.x; k < len; k += kThreads) x1g[vs + k0 + k] = x[k];
    }
  } else {
    beta = g.beta[i];
    if (beta > 0.0) append(beta);
    else append(fresh_start());
  }
  lz_cluster_sync();  // (peers have read this rank's sums; every rank has read the state)
  if (rank == 0 && threadIdx.x == 0) {
    st.steps[i] = steps;
    st.fresh[i] = fresh;
    st.phase[i] = next;
    if (next == 0) st.nV[i] = nV + 1;
    else g.beta[i] = beta;
  }
}

// Rayleigh-Ritz of the subdomains whose expansion is complete: eigenvalues and vectors of the
// projected matrix, convergence count, whether it is done, and the restarted projected matrix.
// The rotations are those of jacobi(), bound by the FP64 units of the SM that makes them (3.7 ms
// for a basis of 58 on one CTA), so a pair of CTAs shares them: rank 0 holds the matrix and
// makes the rotations, rank 1 applies them to the eigenvectors while rank 0 updates the
// matrix.  The update takes two pairs' 2 x 2 block at a time and uses the symmetry (16 FP64
// instructions for its four entries and their mirror images; 32 by rows, then columns), and
// pairs whose entry is so small that all such entries together pass the convergence test are
// left alone (at first most of a Lanczos matrix, near the end most pairs): 1.9 ms so.
constexpr int kMaxHalf = kMaxK / 2, kRitzWarps = (kMaxHalf + 31) / 32;
struct RotMsg {  // the rotations of one round, from rank 0 to rank 1
  int n;         // -1: no more rounds
  int pq[kMaxHalf];
  double c[kMaxHalf], s[kMaxHalf];
};
template <class T>
__device__ __forceinline__ uint32_t lz_remote(const T* p, int rank) {
  uint32_t r;
  asm volatile("mapa.shared::cluster.u32 %0, %1, %2;" : "=r"(r) : "r"((uint32_t)__cvta_generic_to_shared(p)), "r"(rank));
  return r;
}
__device__ __forceinline__ void lz_put(uint32_t at, int v) {
  asm volatile("st.shared::cluster.s32 [%0], %1;" ::"r"(at), "r"(v) : "memory");
}
__device__ __forceinline__ void lz_put(uint32_t at, double v) {
  asm volatile("st.shared::cluster.f64 [%0], %1;" ::"r"(at), "d"(v) : "memory");
}
__device__ __forceinline__ void lz_arrive() {
  __syncwarp();
  asm volatile("barrier.cluster.arrive.release.aligned;" ::: "memory");
}
__device__ __forceinline__ void lz_wait() {
  __syncwarp();
  asm volatile("barrier.cluster.wait.acquire.aligned;" ::: "memory");
}

// Rank 1: S <- S R for every round's rotations R, St = S^T (K x K) in shared memory.  The
// ranks' barrier counts match: one arrive and wait per round and one for the end.
__device__ void ritz_vectors(double* St, int K, int np, RotMsg* msg) {
  for (int e = threadIdx.x; e < np * np; e += kThreads) St[(e / np) * K + e % np] = e / np == e % np ? 1.0 : 0.0;
  for (int turn = 0;; ++turn) {
    lz_arrive();  // the last rotations are applied
    lz_wait();    // the next rotations have come
    const RotMsg& m = msg[turn & 1];
    if (m.n < 0) return;
    for (int e = threadIdx.x; e < m.n * np; e += kThreads) {
      const int k = e / np, row = e - k * np;
      const double c = m.c[k], sn = m.s[k];
      double* a = St + (m.pq[k] & 0xffff) * K + row;
      double* b = St + (m.pq[k] >> 16) * K + row;
      const double sp = *a, sq = *b;
      *a = c * sp - sn * sq;
      *b = sn * sp + c * sq;
    }
  }
}

// Rank 0: the rotations, H <- R^T H R (H np x np in a K x K buffer, upper triangle valid on
// entry) until it is diagonal.
__device__ void ritz_matrix(double* H, int K, int n, int np, RotMsg* msg, double* cs, double* sn, int* pp, int* qq,
                            int (*cnt)[kRitzWarps], double* red) {
  for (int e = threadIdx.x; e < np * np; e += kThreads) {
    const int r = e / np, c = e % np;
    if (r > c && r < n) H[r * K + c] = H[c * K + r];
    if (r >= n || c >= n) H[r * K + c] = 0.0;
  }
  __syncthreads();
  const int half = np / 2;
  int turn = 0;
  for (int sweep = 0; sweep < 40; ++sweep) {
    double off = 0.0, dia = 0.0;
    for (int e = threadIdx.x; e < np * np; e += kThreads) {
      const int r = e / np, c = e % np;
      const double v = H[r * K + c];
      if (r != c) off += v * v; else dia += v * v;
    }
    off = block_sum(off, red);
    dia = block_sum(dia, red);
    if (off <= 1e-30 * (dia + off) || off == 0.0) break;
    const double small = 0.25e-30 * (dia + off) / ((double)np * np);
    for (int round = 0; round < np - 1; ++round, ++turn) {
      RotMsg& out = msg[turn & 1];
      int* count = cnt[turn & 1];
      // The pairs to rotate first, the others from the end, each kind in the order of the pairs
      // (the order decides how a block of two pairs is rounded): a rank within the warp, and
      // the counts of the warps before it.
      const int k = threadIdx.x;
      const bool mine = k < half;
      int p = 0, q = 0;
      bool rot = false;
      double apq = 0.0;
      if (mine) {
        if (k == 0) { p = round; q = np - 1; }
        else { p = (round + k) % (np - 1); q = (round - k + np - 1) % (np - 1); }
        if (p > q) { const int t = p; p = q; q = t; }
        apq = H[p * K + q];
        rot = !(apq * apq <= small);  // (a NaN is rotated, as in jacobi)
      }
      const int w = k >> 5, nw = (half + 31) / 32;
      int before = 0;
      if (w < nw) {
        const unsigned m = __ballot_sync(0xffffffffu, rot);
        before = __popc(m & ((1u << (k & 31)) - 1u));
        if ((k & 31) == 0) count[w] = __popc(m);
      }
      if (nw > 1) {
        __syncthreads();
        for (int v = 0; v < min(w, nw); ++v) before += count[v];
      }
      if (rot) {
        const double app = H[p * K + p], aqq = H[q * K + q];
        const double th = (aqq - app) / (2.0 * apq);
        const double t = (th >= 0 ? 1.0 : -1.0) / (fabs(th) + sqrt(1.0 + th * th));
        const double c = 1.0 / sqrt(1.0 + t * t), s = t * c;
        H[p * K + p] = app - t * apq;
        H[q * K + q] = aqq + t * apq;
        H[p * K + q] = 0.0;
        H[q * K + p] = 0.0;
        pp[before] = p; qq[before] = q; cs[before] = c; sn[before] = s;
        lz_put(lz_remote(&out.pq[before], 1), p | q << 16);
        lz_put(lz_remote(&out.c[before], 1), c);
        lz_put(lz_remote(&out.s[before], 1), s);
      } else if (mine) {
        const int at = half - 1 - (k - before);
        pp[at] = p; qq[at] = q; cs[at] = 1.0; sn[at] = 0.0;
      }
      __syncthreads();
      int na = 0;
      for (int v = 0; v < nw; ++v) na += count[v];
      const int rest = half - na;
      if (threadIdx.x == 0) lz_put(lz_remote(&out.n, 1), na);
      lz_arrive();  // the rotations have gone (and the last ones are read: the wait below)
      const int mixed = na * rest, items = mixed + na * (na - 1) / 2;
      for (int e = threadIdx.x; e < items; e += kThreads) {
        int k, l;  // two different pairs, k < l, the first of them rotated
        if (e < mixed) {
          k = e / rest;
          l = na + e - k * rest;
        } else {
          const int x = e - mixed;  // triangular number: x = l (l - 1) / 2 + k
          l = (int)((1.0f + sqrtf(1.0f + 8.0f * (float)x)) * 0.5f);
          if (l * (l - 1) / 2 > x) --l;
          if (l * (l + 1) / 2 <= x) ++l;
          k = x - l * (l - 1) / 2;
        }
        const int p = pp[k], q = qq[k], u = pp[l], v = qq[l];
        const double ck = cs[k], sk = sn[k], cl = cs[l], sl = sn[l];
        const double a = H[p * K + u], b = H[p * K + v], c = H[q * K + u], d = H[q * K + v];
        const double a1 = ck * a - sk * c, b1 = ck * b - sk * d, c1 = sk * a + ck * c, d1 = sk * b + ck * d;
        const double a2 = cl * a1 - sl * b1, b2 = sl * a1 + cl * b1, c2 = cl * c1 - sl * d1, d2 = sl * c1 + cl * d1;
        H[p * K + u] = a2; H[u * K + p] = a2;
        H[p * K + v] = b2; H[v * K + p] = b2;
        H[q * K + u] = c2; H[u * K + q] = c2;
        H[q * K + v] = d2; H[v * K + q] = d2;
      }
      __syncthreads();
      lz_wait();
    }
  }
  if (threadIdx.x == 0) lz_put(lz_remote(&msg[turn & 1].n, 1), -1);
  lz_arrive();
  lz_wait();
}

__global__ void __cluster_dims__(2, 1, 1) __launch_bounds__(kThreads) k_lz_ritz(EigArgs a, LanczosGrid g) {
  extern __shared__ __align__(16) double M[];  // rank 0: the projected matrix, rank 1: its eigenvectors, transposed
  __shared__ RotMsg msg[2];
  __shared__ double cs[kMaxHalf], sn[kMaxHalf], red[kWarps], th[kMaxK], res[kMaxK];
  __shared__ int pp[kMaxHalf], qq[kMaxHalf], ord[kMaxK], cnt[2][kRitzWarps];
  const int i = blockIdx.x / 2, rank = blockIdx.x % 2;
  const LzState st = lz_state(g, a.P.N);
  if (st.phase[i] != 1) return;  // (both CTAs)
  const int ni = (int)(a.P.om_off[i + 1] - a.P.om_off[i]);
  const int K = a.Kmax, nV = st.nV[i], steps = st.steps[i];
  const int np = nV + (nV & 1);  // even size; the extra index is an isolated zero
  const int kw = min(a.kwant_cap, ni), Keff = min(K, ni);
  const int keep = max(kw, min(a.keep, Keff - 1));
  double* Hg = a.H + (int64_t)i * K * K;
  double* Sg = a.S + (int64_t)i * K * K;
  if (rank == 1) {
    lz_arrive();  // both ranks run: their shared memory may be written
    lz_wait();
    ritz_vectors(M, K, np, msg);
    __syncthreads();
    lz_arrive();  // rank 0 may read the last row
    for (int e = threadIdx.x; e < K * K; e += kThreads) {
      const int r = e / K, c = e % K;
      Sg[e] = r < nV && c < nV ? M[c * K + r] : 0.0;
    }
    lz_wait();
    lz_arrive();  // rank 0 has read it
    lz_wait();
    return;
  }
  for (int e = threadIdx.x; e < K * K; e += kThreads) M[e] = Hg[e];
  __syncthreads();
  lz_arrive();
  lz_wait();
  ritz_matrix(M, K, nV, np, msg, cs, sn, pp, qq, cnt, red);
  for (int t = threadIdx.x; t < nV; t += kThreads) ord[t] = t;
  __syncthreads();
  for (int t = threadIdx.x; t < nV; t += kThreads) {
    const double v = M[t * K + t];
    int r = 0;
    for (int u = 0; u < nV; ++u) {
      const double w = M[u * K + u];
      if (w > v || (w == v && u < t)) ++r;
    }
    ord[r] = t;
  }
  __syncthreads();
  const double beta = g.beta[i];
  const int kk = min(kw, nV);
  lz_arrive();
  lz_wait();
  for (int t = threadIdx.x; t < kk; t += kThreads) res[t] = beta * fabs(lz_peer(&M[ord[t] * K + nV - 1], 1));
  for (int t = threadIdx.x; t < nV; t += kThreads) {
    th[t] = M[ord[t] * K + ord[t]];
    g.ord[(int64_t)i * K + t] = ord[t];
  }
  __syncthreads();
  lz_arrive();
  lz_wait();
  int nconv = 0;
  const double bound = a.tol * fmax(fabs(th[0]), 1e-300);
  while (nconv < kk && res[nconv] <= bound) ++nconv;
  const bool done = nconv >= kk || nV >= ni || steps >= a.maxit;
  const int cntk = done ? kk : keep;
  for (int e = threadIdx.x; e < K * K; e += kThreads) {
    const int r = e / K, c = e % K;
    Hg[e] = (r == c && r < cntk) ? th[r] : 0.0;
  }
  if (done)
    for (int t = threadIdx.x; t < kk; t += kThreads) a.lam[(int64_t)i * a.kwant_cap + t] = th[t];
  if (threadIdx.x == 0) {
    g.rr[i] = cntk;
    g.rr[a.P.N + i] = done ? 1 : 0;
    a.nconv[i] = nconv;
    a.steps[i] = steps;
    if (done && nconv < kk && nV < ni) a.status[i] = 2;
  }
}

// Kept vectors of the other buffer: V'_t = sum_s V_s S[s][ord[t]] (blockIdx.y: 256 entries;
// eight vectors per pass over the basis, their coefficients in shared memory).
constexpr int kRotVecs = 8;
__global__ void __launch_bounds__(kThreads) k_lz_rotate(EigArgs a, LanczosGrid g) {
  __shared__ double co[kMaxK][kRotVecs];
  const int i = blockIdx.x;
  const LzState st = lz_state(g, a.P.N);
  if (st.phase[i] != 1) return;
  const int npad = (int)(a.P.blk_off[i + 1] - a.P.blk_off[i]) * kT;
  const int K = a.Kmax, nV = st.nV[i], cnt = g.rr[i];
  const double* in = lz_basis(a, i, st.buf[i]);
  double* out = lz_basis(a, i, st.buf[i] ^ 1);
  const double* S = a.S + (int64_t)i * K * K;
  const int* ord = g.ord + (int64_t)i * K;
  const int k = blockIdx.y * kThreads + threadIdx.x;
  if (blockIdx.y * kThreads >= npad) return;
  for (int t0 = 0; t0 < cnt; t0 += kRotVecs) {
    __syncthreads();
    for (int e = threadIdx.x; e < nV * kRotVecs; e += kThreads) {
      const int t = t0 + e % kRotVecs;
      co[e / kRotVecs][e % kRotVecs] = t < cnt ? S[(e / kRotVecs) * K + ord[t]] : 0.0;
    }
    __syncthreads();
    if (k < npad) {
      double acc[kRotVecs];
#pragma unroll
      for (int u = 0; u < kRotVecs; ++u) acc[u] = 0.0;
#pragma unroll 4
      for (int s = 0; s < nV; ++s) {
        const double v = in[s * a.vstride + k];
#pragma unroll
        for (int u = 0; u < kRotVecs; ++u) acc[u] += v * co[s][u];
      }
#pragma unroll
      for (int u = 0; u < kRotVecs; ++u)
        if (t0 + u < cnt) out[(int64_t)(t0 + u) * a.vstride + k] = acc[u];
    }
  }
}

__global__ void k_lz_flip(EigArgs a, LanczosGrid g) {
  const LzState st = lz_state(g, a.P.N);
  for (int i = blockIdx.x * blockDim.x + threadIdx.x; i < a.P.N; i += gridDim.x * blockDim.x)
    if (st.phase[i] == 1) {
      st.buf[i] ^= 1;
      st.nV[i] = g.rr[i];
      st.phase[i] = g.rr[a.P.N + i] ? 2 : 3;
    }
}

// Z_i[t, :] = interior entries of L^{-T} U_t (U_t = Ritz vector t); blockIdx.y: the vector,
// or all of them on one CTA when the solve's vector lives in global memory.
__global__ void __launch_bounds__(kThreads) k_eigvec(EigArgs a, const int* __restrict__ buffer,
                                                     const int32_t* __restrict__ coff,
                                                     const int64_t* __restrict__ zoff,
                                                     const int64_t* __restrict__ int_off,
                                                     const int32_t* __restrict__ int_loc, double* __restrict__ Z,
                                                     int use_smem) {
  extern __shared__ __align__(16) unsigned char smem_raw[];
  const int i = blockIdx.x;
  const int64_t b0 = a.P.blk_off[i];
  const int nb = (int)(a.P.blk_off[i + 1] - b0);
  const int npad = nb * kT;
  const int64_t vs = a.vstride;
  double* base = reinterpret_cast<double*>(smem_raw);
  double* x1 = use_smem ? base : a.vec + (int64_t)i * 2 * vs;
  double* dt = base + (use_smem ? vs : 0);
  double* tmp = dt + kT * 33;
  BandRef B{a.P.blk_tf + b0, a.P.blk_poff + b0, nb};
  const double* V = lz_basis(a, i, buffer ? buffer[i] : 0);
  const int k = coff[i + 1] - coff[i];
  const int64_t io = int_off[i];
  const int nIi = (int)(int_off[i + 1] - io);
  for (int t = blockIdx.y; t < k; t += gridDim.y) {
    for (int e = threadIdx.x; e < npad; e += blockDim.x) x1[e] = V[t * vs + e];
    __syncthreads();
    band_backward<double, double>(a.Bfac, nullptr, a.Bidiag + b0 * kT, B, x1, dt, tmp);
    for (int jj = threadIdx.x; jj < nIi; jj += blockDim.x) Z[zoff[i] + (int64_t)t * nIi + jj] = x1[int_loc[io + jj]];
    __syncthreads();
  }
}

}  // namespace

size_t lanczos_smem(int max_nb) {
  const size_t vec = 2 * (size_t)max_nb * kT * sizeof(double);
  const size_t rest = (kT * 33 + kT + 2 * kMaxK + kMaxK + kWarps) * sizeof(double) + 2 * kMaxK * sizeof(int);
  return vec + rest;
}

void launch_lanczos(const EigArgs& a, cudaStream_t st) {
  const size_t full = lanczos_smem((int)(a.vstride / kT));
  const int use = full <= 200 * 1024;
  const size_t sm = use ? full : lanczos_smem(0);
  cudaFuncSetAttribute(k_lanczos, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)sm);
  k_lanczos<<<a.P.N, kThreads, sm, st>>>(a, use);
}

bool run_lanczos_grid(const EigArgs& a, const LanczosGrid& g, cudaStream_t st) {
  const int N = a.P.N, K = a.Kmax;
  SuperArgs bwd = g.fac;
  bwd.src = a.vec; bwd.src_stride = 2 * a.vstride;  // x1 <- L^{-T} x1
  bwd.dst = a.vec; bwd.dst_stride = 2 * a.vstride;
  bwd.skip = g.state + 2 * N;
  bwd.sweeps = 2;
  bwd.R = 1;
  bwd.err = g.err;
  SuperArgs fwd = bwd;
  fwd.src = a.vec + a.vstride;  // x2 <- L^{-1} x2
  fwd.dst = a.vec + a.vstride;
  fwd.sweeps = 1;
  const size_t orth_sm = (size_t)((a.vstride / kT + kOrthCluster - 1) / kOrthCluster * kT) * sizeof(double);
  const size_t ritz_sm = (size_t)K * K * sizeof(double);  // (K <= 160: at most 200 KB)
  if (cudaFuncSetAttribute(k_lz_orth, cudaFuncAttributeMaxDynamicSharedMemorySize, 200 * 1024) != cudaSuccess ||
      cudaFuncSetAttribute(k_lz_ritz, cudaFuncAttributeMaxDynamicSharedMemorySize, 200 * 1024) != cudaSuccess)
    return false;
  auto grid = [](int64_t threads) {
    return (unsigned)std::max<int64_t>(1, std::min<int64_t>((threads + kThreads - 1) / kThreads, 1 << 15));
  };
  const dim3 rot_grid((unsigned)N, (unsigned)((a.vstride + kThreads - 1) / kThreads));
  std::vector<int> phase((size_t)N);
  double err = 0.0;
  k_lz_start<<<N, kThreads, 0, st>>>(a, g);
  k_lz_xpos<<<grid(g.total_local * 32), kThreads, 0, st>>>(a, g);
  int steps = 0, basis = 1;
  for (;;) {
    const int run = std::max(1, std::min(K - basis + 1, a.maxit - steps));
    for (int k = 0; k < run; ++k) {
      if (!launch_local_super(bwd, g.shape, 0, N, g.max_nb, g.optin, st)) return false;
      k_lz_rows<<<grid(g.total_xi), kThreads, 0, st>>>(a, g);
      k_lz_cols<<<grid(g.total_local * kLzLanes), kThreads, 0, st>>>(a, g);
      if (!launch_local_super(fwd, g.shape, 0, N, g.max_nb, g.optin, st)) return false;
      k_lz_orth<<<N * kOrthCluster, kThreads, orth_sm, st>>>(a, g);
    }
    steps += run;
    basis = a.keep + 1;
    k_lz_ritz<<<2 * N, kThreads, ritz_sm, st>>>(a, g);
    k_lz_rotate<<<rot_grid, kThreads, 0, st>>>(a, g);
    k_lz_flip<<<(N + 127) / 128, 128, 0, st>>>(a, g);
    k_lz_orth<<<N * kOrthCluster, kThreads, orth_sm, st>>>(a, g);  // (the restarting ones append their residual)
    if (cudaMemcpyAsync(phase.data(), g.state + 2 * N, sizeof(int) * N, cudaMemcpyDeviceToHost, st) != cudaSuccess ||
        cudaMemcpyAsync(&err, g.err, sizeof(double), cudaMemcpyDeviceToHost, st) != cudaSuccess ||
        cudaStreamSynchronize(st) != cudaSuccess || cudaGetLastError() != cudaSuccess || err != 0.0)
      return false;
    bool all = true;
    for (int p : phase) all = all && p == 2;
    if (all) return true;
  }
}

void launch_eigvec(const EigArgs& a, const int* buffer, int kmax, const int32_t* coff, const int64_t* zoff,
                   const int64_t* int_off, const int32_t* int_loc, double* Z, cudaStream_t st) {
  if (kmax < 1) return;
  const size_t full = ((size_t)a.vstride + kT * 33 + kT) * sizeof(double);
  const int use = full <= 200 * 1024;
  const size_t sm = use ? full : (kT * 33 + kT) * sizeof(double);
  cudaFuncSetAttribute(k_eigvec, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)sm);
  const dim3 grid((unsigned)a.P.N, use ? (unsigned)kmax : 1u);
  k_eigvec<<<grid, kThreads, sm, st>>>(a, buffer, coff, zoff, int_off, int_loc, Z, use);
}

}  // namespace lsq
