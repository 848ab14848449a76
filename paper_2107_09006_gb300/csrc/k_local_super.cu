// Batched local solves over superblocks of four 32-row block rows, each subdomain on one
// CTA or on a cluster of C CTAs: y_i = C_ii^{-1} R_i r for every subdomain in one launch.
//
// Why.  A subdomain's sweep is a chain of dependent block steps.  With 32-row steps the
// chain (barriers, a 32 x 32 product on one warp, the message to the next step) takes
// longer than the step's data: ncu on 16 lone CTAs shows the issue slots 24-36 % used and
// DRAM idle.  Here a step covers 128 rows: the tiles of the factor inside a superblock's
// diagonal are replaced by those of its inverse X = L_ss^{-1} (the same storage: both are
// lower triangular), so a step is two dense products,
//   forward   u_s = r_s - sum_{t < s} L(s, t) v_t,   v_s = X u_s
//   backward  x_s = X^T w_s,   w_t -= L(s, t)^T x_s for t < s
// with a quarter of the barriers, and all 16 warps have tiles in both.
//
// Streaming.  The work is cut into units of 32 rows x UC columns (4 KB: 32 FP32 or 16
// FP64 columns; BF16: 2 KB behind a 16-byte header with the tile's scale, X in FP32).  Every warp
// consumes its own fixed list of units, copied ahead of the dependency chain: loads for
// later steps are in flight across the barriers of the current one.
// FP32 and BF16: the next unit is loaded straight into registers (16 bytes a lane and
// load) as soon as the last one is used, so the factor never passes through shared memory.
// Through a ring of shared-memory slots, written by bulk copies and read back, a 4 KB unit
// took 96 shared-memory wavefronts (32 in, 32 out, 32 for the broadcast vector entries)
// and a 128-row step 4,200-5,200 cycles; from registers it takes about 40.
// FP64: the two FMAs per SM and cycle bound the kernel (256 cycles a unit), and the
// register layout would add half as many FP64 additions in the backward sweep; the units
// go through private rings of shared-memory slots, filled by a producer warp (lane k
// issues the bulk copies of the k-th consumer's list as its slots become free), since a
// warp that issues its own copies holds up the chain while the SM's intake (62 bytes per
// cycle with copies of this size) is used up.
//
// Work split.  The warps form four teams, one per block row of the superblock; the unit
// columns of the row are dealt to the team's warps (of all CTAs of the cluster) by their
// index, so each warp has at most one unit more than the others (dealing whole columns of
// the superblock to warps left half of their time at the barriers).  Forward: a warp adds
// its units' products, the team's sums meet in shared memory.  Backward: team q adds
// L(s, t)^T x_q into its own copy q of the window's sums (a ring over the tile columns),
// each entry written by one warp, and the four copies are added when their superblock is
// reached.  CTAs of a cluster exchange 128-entry vectors through distributed shared memory
// and every rank adds what it receives in rank order, so the result does not depend on
// timing.  In FP32 each rank does the whole X product (cheaper than another exchange); in
// FP64, where the products bound the kernel (two FMAs per SM and cycle), it is split too.
// The messages are asynchronous remote stores that complete a transaction barrier of the
// receiver (a cluster barrier took 1,200 cycles a step); buffers and barriers alternate
// between two places, and a rank is never more than one exchange ahead.
//
// Every wait is bounded; a warp that gives up sets the CTA's flag, later waits and copies
// are skipped, all barriers are still met, and the error slot is set.  The thread that arms the
// message barriers waits on every phase of them itself and stops at the first that does not
// complete: none is armed again while a phase of it is open.
#include <type_traits>

#include "common.cuh"
#include "kernels.h"
#include "tile.cuh"

namespace lsq {

namespace {

constexpr int kQ = kSuperRows;  // block rows of a superblock
constexpr long long kSuperWait = 4000000000ll;  // about two seconds at GB300 clocks
constexpr long long kSuperDrain = 1000000ll;    // about half a millisecond: far above a message's flight

// Test hook of the bounds-checked build (ls_debug_stall): 1 the producer issues no copies, 2 the
// last CTA of a cluster sends no messages, so that the waits for them run out.
#ifdef LS_DEBUG_BOUNDS
int g_super_stall = 0;
__device__ __forceinline__ int stalled(const SuperArgs& a) { return a.stall; }
#else
__device__ __forceinline__ int stalled(const SuperArgs&) { return 0; }
#endif

__device__ __forceinline__ uint32_t s32(const void* p) { return (uint32_t)__cvta_generic_to_shared(p); }
__device__ __forceinline__ void bar_init(uint64_t* bar, uint32_t count) {
  asm volatile("mbarrier.init.shared::cta.b64 [%0], %1;" ::"r"(s32(bar)), "r"(count) : "memory");
}
__device__ __forceinline__ void bar_arrive(uint64_t* bar) {
  asm volatile("mbarrier.arrive.shared::cta.b64 _, [%0];" ::"r"(s32(bar)) : "memory");
}
__device__ __forceinline__ void bar_expect(uint64_t* bar, uint32_t bytes) {
  asm volatile("mbarrier.arrive.expect_tx.shared::cta.b64 _, [%0], %1;" ::"r"(s32(bar)), "r"(bytes) : "memory");
}
__device__ __forceinline__ void copy_unit(void* dst, const void* src, uint32_t bytes, uint64_t* bar) {
  asm volatile("fence.proxy.async.shared::cta;" ::: "memory");
  bar_expect(bar, bytes);
  asm volatile("cp.async.bulk.shared::cluster.global.mbarrier::complete_tx::bytes [%0], [%1], %2, [%3];" ::"r"(s32(dst)),
               "l"(src), "r"(bytes), "r"(s32(bar))
               : "memory");
}
__device__ __forceinline__ bool try_wait(uint64_t* bar, uint32_t parity) {
  uint32_t ok;
  asm volatile(
      "{\n\t.reg .pred p;\n\tmbarrier.try_wait.parity.shared::cta.b64 p, [%1], %2;\n\tselp.u32 %0, 1, 0, p;\n\t}"
      : "=r"(ok)
      : "r"(s32(bar)), "r"(parity)
      : "memory");
  return ok != 0;
}
__device__ __forceinline__ bool test_wait(uint64_t* bar, uint32_t parity) {
  uint32_t ok;
  asm volatile(
      "{\n\t.reg .pred p;\n\tmbarrier.test_wait.parity.shared::cta.b64 p, [%1], %2;\n\tselp.u32 %0, 1, 0, p;\n\t}"
      : "=r"(ok)
      : "r"(s32(bar)), "r"(parity)
      : "memory");
  return ok != 0;
}
// messages from peers: the barrier's phase completes with acquire at cluster scope
__device__ __forceinline__ bool try_msg(uint64_t* bar, uint32_t parity) {
  uint32_t ok;
  asm volatile(
      "{\n\t.reg .pred p;\n\tmbarrier.try_wait.parity.acquire.cluster.shared::cta.b64 p, [%1], %2;\n\t"
      "selp.u32 %0, 1, 0, p;\n\t}"
      : "=r"(ok)
      : "r"(s32(bar)), "r"(parity)
      : "memory");
  return ok != 0;
}
template <bool kMsg>
__device__ __forceinline__ bool bounded_wait(uint64_t* bar, uint32_t parity, volatile int* abort_flag) {
  auto probe = [&]() { return kMsg ? try_msg(bar, parity) : try_wait(bar, parity); };
  if (probe()) return true;
  if (*abort_flag) return false;
  const long long t0 = clock64();
  while (!probe()) {
    if (*abort_flag) return false;
    if (clock64() - t0 > kSuperWait) {
      *abort_flag = 1;
      return false;
    }
  }
  return true;
}
__device__ __forceinline__ void cluster_arrive() {
  __syncwarp();
  asm volatile("barrier.cluster.arrive.release.aligned;" ::: "memory");
}
__device__ __forceinline__ void cluster_wait() {
  __syncwarp();
  asm volatile("barrier.cluster.wait.acquire.aligned;" ::: "memory");
}
// Named barriers: 1 .. Q one team's warps, Q + 1 all consumer warps (0 is the CTA's).
__device__ __forceinline__ void named_barrier(int id, int threads) {
  asm volatile("bar.sync %0, %1;" ::"r"(id), "r"(threads) : "memory");
}
__device__ __forceinline__ int cluster_rank() {
  uint32_t r;
  asm volatile("mov.u32 %0, %%cluster_ctarank;" : "=r"(r));
  return (int)r;
}
__device__ __forceinline__ uint32_t peer(const void* p, int rank) {
  uint32_t r;
  asm volatile("mapa.shared::cluster.u32 %0, %1, %2;" : "=r"(r) : "r"(s32(p)), "r"(rank));
  return r;
}
__device__ __forceinline__ void send(uint32_t a, float v, uint32_t bar) {
  asm volatile("st.async.weak.shared::cluster.mbarrier::complete_tx::bytes.b32 [%0], %1, [%2];" ::"r"(a),
               "r"(__float_as_uint(v)), "r"(bar)
               : "memory");
}
__device__ __forceinline__ void send(uint32_t a, double v, uint32_t bar) {
  asm volatile("st.async.weak.shared::cluster.mbarrier::complete_tx::bytes.b64 [%0], %1, [%2];" ::"r"(a),
               "l"(__double_as_longlong(v)), "r"(bar)
               : "memory");
}

// NR right-hand sides of one vector entry.
template <class TA, int NR>
struct alignas(NR == 1 ? sizeof(TA) : 16) Vec {
  TA a[NR];
  __device__ __forceinline__ Vec& operator+=(const Vec& o) {
#pragma unroll
    for (int n = 0; n < NR; ++n) a[n] += o.a[n];
    return *this;
  }
  __device__ __forceinline__ Vec operator+(const Vec& o) const {
    Vec r = *this;
    r += o;
    return r;
  }
  __device__ __forceinline__ Vec operator-(const Vec& o) const {
    Vec r;
#pragma unroll
    for (int n = 0; n < NR; ++n) r.a[n] = a[n] - o.a[n];
    return r;
  }
  __device__ __forceinline__ void fma(TA t, const Vec& o) {  // += t o
#pragma unroll
    for (int n = 0; n < NR; ++n) a[n] += t * o.a[n];
  }
  __device__ __forceinline__ void clear() {
#pragma unroll
    for (int n = 0; n < NR; ++n) a[n] = 0;
  }
};
template <class TA, int NR>
__device__ __forceinline__ void send(uint32_t at, const Vec<TA, NR>& v, uint32_t bar) {
#pragma unroll
  for (int n = 0; n < NR; ++n) send(at + n * (uint32_t)sizeof(TA), v.a[n], bar);
}

// Units of one storage type: UC columns of 32 rows, U units a tile; a panel tile takes REC
// bytes, a tile of X RECX, a unit UB (of the types that pass through the ring).
template <class TF> struct Unit;
template <> struct Unit<double> { static constexpr int UC = 16, U = 2, REC = 8192, RECX = 8192, UB = 4096; };
template <> struct Unit<float> { static constexpr int UC = 32, U = 1, REC = 4096, RECX = 4096, UB = 4096; };
template <> struct Unit<__nv_bfloat16> { static constexpr int UC = 32, U = 1, REC = 2064, RECX = 4096, UB = 4096; };

// Shared memory: [NW][depth] unit slots | full, empty barriers [NW][depth], message
// barriers [6], abort flag | red [NW][32] | ub [Q][32] | ws [1 or 2][Q][32] | dbuf [1 or 2][kItems][32] |
// xbuf [2][C][Q][32] (C > 1) | acc4 [Q][ring][32] | v [nb][32] | tf [nb], toff [nb].
template <class TF, class V, int NW, int C>
struct Layout {
  static constexpr int kItems = Unit<TF>::U * kQ * (kQ + 1) / 2;
  // (a cluster's FP64 X shares and its w_s alternate between two places)
  static constexpr int kRed = NW * 32, kUb = kQ * 32, kWs = (C > 1 ? 2 : 1) * kQ * 32,
                       kDb = (C > 1 && sizeof(TF) == 8 ? 2 : 1) * kItems * 32,
                       kXb = C > 1 ? 2 * C * kQ * 32 : 0;
  // (depth 0: no ring, the units are loaded into registers)
  __host__ __device__ static size_t bars(int depth) { return (size_t)NW * depth * Unit<TF>::UB; }
  __host__ __device__ static size_t red(int depth) { return bars(depth) + (size_t)(2 * NW * depth + 6 + 2) * 8; }
  __host__ __device__ static size_t total(int depth, int nb, int ring) {
    return red(depth) + (size_t)(kRed + kUb + kWs + kDb + kXb + kQ * ring * 32 + nb * kT) * sizeof(V) +
           (size_t)2 * nb * 4;
  }
};

// The units of one warp in the order it consumes them, named by their unit column u of the
// warp's block row b = s Q + q: panel columns u = cls, cls + ST, ... below U s Q, columns
// of X u = U s Q + clx, + SX, ... below U (b + 1).
template <class K, int ST, int SX>
struct UnitList {
  static constexpr int U = K::U;
  const int32_t* tf;
  const int32_t* toff;
  int nb, nsb, q, cls, clx;
  int sweeps;  // 1 forward, 2 backward, 3 both
  int64_t back;  // bytes from a unit to its copy for the backward sweep (0: the same)
  int s = 0, sweep = 0, ph = -1, u = 0, end = 0, step = 0;
  int64_t row = 0;  // byte offset that tile column 0 of the row would have, tiles of rec bytes
  int rec = 0;
  __device__ void start() {
    if (!(sweeps & 1)) { sweep = 1; s = nsb - 1; }
    seek();
  }
  __device__ void seek() {  // to the next phase that has a unit
    while (u >= end) {
      if (++ph == 2) {
        ph = 0;
        if (sweep == 0) {
          if (++s == nsb) {
            sweep = (sweeps & 2) ? 1 : 2;
            if (sweep == 2) return;
            s = nsb - 1;
          }
        } else if (--s < 0) {
          sweep = 2;
          return;
        }
      }
      const int b = s * kQ + q;
      if (b >= nb) { u = end = 0; continue; }
      if (ph == sweep) {  // panel (first in the forward sweep, second in the backward one)
        const int lo = U * tf[b];
        u = cls + (lo > cls ? (lo - cls + ST - 1) / ST * ST : 0);
        end = U * s * kQ;
        step = ST;
        rec = K::REC;
        row = (int64_t)toff[b] * 16 - (int64_t)tf[b] * K::REC;
      } else {
        u = U * s * kQ + clx;
        end = U * (b + 1);
        step = SX;
        rec = K::RECX;
        row = (int64_t)toff[b] * 16 + (int64_t)(s * kQ - tf[b]) * K::REC - (int64_t)s * kQ * K::RECX;
      }
    }
  }
  __device__ bool done() const { return sweep == 2; }
  __device__ bool is_x() const { return ph != sweep; }
  __device__ int64_t offset() const { return row + (int64_t)(u / U) * rec + (u % U) * K::UB + (sweep == 1 ? back : 0); }
  __device__ void next() {
    u += step;
    if (u >= end) seek();
  }
};

// ---- products with one unit (T: column-major, 32 rows) ------------------------------------
// Forward: row sums acc += sum_c T(., c) v_c over any number of units, then out() gives the
// lane one row's sum.  Backward: bwd() gives the lane the sum over the rows of T(., c) x for
// one column c of the unit.

// FP64 units in shared memory: lane = row, forward; lane (h, c) sums the rows [16 h, 16 h +
// 16) of column c, backward, 16-byte reads in a lane-rotated order (eight lanes hit eight
// bank groups).
template <int NR>
struct RingUnit {
  using T = double;
  using V = Vec<double, NR>;
  __device__ __forceinline__ RingUnit& X() { return *this; }
  V acc;
  const V* x;
  __device__ __forceinline__ void zero() { acc.clear(); }
  __device__ __forceinline__ void fwd(const unsigned char* unit, const V* v, int lane) {
    const double* t = reinterpret_cast<const double*>(unit) + lane;
    if constexpr (NR == 1) {
      double s0 = 0.0, s1 = 0.0;
#pragma unroll
      for (int c = 0; c < 16; c += 2) {
        const double2 w = *reinterpret_cast<const double2*>(v + c);
        s0 += t[c * 32] * w.x;
        s1 += t[(c + 1) * 32] * w.y;
      }
      acc.a[0] += s0 + s1;
    } else {
#pragma unroll
      for (int c = 0; c < 16; ++c) acc.fma(t[c * 32], v[c]);
    }
  }
  __device__ __forceinline__ V out(int lane, int& r) {
    r = lane;
    return acc;
  }
  __device__ __forceinline__ void load_x(const V* xs, int) { x = xs; }
  __device__ __forceinline__ V bwd(const unsigned char* unit, int lane, int& c) const {
    const double2* t2 = reinterpret_cast<const double2*>(reinterpret_cast<const double*>(unit) + (lane & 15) * 32 + (lane >> 4) * 16);
    V s;
    if constexpr (NR == 1) {
      const double2* x2 = reinterpret_cast<const double2*>(x + (lane >> 4) * 16);
      double s0 = 0.0, s1 = 0.0;
#pragma unroll
      for (int k = 0; k < 8; ++k) {
        const int j = (k + lane) & 7;
        const double2 t = t2[j], y = x2[j];
        s0 += t.x * y.x;
        s1 += t.y * y.y;
      }
      s.a[0] = s0 + s1;
    } else {
      const V* xr = x + (lane >> 4) * 16;
      s.clear();
#pragma unroll
      for (int k = 0; k < 8; ++k) {
        const int j = (k + lane) & 7;
        const double2 t = t2[j];
        s.fma(t.x, xr[2 * j]);
        s.fma(t.y, xr[2 * j + 1]);
      }
    }
    c = lane & 15;
#pragma unroll
    for (int n = 0; n < NR; ++n) s.a[n] += __shfl_xor_sync(0xffffffffu, s.a[n], 16);
    return s;
  }
};

// One step of a transposing sum: the lanes with bit `o` keep the upper half of a[0 .. 2n),
// the others the lower half, each adding what its partner holds of it.
template <int n>
__device__ __forceinline__ void fold(float* a, int o, int lane) {
  const bool hi = lane & o;
#pragma unroll
  for (int k = 0; k < n; ++k) {
    const float give = hi ? a[k] : a[n + k], keep = hi ? a[n + k] : a[k];
    a[k] = keep + __shfl_xor_sync(0xffffffffu, give, o);
  }
}

// FP32 units in registers: load k of lane l holds rows 4 (l % 8) .. + 3 of column 4 k + l / 8.
template <int NR>
struct RegUnit32 {
  using T = float;
  using V = Vec<float, NR>;
  __device__ __forceinline__ RegUnit32& X() { return *this; }
  float4 t[8];
  V acc[4], x[4];
  __device__ __forceinline__ void load(const unsigned char* unit, int lane) {
    const float4* p = reinterpret_cast<const float4*>(unit) + lane;
#pragma unroll
    for (int k = 0; k < 8; ++k) t[k] = __ldcg(p + 32 * k);
  }
  __device__ __forceinline__ void zero() {
#pragma unroll
    for (int k = 0; k < 4; ++k) acc[k].clear();
  }
  __device__ __forceinline__ void fwd(const unsigned char*, const V* v, int lane) {
#pragma unroll
    for (int k = 0; k < 8; ++k) {
      const V w = v[4 * k + (lane >> 3)];
      acc[0].fma(t[k].x, w);
      acc[1].fma(t[k].y, w);
      acc[2].fma(t[k].z, w);
      acc[3].fma(t[k].w, w);
    }
  }
  __device__ __forceinline__ V out(int lane, int& r) {
    V o;
#pragma unroll
    for (int n = 0; n < NR; ++n) {
      float p[4] = {acc[0].a[n], acc[1].a[n], acc[2].a[n], acc[3].a[n]};
      fold<2>(p, 16, lane);
      fold<1>(p, 8, lane);
      o.a[n] = p[0];
    }
    r = 4 * (lane & 7) + ((lane >> 4) & 1) * 2 + ((lane >> 3) & 1);
    return o;
  }
  __device__ __forceinline__ void load_x(const V* xs, int lane) {
    if constexpr (NR == 1) {
      const float4 y = *reinterpret_cast<const float4*>(xs + 4 * (lane & 7));
      x[0].a[0] = y.x; x[1].a[0] = y.y; x[2].a[0] = y.z; x[3].a[0] = y.w;
    } else {
#pragma unroll
      for (int k = 0; k < 4; ++k) x[k] = xs[4 * (lane & 7) + k];
    }
  }
  __device__ __forceinline__ V bwd(const unsigned char*, int lane, int& c) const {
    V o;
#pragma unroll
    for (int n = 0; n < NR; ++n) {
      float p[8];
#pragma unroll
      for (int k = 0; k < 8; ++k)
        p[k] = (t[k].x * x[0].a[n] + t[k].y * x[1].a[n]) + (t[k].z * x[2].a[n] + t[k].w * x[3].a[n]);
      fold<4>(p, 4, lane);
      fold<2>(p, 2, lane);
      fold<1>(p, 1, lane);
      o.a[n] = p[0];
    }
    c = 4 * (lane & 7) + (lane >> 3);
    return o;
  }
};

// BF16 units in registers: load k of lane l holds rows 8 (l % 4) .. + 7 of column 8 k + l / 4.
// The tiles of X are FP32 (RegUnit32 in the same registers).
template <int NR>
struct RegUnit16 {
  using T = __nv_bfloat16;
  using V = Vec<float, NR>;
  RegUnit32<NR> f;
  float sc;
  V acc[8], x[8];
  __device__ __forceinline__ RegUnit32<NR>& X() { return f; }
  __device__ __forceinline__ void load(const unsigned char* unit, int lane) {
    sc = __ldcg(reinterpret_cast<const float*>(unit));
    const float4* p = reinterpret_cast<const float4*>(unit + 16) + lane;
#pragma unroll
    for (int k = 0; k < 4; ++k) f.t[k] = __ldcg(p + 32 * k);
  }
  __device__ __forceinline__ void zero() {
#pragma unroll
    for (int k = 0; k < 8; ++k) acc[k].clear();
  }
  static __device__ __forceinline__ float lo(float w) { return __uint_as_float(__float_as_uint(w) << 16); }
  static __device__ __forceinline__ float hi(float w) { return __uint_as_float(__float_as_uint(w) & 0xffff0000u); }
  __device__ __forceinline__ void fwd(const unsigned char*, const V* v, int lane) {
#pragma unroll
    for (int k = 0; k < 4; ++k) {
      V w = v[8 * k + (lane >> 2)];
#pragma unroll
      for (int n = 0; n < NR; ++n) w.a[n] *= sc;
      const float4 t = f.t[k];
      acc[0].fma(lo(t.x), w); acc[1].fma(hi(t.x), w);
      acc[2].fma(lo(t.y), w); acc[3].fma(hi(t.y), w);
      acc[4].fma(lo(t.z), w); acc[5].fma(hi(t.z), w);
      acc[6].fma(lo(t.w), w); acc[7].fma(hi(t.w), w);
    }
  }
  __device__ __forceinline__ V out(int lane, int& r) {
    V o;
#pragma unroll
    for (int n = 0; n < NR; ++n) {
      float p[8];
#pragma unroll
      for (int k = 0; k < 8; ++k) p[k] = acc[k].a[n];
      fold<4>(p, 16, lane);
      fold<2>(p, 8, lane);
      fold<1>(p, 4, lane);
      o.a[n] = p[0];
    }
    r = 8 * (lane & 3) + ((lane >> 4) & 1) * 4 + ((lane >> 3) & 1) * 2 + ((lane >> 2) & 1);
    return o;
  }
  __device__ __forceinline__ void load_x(const V* xs, int lane) {
    if constexpr (NR == 1) {
      const float4 a = *reinterpret_cast<const float4*>(xs + 8 * (lane & 3));
      const float4 b = *reinterpret_cast<const float4*>(xs + 8 * (lane & 3) + 4);
      x[0].a[0] = a.x; x[1].a[0] = a.y; x[2].a[0] = a.z; x[3].a[0] = a.w;
      x[4].a[0] = b.x; x[5].a[0] = b.y; x[6].a[0] = b.z; x[7].a[0] = b.w;
    } else {
#pragma unroll
      for (int k = 0; k < 8; ++k) x[k] = xs[8 * (lane & 3) + k];
    }
  }
  __device__ __forceinline__ V bwd(const unsigned char*, int lane, int& c) const {
    V o;
#pragma unroll
    for (int n = 0; n < NR; ++n) {
      float p[4];
#pragma unroll
      for (int k = 0; k < 4; ++k) {
        const float4 t = f.t[k];
        p[k] = ((lo(t.x) * x[0].a[n] + hi(t.x) * x[1].a[n]) + (lo(t.y) * x[2].a[n] + hi(t.y) * x[3].a[n])) +
               ((lo(t.z) * x[4].a[n] + hi(t.z) * x[5].a[n]) + (lo(t.w) * x[6].a[n] + hi(t.w) * x[7].a[n]));
      }
      fold<2>(p, 2, lane);
      fold<1>(p, 1, lane);
      o.a[n] = p[0] * sc;
    }
    c = 8 * (lane & 3) + (lane >> 2);
    return o;
  }
};

// Eight right-hand sides on the tensor cores (FP32 factors of the multi right-hand-side path):
// the tile is stored in the order of m16n8k8's A fragments (lane 4 g + t: rows g, g + 8,
// columns t, t + 4 of every 16 x 8 piece), a second copy transposed for the backward sweep, so
// a unit goes from memory into the registers the MMAs read and both sweeps are the same
// product.  The tiles of L are TF32, the vector entries split into a TF32 head and tail; the
// FP32 tiles of X are split too (the tail-tail product, below 2^-22, is left out).  On the
// FP32 units eight right-hand sides take 256 FMAs, 64 shared-memory wavefronts and, backward,
// 56 shuffles a tile; here 16 MMAs and 8 conflict-free reads.
struct MmaUnit32 {
  using T = float;
  using V = Vec<float, 8>;
  struct Exact {  // the tiles of X
    MmaUnit32& u;
    __device__ __forceinline__ void load(const unsigned char* unit, int lane) { u.load(unit, lane); }
    __device__ __forceinline__ void zero() { u.zero(); }
    __device__ __forceinline__ void fwd(const unsigned char*, const V* v, int lane) { u.product<true>(v, lane); }
    __device__ __forceinline__ void load_x(const V* xs, int lane) { u.load_x(xs, lane); }
  };
  __device__ __forceinline__ Exact X() { return Exact{*this}; }
  float4 t[8];  // piece (m, k) in t[4 m + k]
  float d[2][4], e[2][4];
  const V* x;
  __device__ __forceinline__ void load(const unsigned char* unit, int lane) {
    const float4* p = reinterpret_cast<const float4*>(unit) + lane;
#pragma unroll
    for (int k = 0; k < 8; ++k) t[k] = __ldcg(p + 32 * k);
  }
  __device__ __forceinline__ void zero() {
#pragma unroll
    for (int m = 0; m < 2; ++m)
#pragma unroll
      for (int k = 0; k < 4; ++k) d[m][k] = e[m][k] = 0.f;
  }
  static __device__ __forceinline__ uint32_t tf32(float v) {
    uint32_t y;
    asm("cvt.rna.tf32.f32 %0, %1;" : "=r"(y) : "f"(v));
    return y;
  }
  static __device__ __forceinline__ void mma(float c[4], const float4& a, uint32_t b0, uint32_t b1) {
    asm volatile(
        "mma.sync.aligned.m16n8k8.row.col.f32.tf32.tf32.f32 {%0,%1,%2,%3}, {%4,%5,%6,%7}, {%8,%9}, {%0,%1,%2,%3};"
        : "+f"(c[0]), "+f"(c[1]), "+f"(c[2]), "+f"(c[3])
        : "r"(__float_as_uint(a.x)), "r"(__float_as_uint(a.y)), "r"(__float_as_uint(a.z)), "r"(__float_as_uint(a.w)),
          "r"(b0), "r"(b1));
  }
  template <bool kExact>
  __device__ __forceinline__ void product(const V* v, int lane) {
    const float* b = reinterpret_cast<const float*>(v) + (lane & 3) * 8 + (lane >> 2);
#pragma unroll
    for (int k = 0; k < 4; ++k) {
      const float v0 = b[k * 64], v1 = b[k * 64 + 32];
      const uint32_t h0 = tf32(v0), h1 = tf32(v1);
      const uint32_t l0 = tf32(v0 - __uint_as_float(h0)), l1 = tf32(v1 - __uint_as_float(h1));
#pragma unroll
      for (int m = 0; m < 2; ++m) {
        float4 a = t[4 * m + k];
        if constexpr (kExact) {
          const float4 f = a;
          a.x = __uint_as_float(tf32(f.x)); a.y = __uint_as_float(tf32(f.y));
          a.z = __uint_as_float(tf32(f.z)); a.w = __uint_as_float(tf32(f.w));
          const float4 r = make_float4(__uint_as_float(tf32(f.x - a.x)), __uint_as_float(tf32(f.y - a.y)),
                                       __uint_as_float(tf32(f.z - a.z)), __uint_as_float(tf32(f.w - a.w)));
          mma(e[m], r, h0, h1);
        }
        mma(d[m], a, h0, h1);
        mma(e[m], a, l0, l1);
      }
    }
  }
  __device__ __forceinline__ void fwd(const unsigned char*, const V* v, int lane) { product<false>(v, lane); }
  __device__ __forceinline__ void load_x(const V* xs, int) { x = xs; }
};
template <class P> struct IsMma { static constexpr bool v = false; };
template <> struct IsMma<MmaUnit32> { static constexpr bool v = true; };
// A warp's result for the 32 entries at dst: assigned, or added.
template <bool kAdd>
__device__ __forceinline__ void mma_put(const MmaUnit32& u, Vec<float, 8>* dst, int lane) {
  float* o = reinterpret_cast<float*>(dst) + (lane >> 2) * 8 + 2 * (lane & 3);
#pragma unroll
  for (int m = 0; m < 2; ++m)
#pragma unroll
    for (int h = 0; h < 2; ++h) {
      float2* at = reinterpret_cast<float2*>(o + (16 * m + 8 * h) * 8);
      float2 r = make_float2(u.d[m][2 * h] + u.e[m][2 * h], u.d[m][2 * h + 1] + u.e[m][2 * h + 1]);
      if (kAdd) {
        const float2 p = *at;
        r.x += p.x;
        r.y += p.y;
      }
      *at = r;
    }
}

// P: how the units reach the FMAs (RingUnit, RegUnit32, RegUnit16, each for NR right-hand
// sides at a time: blockIdx.y takes the next NR); NW consumer warps, OCC CTAs per SM, C CTAs
// per subdomain.
template <class P, int NR, int NW, int OCC, int C>
__global__ void __launch_bounds__(NW * 32 + (sizeof(typename P::T) == 8 ? 32 : 0), OCC) k_local_super(SuperArgs a) {
  using TF = typename P::T;
  using TA = typename P::V;  // a vector entry: NR values
  using TS = typename std::conditional<sizeof(TF) == 8, double, float>::type;
  using K = Unit<TF>;
  using LY = Layout<TF, TA, NW, C>;
  constexpr bool kMma = IsMma<P>::v;
  constexpr bool kRing = sizeof(TF) == 8;  // (else the units are loaded into registers)
  constexpr int kAll = NW * 32 + (kRing ? 32 : 0);
  constexpr int U = K::U, UC = K::UC;
  constexpr int NT = NW * 32;        // consumer threads
  constexpr int JW = NW / kQ;        // warps of a team
  constexpr int ST = C * JW;         // unit columns of a row are dealt modulo ST
  constexpr bool kSplitX = C > 1 && sizeof(TF) == 8;  // the X products are dealt over the cluster
  constexpr int SX = kSplitX ? ST : JW;
  constexpr int kItems = LY::kItems;
  static_assert(JW * kQ == NW && NW <= 32, "team geometry");
  using List = UnitList<K, ST, SX>;
  extern __shared__ __align__(128) unsigned char sm[];
  const int depth = a.depth;
  uint64_t* full = reinterpret_cast<uint64_t*>(sm + LY::bars(depth));
  uint64_t* empty = full + NW * depth;
  uint64_t* mbar = empty + NW * depth;  // message barriers: [2] partial sums, [2] w_s, [2] X shares
  volatile int* abort_flag = reinterpret_cast<int*>(mbar + 6);
  TA* red = reinterpret_cast<TA*>(sm + LY::red(depth));
  TA* ub = red + LY::kRed;
  TA* ws = ub + LY::kUb;
  TA* dbuf = ws + LY::kWs;
  TA* xbuf = dbuf + LY::kDb;
  TA* acc4 = xbuf + LY::kXb;
  const int ring = a.ring;
  TA* v = acc4 + (size_t)kQ * ring * 32;

  const int rank = C > 1 ? cluster_rank() : 0;
  const int i = a.order[blockIdx.x / C];
  const int tid = threadIdx.x, lane = tid & 31, w = tid >> 5;
  const int64_t o0 = a.om_off[i];
  const int ni = (int)(a.om_off[i + 1] - o0);
  const int64_t g0 = a.blk_off[i];
  const int nb = (int)(a.blk_off[i + 1] - g0);
  if (nb == 0 || (a.skip && a.skip[i] != 0)) return;  // (the whole cluster leaves)
  const int nsb = (nb + kQ - 1) / kQ;
  int32_t* tf = reinterpret_cast<int32_t*>(v + (size_t)nb * kT);
  int32_t* toff = tf + nb;
  const int64_t base = a.toff[g0];
  const unsigned char* fac = a.fac + base;
  for (int k = tid; k < nb; k += kAll) {
    tf[k] = a.tf[g0 + k];
    toff[k] = (int32_t)((a.toff[g0 + k] - base) >> 4);
  }
  for (int k = tid; k < 2 * NW * depth + 6; k += kAll) bar_init(&full[k], 1);
  if (tid == 0) *abort_flag = 0;
  asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
  __syncthreads();
  if (C > 1) cluster_arrive();  // (this CTA's barriers may be used by its peers)

  if (kRing && w == NW) {
    // ---- producer: lane k streams the units of consumer warp k, in its order ----------------
    if (lane < NW) {
      const int q = lane / JW, jq = (lane % JW + q) % JW, cls = rank + C * jq;
      List l{tf, toff, nb, nsb, q, cls, kSplitX ? cls : jq, a.sweeps, a.back};
      unsigned char* slots = sm + (size_t)lane * depth * K::UB;
      uint64_t* fb = full + lane * depth;
      uint64_t* eb = empty + lane * depth;
      l.start();
      int slot = 0, used = 0;  // used: slots filled so far, at most depth
      uint32_t par = 1;        // parity of the empty phase a slot waits for (0 after the first wrap)
      int64_t issued = 0;
      long long t0 = clock64();
      while (!l.done() && !*abort_flag && stalled(a) != 1) {
        if (used < depth || test_wait(&eb[slot], par)) {
          if (in_range(base + l.offset(), a.fac_bytes, a.err))
            copy_unit(slots + (size_t)slot * K::UB, fac + l.offset(), K::UB, &fb[slot]);
          else
            *abort_flag = 1;  // (bounds-checked build: not issued)
          if (used < depth) ++used;
          ++issued;
          if (++slot == depth) { slot = 0; par ^= 1u; }
          l.next();
          t0 = clock64();
        } else if (clock64() - t0 > 2 * kSuperWait) {
          *abort_flag = 1;
        }
      }
      // every copy has landed before the CTA's shared memory is released (they have, unless a
      // wait gave up)
      for (int64_t k = issued > depth ? issued - depth : 0; k < issued; ++k) {
        const long long t1 = clock64();
        while (!test_wait(&fb[k % depth], (uint32_t)((k / depth) & 1)) && clock64() - t1 < kSuperWait) {
        }
      }
    }
    __syncwarp();
  } else {
    // ---- consumers ----------------------------------------------------------------------------
    const int q = w / JW, j = w % JW;  // team (block row of the superblock), warp of the team
    // (the teams deal their columns to warps one further on: a warp with one unit more than the
    // others then sits in another sub-partition of the SM in every team)
    const int jq = (j + q) % JW, cls = rank + C * jq, clx = kSplitX ? cls : jq;
    auto first_u = [&](int b) {
      const int lo = U * tf[b];
      return cls + (lo > cls ? (lo - cls + ST - 1) / ST * ST : 0);
    };
    auto team_barrier = [&]() { named_barrier(q + 1, JW * 32); };
    auto all_barrier = [&]() { named_barrier(kQ + 1, NT); };
    P p;
    const unsigned char* slots = sm + (size_t)w * depth * K::UB;
    uint64_t* fb = full + w * depth;
    uint64_t* eb = empty + w * depth;
    int slot = 0;
    uint32_t par = 0;
    List l{tf, toff, nb, nsb, q, cls, clx, a.sweeps, a.back};
    auto fetch = [&]() {  // (registers) the next unit of the list
      if constexpr (!kRing)
        if (!l.done()) {
          if (in_range(base + l.offset(), a.fac_bytes, a.err)) {
            if (K::REC != K::RECX && l.is_x()) p.X().load(fac + l.offset(), lane);
            else p.load(fac + l.offset(), lane);
          }
          l.next();
        }
    };
    if constexpr (!kRing) {
      l.start();
      fetch();
    }
    auto acquire = [&]() -> const unsigned char* {  // the next unit of the list has arrived
      if constexpr (kRing) bounded_wait<false>(&fb[slot], par, abort_flag);
      return slots + (size_t)slot * K::UB;
    };
    auto release = [&]() {  // it is used: the next copy may take its place
      if constexpr (kRing) {
        __syncwarp();
        if (lane == 0) bar_arrive(&eb[slot]);
        if (++slot == depth) { slot = 0; par ^= 1u; }
      } else {
        fetch();
      }
    };
    // r(Omega_i), scaled by the equilibration, while the first units load
    const int kb = blockIdx.y * NR;
    for (int k = tid; k < nb * kT; k += NT) {
      TA x;
      x.clear();
      if (a.src) {
        x.a[0] = (TS)a.src[(int64_t)i * a.src_stride + k];
      } else if (k < ni && in_range(a.om_glob[o0 + k], a.n_cols, a.err)) {
        const double* r = a.r + (int64_t)a.om_glob[o0 + k] * a.R + kb;
        const double e = a.eqs[o0 + k];
#pragma unroll
        for (int n = 0; n < NR; ++n)
          if (NR == 1 || kb + n < a.R) x.a[n] = (TS)(r[n] * e);
      }
      v[k] = x;
    }
    for (int k = tid; k < kQ * ring * 32; k += NT) acc4[k].clear();
    if (C > 1) cluster_wait();  // every CTA's barriers are ready
    all_barrier();

    const bool mute = C > 1 && stalled(a) == 2 && rank == C - 1;
    bool live = true;  // every message that this thread waited for has come
    auto message = [&](uint64_t* bar, uint32_t parity) { live = bounded_wait<true>(bar, parity, abort_flag) && live; };
    // ---- forward sweep ------------------------------------------------------------------------
    for (int s = 0; s < nsb && (a.sweeps & 1); ++s) {
      const int b0 = s * kQ, b = b0 + q, lim = U * b0, nr = min(nb - b0, kQ);
      const bool has = b < nb;
      const uint32_t mpar = (uint32_t)((s >> 1) & 1);
      if (C > 1 && tid == 0 && live) {
        bar_expect(&mbar[s & 1], (uint32_t)(nr * 32 * C * sizeof(TA)));
        if (kSplitX) bar_expect(&mbar[4 + (s & 1)], (uint32_t)(U * nr * (nr + 1) / 2 * 32 * sizeof(TA)));
      }
      if (has) {
        p.zero();
        for (int u = first_u(b); u < lim; u += ST) {
          p.fwd(acquire(), v + u * UC, lane);
          release();
        }
        if constexpr (kMma) {
          mma_put<false>(p, red + w * 32, lane);
        } else {
          int row;
          const TA sum = p.out(lane, row);
          red[w * 32 + row] = sum;
        }
        team_barrier();
        if (j == 0) {
          // u_q = r_q - the team's sums (and, in a cluster, the other ranks')
          TA x = red[w * 32 + lane];
#pragma unroll
          for (int k = 1; k < JW; ++k) x += red[(w + k) * 32 + lane];
          if constexpr (C > 1) {
            TA* xb = xbuf + (s & 1) * C * kQ * 32 + q * 32 + lane;
            if (live && !mute)
#pragma unroll
              for (int r = 0; r < C; ++r) send(peer(xb + rank * kQ * 32, r), x, peer(&mbar[s & 1], r));
            message(&mbar[s & 1], mpar);
            x = xb[0];
#pragma unroll
            for (int r = 1; r < C; ++r) x += xb[r * kQ * 32];
          }
          ub[q * 32 + lane] = v[b * 32 + lane] - x;
        }
      }
      all_barrier();
      // v_s = X u_s
      if (has) {
        TA* db = dbuf + ((kSplitX ? (s & 1) * kItems : 0) + U * (q * (q + 1) / 2)) * 32;
        for (int uu = clx; uu < U * (q + 1); uu += SX) {
          p.X().zero();
          p.X().fwd(acquire(), ub + uu * UC, lane);
          release();
          if constexpr (kMma) {
            mma_put<false>(p, db + uu * 32, lane);
            continue;
          } else {
            int row;
            const TA x = p.X().out(lane, row);
            if constexpr (kSplitX) {
              if (live && !mute)
#pragma unroll
                for (int r = 0; r < C; ++r) send(peer(db + uu * 32 + row, r), x, peer(&mbar[4 + (s & 1)], r));
            } else {
              db[uu * 32 + row] = x;
            }
          }
        }
        if (!kSplitX) team_barrier();
        if (j == 0) {
          if (kSplitX) message(&mbar[4 + (s & 1)], mpar);
          TA x = db[lane];
          for (int k = 1; k < U * (q + 1); ++k) x += db[k * 32 + lane];
          v[b * 32 + lane] = x;
        }
      }
      all_barrier();
    }
    // ---- backward sweep -----------------------------------------------------------------------
    for (int s = nsb - 1; s >= 0 && (a.sweeps & 2); --s) {
      const int b0 = s * kQ, b = b0 + q, lim = U * b0, nr = min(nb - b0, kQ);
      const bool has = b < nb;
      const int m = nsb - 1 - s, e = m + ((a.sweeps & 1) ? nsb : 0);  // exchanges so far: of w_s, of X shares
      if (C > 1 && tid == 0 && live) {
        bar_expect(&mbar[2 + (m & 1)], (uint32_t)(nr * 32 * sizeof(TA)));
        if (kSplitX) bar_expect(&mbar[4 + (e & 1)], (uint32_t)(U * nr * (nr + 1) / 2 * UC * sizeof(TA)));
      }
      // w_q = v_q - the teams' sums; in a cluster a unit column's sums are with one rank
      TA* wq = ws + (C > 1 ? (m & 1) * kQ * 32 : 0) + q * 32;
      TA* db = dbuf + (kSplitX ? (e & 1) * kItems * 32 : 0);
      if (has) {
        if (j == 0) {
          TA* ac = acc4 + (size_t)(b % ring) * 32 + lane;
          const TA x = v[b * 32 + lane] - ((ac[0] + ac[(size_t)ring * 32]) +
                                           (ac[(size_t)ring * 64] + ac[(size_t)ring * 96]));
#pragma unroll
          for (int k = 0; k < kQ; ++k) ac[(size_t)k * ring * 32].clear();
          if constexpr (C > 1) {
            if (live && !mute && (U * b + lane / UC) % C == rank)
#pragma unroll
              for (int r = 0; r < C; ++r) send(peer(wq + lane, r), x, peer(&mbar[2 + (m & 1)], r));
          } else {
            wq[lane] = x;
          }
        }
        if (C > 1) message(&mbar[2 + (m & 1)], (uint32_t)((m >> 1) & 1));
        else team_barrier();
        // x_s = X^T w_s: unit (q, uu) gives UC columns of its row's share
        p.X().load_x(wq, lane);
        for (int uu = clx; uu < U * (q + 1); uu += SX) {
          TA* d = db + (U * (q * (q + 1) / 2) + uu) * 32;
          if constexpr (kMma) {
            p.X().zero();
            p.X().fwd(acquire(), wq, lane);
            release();
            mma_put<false>(p, d, lane);
            continue;
          } else {
            int c;
            const TA x = p.X().bwd(acquire(), lane, c);
            release();
            d += c;
            if (lane < UC) {
              if constexpr (kSplitX) {
                if (live && !mute)
#pragma unroll
                  for (int r = 0; r < C; ++r) send(peer(d, r), x, peer(&mbar[4 + (e & 1)], r));
              } else {
                *d = x;
              }
            }
          }
        }
      }
      if (!kSplitX) all_barrier();
      if (has) {
        if (j == 0) {
          if (kSplitX) message(&mbar[4 + (e & 1)], (uint32_t)((e >> 1) & 1));
          // rows p >= q of the superblock reach block q: unit column U q + lane / UC
          const int uu = U * q + lane / UC;
          TA x;
          x.clear();
          for (int p = q; p < nr; ++p) x += db[(U * (p * (p + 1) / 2) + uu) * 32 + (lane & (UC - 1))];
          v[b * 32 + lane] = x;
        }
        team_barrier();
        // the team's sums += L(b, t)^T x_b
        TA* ac = acc4 + (size_t)q * ring * 32;
        p.load_x(v + b * 32, lane);
        for (int u = first_u(b); u < lim; u += ST) {
          if constexpr (kMma) {
            p.zero();
            p.fwd(acquire(), v + b * 32, lane);
            release();
            mma_put<true>(p, ac + (u % ring) * 32, lane);
          } else {
            int c;
            const TA x = p.bwd(acquire(), lane, c);
            release();
            if (lane < UC) ac[((u / U) % ring) * 32 + (u % U) * UC + c] += x;
          }
        }
      }
      all_barrier();
    }
    if (*abort_flag) {
      if (tid == 0 && a.err[0] == 0.0) a.err[0] = kErrTimeout;
    } else if (a.dst) {
      for (int k = rank * NT + tid; k < nb * kT; k += C * NT) a.dst[(int64_t)i * a.dst_stride + k] = (double)v[k].a[0];
    } else {
      for (int k = rank * NT + tid; k < ni; k += C * NT) {
        double* y = a.y + (o0 + k) * a.R + kb;
        const double e = a.eqs[o0 + k];
#pragma unroll
        for (int n = 0; n < NR; ++n)
          if (NR == 1 || kb + n < a.R) y[n] = (double)v[k].a[n] * e;
      }
    }
  }
  if (C > 1) {
    if (kRing && w == NW) cluster_wait();  // (the start's barrier)
    cluster_arrive();             // no CTA leaves while a peer may still write into its shared memory
    cluster_wait();
    // Every message was waited for, unless a wait gave up: then those that peers sent before the
    // barrier may still be on their way, and this CTA's shared memory stays until they have come.
    if (*abort_flag)
      for (const long long t0 = clock64(); clock64() - t0 < kSuperDrain;) {
      }
  }
}

// ---- storage ------------------------------------------------------------------------------

// Tile S (row pitch 33) -> column-major record at dst.
template <class T>
__device__ __forceinline__ void put_tile(const double* S, unsigned char* dst) {
  T* d = reinterpret_cast<T*>(dst);
  for (int e = threadIdx.x; e < 1024; e += blockDim.x) d[e] = (T)S[(e & 31) * 33 + (e >> 5)];
}
// Largest magnitude of the tile (1 if zero), the BF16 tile's scale.
__device__ __forceinline__ double tile_scale(const double* S, double* redm) {
  double mx = 0.0;
  for (int e = threadIdx.x; e < 1024; e += blockDim.x) mx = fmax(mx, fabs(S[(e & 31) * 33 + (e >> 5)]));
  for (int o = 16; o > 0; o >>= 1) mx = fmax(mx, __shfl_xor_sync(0xffffffffu, mx, o));
  if ((threadIdx.x & 31) == 0) redm[threadIdx.x >> 5] = mx;
  __syncthreads();
  double m = 0.0;
  for (int k = 0; k < kWarps; ++k) m = fmax(m, redm[k]);
  __syncthreads();
  return m > 0.0 ? m : 1.0;
}
__device__ __forceinline__ void put_bf16(const double* S, unsigned char* rec, double* redm) {
  const double sc = tile_scale(S, redm);
  if (threadIdx.x < 4) reinterpret_cast<float*>(rec)[threadIdx.x] = threadIdx.x == 0 ? (float)sc : 0.f;
  __nv_bfloat16* d = reinterpret_cast<__nv_bfloat16*>(rec + 16);
  for (int e = threadIdx.x; e < 1024; e += blockDim.x) d[e] = __float2bfloat16_rn((float)(S[(e & 31) * 33 + (e >> 5)] / sc));
}
// The tile as its BF16 storage holds it.
__device__ __forceinline__ void round_bf16(double* S, double* redm) {
  const double sc = tile_scale(S, redm);
  for (int e = threadIdx.x; e < 1024; e += blockDim.x) {
    double& x = S[(e & 31) * 33 + (e >> 5)];
    x = (double)__bfloat162float(__float2bfloat16_rn((float)(x / sc))) * (double)(float)sc;
  }
  __syncthreads();
}

// Where the tiles of a factor come from: load(D, b, t) leaves L(b, t) (zero left of the block
// row's envelope), diag(D, b) L_bb^{-1} in the shared tile D (row pitch 33); both end with a
// barrier.  BandSrc: the FP64 factor as setup leaves it (row-major panels, the inverse diagonal
// tiles apart).  SolveSrc: the solve storage of the 32-row sweeps (column-major panels, the
// inverse diagonal tile last; BF16 with a scale per tile).
struct BandSrc {
  const int32_t* tf; const int64_t* poff; const double* L; const double* dinv;
  __device__ void load(double* D, int64_t g0, int b, int t) const {
    const int t0 = tf[g0 + b];
    const int64_t width = (int64_t)(b - t0 + 1) * kT;
    const double* src = L + poff[g0 + b] + (int64_t)(t - t0) * kT;
    for (int e = threadIdx.x; e < 1024; e += blockDim.x)
      D[(e >> 5) * 33 + (e & 31)] = t < t0 ? 0.0 : src[(int64_t)(e >> 5) * width + (e & 31)];
    __syncthreads();
  }
  __device__ void diag(double* D, int64_t g0, int b) const {
    for (int e = threadIdx.x; e < 1024; e += blockDim.x) D[(e >> 5) * 33 + (e & 31)] = dinv[(g0 + b) * 1024 + e];
    __syncthreads();
  }
};
template <class T>
struct SolveSrc {
  const int32_t* tf; const int64_t* poff; const T* L; const float* tsc;
  __device__ void tile(double* D, int64_t off, bool zero) const {
    const double sc = tsc && !zero ? (double)tsc[off / 1024] : 1.0;
    for (int e = threadIdx.x; e < 1024; e += blockDim.x) {
      double x = 0.0;
      if (!zero) {
        if constexpr (sizeof(T) == 2) x = (double)__bfloat162float(L[off + e]) * sc;
        else x = (double)L[off + e];
      }
      D[(e & 31) * 33 + (e >> 5)] = x;
    }
    __syncthreads();
  }
  __device__ void load(double* D, int64_t g0, int b, int t) const {
    const int t0 = tf[g0 + b];
    tile(D, poff[g0 + b] + (int64_t)(t - t0) * 1024, t < t0);
  }
  __device__ void diag(double* D, int64_t g0, int b) const { tile(D, poff[g0 + b] + (int64_t)(b - tf[g0 + b]) * 1024, false); }
};

// One CTA per superblock: its panel tiles converted, its diagonal tiles replaced by those of
// the inverse, X(t, t) = L_tt^{-1}, X(b, t) = -L_bb^{-1} sum_{t <= k < b} L(b, k) X(k, t), in
// FP64.  BF16: X is that of the factor as rounded to BF16 (the tiles L(b, k) and L_bb^{-1} of
// the 32-row sweeps), kept in FP32: the operator stays the one of BF16 factors.  tf32: the
// tiles L(b, t) are rounded to TF32 first and X is that of the rounded factor: the operator
// of the tensor-core kernels of the multi right-hand-side path.
// frag > 0 (FP32): records in the fragment order of MmaUnit32, and at `frag` bytes from each its
// transposed copy.
__device__ __forceinline__ void put_fragments(const double* S, unsigned char* dst, int64_t frag) {
  float* d = reinterpret_cast<float*>(dst);
  float* b = reinterpret_cast<float*>(dst + frag);
  for (int e = threadIdx.x; e < 1024; e += blockDim.x) {
    const int j = e & 3, lane = (e >> 2) & 31, k = (e >> 7) & 3, m = e >> 9;
    const int r = 16 * m + (lane >> 2) + 8 * (j & 1), c = 8 * k + (lane & 3) + 4 * (j >> 1);
    d[e] = (float)S[r * 33 + c];
    b[e] = (float)S[c * 33 + r];
  }
}
template <class TF, class Src>
__global__ void __launch_bounds__(kThreads) k_super_pack(const int64_t* __restrict__ blk_off, Src src,
                                                         const int32_t* __restrict__ stf,
                                                         const int64_t* __restrict__ stoff, int tf32, int64_t frag,
                                                         unsigned char* __restrict__ dst) {
  using K = Unit<TF>;
  constexpr bool kBf16 = sizeof(TF) == 2;
  using TX = typename std::conditional<kBf16, float, TF>::type;
  __shared__ double X[kQ - 1][kT * 33], P[kT * 33], S[kT * 33];
  __shared__ double redm[kWarps];
  const int i = blockIdx.x, s = blockIdx.y;  // (more than 65,535 subdomains: in x)
  const int64_t g0 = blk_off[i];
  const int nb = (int)(blk_off[i + 1] - g0);
  const int b0 = s * kQ, b1 = min(nb, b0 + kQ);
  if (b0 >= nb) return;
  auto round = [&](double* D) {
    if (kBf16) round_bf16(D, redm);
    if (tf32) {
      for (int e = threadIdx.x; e < 1024; e += blockDim.x) {
        double& x = D[(e >> 5) * 33 + (e & 31)];
        uint32_t y;
        asm("cvt.rna.tf32.f32 %0, %1;" : "=r"(y) : "f"((float)x));
        x = (double)__uint_as_float(y);
      }
      __syncthreads();
    }
  };
  for (int b = b0; b < b1; ++b)
    for (int t = stf[g0 + b]; t < b0; ++t) {
      src.load(S, g0, b, t);
      unsigned char* rec = dst + stoff[g0 + b] + (int64_t)(t - stf[g0 + b]) * K::REC;
      if constexpr (kBf16) {
        put_bf16(S, rec, redm);
      } else {
        round(S);
        if (frag) put_fragments(S, rec, frag);
        else put_tile<TF>(S, rec);
      }
      __syncthreads();
    }
  auto put_x = [&](const double* D, int b, int t) {
    unsigned char* rec = dst + stoff[g0 + b] + (int64_t)(b0 - stf[g0 + b]) * K::REC + (int64_t)(t - b0) * K::RECX;
    if (frag) put_fragments(D, rec, frag);
    else put_tile<TX>(D, rec);
  };
  for (int t = b0; t < b1; ++t) {
    src.diag(X[0], g0, t);
    if (kBf16) round_bf16(X[0], redm);
    put_x(X[0], t, t);
    for (int b = t + 1; b < b1; ++b) {
      for (int e = threadIdx.x; e < kT * 33; e += blockDim.x) S[e] = 0.0;
      for (int k = t; k < b; ++k) {
        src.load(P, g0, b, k);
        round(P);
        tile_mm<false, false>(S, P, X[k - t], -1);
        __syncthreads();
      }
      src.diag(P, g0, b);
      if (kBf16) round_bf16(P, redm);
      // X(b, t) = L_bb^{-1} S; the last row's tile is not needed by a later one: over X(t, t)'s place
      double* out = b - t < kQ - 1 ? X[b - t] : X[0];
      tile_mm<false, false>(out, P, S, 0);
      __syncthreads();
      put_x(out, b, t);
    }
    __syncthreads();
  }
}

template <class P, int NR, int NW, int OCC, int C>
bool launch_impl(SuperArgs a, int N, int max_nb, size_t optin, bool probe, cudaStream_t st) {
  using LY = Layout<typename P::T, typename P::V, NW, C>;
  constexpr bool kRing = sizeof(typename P::T) == 8;
  // OCC CTAs share what the SM holds, 1 KB of each share the system's
  const size_t limit = (optin + 1024) / OCC - 1024;
  int d = kRing ? 6 : 0;
  while (LY::total(d, max_nb, a.ring) > limit && d > 2) --d;
  const size_t bytes = LY::total(d, max_nb, a.ring);
  if (bytes > limit) return false;
  a.depth = d;
  cudaLaunchConfig_t cfg = {};
  cfg.gridDim = dim3((unsigned)N * C, (unsigned)((a.R + NR - 1) / NR), 1);
  cfg.blockDim = dim3(NW * 32 + (kRing ? 32 : 0), 1, 1);
  cfg.dynamicSmemBytes = bytes;
  cfg.stream = st;
  cudaLaunchAttribute at[1];
  at[0].id = cudaLaunchAttributeClusterDimension;
  at[0].val.clusterDim.x = C;
  at[0].val.clusterDim.y = 1;
  at[0].val.clusterDim.z = 1;
  cfg.attrs = at;
  cfg.numAttrs = C > 1 ? 1 : 0;
  auto* fn = k_local_super<P, NR, NW, OCC, C>;
  if (probe) {
    // the kernel's limit is the device's, not this factor's need: handles share the kernels
    if (cudaFuncSetAttribute(fn, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)optin) != cudaSuccess) {
      cudaGetLastError();
      return false;
    }
    if (C == 1) return true;
    int clusters = 0;
    if (cudaOccupancyMaxActiveClusters(&clusters, fn, &cfg) != cudaSuccess) {
      cudaGetLastError();
      return false;
    }
    return clusters >= N;
  }
  return cudaLaunchKernelEx(&cfg, fn, a) == cudaSuccess;
}

// The shapes the rules below pick.
template <template <int> class P>
bool by_shape(const SuperArgs& a, const SuperShape& f, int N, int max_nb, size_t optin, bool probe, cudaStream_t st) {
  if (f.occ == 2) return launch_impl<P<1>, 1, 16, 2, 1>(a, N, max_nb, optin, probe, st);
  if (f.warps == 24)
    return f.cluster == 2 ? launch_impl<P<1>, 1, 24, 1, 2>(a, N, max_nb, optin, probe, st)
                          : launch_impl<P<1>, 1, 24, 1, 1>(a, N, max_nb, optin, probe, st);
  return f.cluster == 4 ? launch_impl<P<1>, 1, 16, 1, 4>(a, N, max_nb, optin, probe, st)
                        : launch_impl<P<1>, 1, 16, 1, 1>(a, N, max_nb, optin, probe, st);
}

bool by_prec(const SuperArgs& a, const SuperShape& f, int prec, int N, int max_nb, size_t optin, bool probe,
             cudaStream_t st) {
  if (prec == 1 && f.nr == 8)
    return f.cluster == 2 ? launch_impl<MmaUnit32, 8, 16, 1, 2>(a, N, max_nb, optin, probe, st)
                          : launch_impl<MmaUnit32, 8, 16, 1, 1>(a, N, max_nb, optin, probe, st);
  if (prec == 1) return by_shape<RegUnit32>(a, f, N, max_nb, optin, probe, st);
  if (prec == 2 && f.nr == 4)
    return f.cluster == 2 ? launch_impl<RegUnit16<4>, 4, 16, 1, 2>(a, N, max_nb, optin, probe, st)
                          : launch_impl<RegUnit16<4>, 4, 16, 1, 1>(a, N, max_nb, optin, probe, st);
  if (prec == 2) return by_shape<RegUnit16>(a, f, N, max_nb, optin, probe, st);
  if (f.nr == 4) {
    switch (f.cluster) {
      case 2: return launch_impl<RingUnit<4>, 4, 8, 1, 2>(a, N, max_nb, optin, probe, st);
      case 4: return launch_impl<RingUnit<4>, 4, 8, 1, 4>(a, N, max_nb, optin, probe, st);
      default: return launch_impl<RingUnit<4>, 4, 8, 1, 1>(a, N, max_nb, optin, probe, st);
    }
  }
  if (f.occ == 2) return launch_impl<RingUnit<1>, 1, 8, 2, 1>(a, N, max_nb, optin, probe, st);
  switch (f.cluster) {
    case 2: return launch_impl<RingUnit<1>, 1, 16, 1, 2>(a, N, max_nb, optin, probe, st);
    case 4: return launch_impl<RingUnit<1>, 1, 16, 1, 4>(a, N, max_nb, optin, probe, st);
    case 8: return launch_impl<RingUnit<1>, 1, 16, 1, 8>(a, N, max_nb, optin, probe, st);
    default: return launch_impl<RingUnit<1>, 1, 16, 1, 1>(a, N, max_nb, optin, probe, st);
  }
}

}  // namespace

#ifdef LS_DEBUG_BOUNDS
void set_super_stall(int mode) { g_super_stall = mode; }
#endif

size_t local_super_record(int prec, bool x) {
  if (x) return prec == 0 ? Unit<double>::RECX : Unit<float>::RECX;
  return prec == 0 ? Unit<double>::REC : prec == 1 ? Unit<float>::REC : Unit<__nv_bfloat16>::REC;
}

// The rule, from sweeps over grids of N subdomains of p x p columns (p = 10 .. 64, N = 4 ..
// 256, entries within radius 3; us of a whole apply call, of which about 60 are the call).
// More subdomains than SMs: two CTAs per SM (p = 32, N = 225: FP32 197 against 275 for
// configuration 1 of the 32-row sweeps, FP64 790 against 1068; p = 64, N = 256: FP32 858
// against 936, BF16 508 against 748).
// FP64: the largest cluster whose CTAs all run at once, since the FP64 units bound it (p =
// 32, N = 16: 443, 276, 207 with 1, 2, 4 CTAs, 711 before; p = 20, N = 9: 106 with 8).
// FP32, BF16, by the mean width of a block row in tiles: one CTA is bound by the SM's intake, a
// pair by its exchanges; near the line of 8 tiles the two are within 4 %.  Below 8 tiles one CTA
// of 16 warps (a 211 x 173 grid in 50 uneven pieces, 7.3 tiles: kernel 53, pair 55, 24 warps 62,
// pair of 24 warps 66; 133 before); from 8 tiles on a pair of 24 warps when two CTAs per
// subdomain have an SM each (p = 48, 12 tiles, N = 64: 178, pair of 16 warps 198, one CTA 202; p
// = 32, 8.5 tiles: 126, 127, 130), else one CTA of 24 warps (p = 48, N = 144: 280 against 296
// with 16); from 13 tiles on four CTAs of 16 warps where there is room (p = 64, 14.5 tiles, N =
// 16: 225 against 277 for the pair; 571 before).
bool local_super_plan(int prec, int N, int max_nb, int wmax, double wmean, int sms, size_t optin, SuperShape& out) {
  auto fits = [&](int cluster, int warps, int occ) {
    out = SuperShape{cluster, warps, occ, wmax + kQ, 1};
    SuperArgs a{};
    a.ring = out.ring;
    a.R = 1;
    return by_prec(a, out, prec, N, max_nb, optin, true, nullptr);
  };
  if (N > sms && fits(1, prec == 0 ? 8 : 16, 2)) return true;
  if (prec == 0) {
    for (int c = 8; c >= 2; c >>= 1)
      if ((int64_t)N * c <= sms && fits(c, 16, 1)) return true;
    return fits(1, 16, 1);
  }
  if (N > sms) return false;
  if (wmean < 8.0) return fits(1, 16, 1);
  if (wmean >= 13.0 && 4 * (int64_t)N <= sms && fits(4, 16, 1)) return true;
  if (2 * (int64_t)N <= sms && fits(2, 24, 1)) return true;
  return fits(1, 24, 1);
}

// R right-hand sides: eight per CTA with FP32 factors (one MMA's columns), else four (BF16: eight
// do not fit the registers; FP64: the ring leaves no room for more, and the FP64 units bound
// it anyway); clusters while all CTAs then have an SM each.
bool local_super_plan_multi(int prec, int R, int N, int max_nb, int wmax, int sms, size_t optin, SuperShape& out) {
  const int nr = prec == 1 ? 8 : 4;
  auto fits = [&](int cluster) {
    out = SuperShape{cluster, prec == 0 ? 8 : 16, 1, wmax + kQ, nr};
    SuperArgs a{};
    a.ring = out.ring;
    a.R = R;
    return by_prec(a, out, prec, N, max_nb, optin, true, nullptr);
  };
  const int64_t ctas = (int64_t)N * ((R + nr - 1) / nr);
  for (int c = prec == 0 ? 4 : 2; c >= 2; c >>= 1)
    if (ctas * c <= sms && fits(c)) return true;
  return fits(1);
}

bool launch_local_super(const SuperArgs& a, const SuperShape& f, int prec, int N, int max_nb, size_t optin,
                        cudaStream_t st) {
  SuperArgs b = a;
  b.ring = f.ring;
#ifdef LS_DEBUG_BOUNDS
  b.stall = g_super_stall;
#endif
  return by_prec(b, f, prec, N, max_nb, optin, false, st);
}

void launch_super_pack(int prec, int N, int max_nb, const int64_t* blk_off, const int32_t* blk_tf,
                       const int64_t* blk_poff, const int32_t* stf, const int64_t* stoff, const double* L,
                       const double* dinv, unsigned char* dst, cudaStream_t st) {
  const dim3 grid((unsigned)N, (unsigned)((max_nb + kQ - 1) / kQ));
  const BandSrc src{blk_tf, blk_poff, L, dinv};
  if (prec == 0) k_super_pack<double><<<grid, kThreads, 0, st>>>(blk_off, src, stf, stoff, 0, 0, dst);
  else if (prec == 1) k_super_pack<float><<<grid, kThreads, 0, st>>>(blk_off, src, stf, stoff, 0, 0, dst);
  else k_super_pack<__nv_bfloat16><<<grid, kThreads, 0, st>>>(blk_off, src, stf, stoff, 0, 0, dst);
}

void launch_super_pack_solve(int prec, int N, int max_nb, const int64_t* blk_off, const int32_t* blk_tf,
                             const int64_t* blk_poff, const int32_t* stf, const int64_t* stoff, const void* fac,
                             const float* tsc, int64_t frag, unsigned char* dst, cudaStream_t st) {
  const dim3 grid((unsigned)N, (unsigned)((max_nb + kQ - 1) / kQ));
  if (prec == 0)
    k_super_pack<double><<<grid, kThreads, 0, st>>>(
        blk_off, SolveSrc<double>{blk_tf, blk_poff, (const double*)fac, nullptr}, stf, stoff, 0, 0, dst);
  else if (prec == 1)
    k_super_pack<float><<<grid, kThreads, 0, st>>>(
        blk_off, SolveSrc<float>{blk_tf, blk_poff, (const float*)fac, nullptr}, stf, stoff, 1, frag, dst);
  else
    k_super_pack<__nv_bfloat16><<<grid, kThreads, 0, st>>>(
        blk_off, SolveSrc<__nv_bfloat16>{blk_tf, blk_poff, (const __nv_bfloat16*)fac, tsc}, stf, stoff, 0, 0, dst);
}

}  // namespace lsq
