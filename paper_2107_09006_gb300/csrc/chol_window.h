// Launch geometry of the batched right-looking Cholesky (k_band.cu): which subdomains share
// its launches, and which pair of block rows a CTA updates.
#pragma once
#include <algorithm>
#include <cmath>
#include <cstdint>
#include <vector>

#ifdef __CUDACC__
#define LSQ_HD __host__ __device__ __forceinline__
#else
#define LSQ_HD inline
#endif

namespace lsq {

// Subdomains [first, first + count) of the order; none has more than max_nb block rows or a
// block row that reaches more than `below` rows down.
struct CholGroup { int first, count, max_nb, below; };

// gridDim.y ends at 65,535, which the pairs of a window of 362 block rows pass: CTAs stride.
constexpr int64_t kCholGridY = 65535;
LSQ_HD int64_t chol_pairs(int below) { return (int64_t)below * (below + 1) / 2; }
inline unsigned chol_grid_y(int below) { return (unsigned)std::min<int64_t>(chol_pairs(below), kCholGridY); }
// Pair e of a window: rows 0 <= c <= b, e = b (b + 1) / 2 + c.
LSQ_HD void chol_pair(int64_t e, int& b, int& c) {
  b = (int)((sqrtf(8.f * (float)e + 1.f) - 1.f) * 0.5f);
  while ((int64_t)(b + 1) * (b + 2) / 2 <= e) ++b;
  while ((int64_t)b * (b + 1) / 2 > e) --b;
  c = (int)(e - (int64_t)b * (b + 1) / 2);
}

// A launch covers its group's widest window for each of its subdomains, so subdomains by
// decreasing window, a new group from a quarter of the group's widest on: at most 16 times the
// CTAs that have work (one subdomain of 363 tiles among thousands of a few tiles would
// otherwise launch 65 thousand idle CTAs for each of them and each block column).  Even
// partitions make one group.
inline std::vector<CholGroup> chol_groups(int N, const int64_t* blk_off, const int32_t* blk_tf,
                                          std::vector<int32_t>& order) {
  std::vector<int> below((size_t)N, 0);
  order.resize((size_t)N);
  for (int i = 0; i < N; ++i) {
    order[i] = i;
    for (int64_t g = blk_off[i]; g < blk_off[i + 1]; ++g) below[i] = std::max(below[i], (int)(g - blk_off[i]) - blk_tf[g]);
  }
  std::stable_sort(order.begin(), order.end(), [&](int a, int b) { return below[a] > below[b]; });
  std::vector<CholGroup> groups;
  for (int k = 0; k < N; ++k) {
    const int i = order[k];
    if (groups.empty() || 4 * (below[i] + 1) < groups.back().below + 1) groups.push_back(CholGroup{k, 0, 0, below[i]});
    CholGroup& g = groups.back();
    ++g.count;
    g.max_nb = std::max(g.max_nb, (int)(blk_off[i + 1] - blk_off[i]));
  }
  return groups;
}

}  // namespace lsq
