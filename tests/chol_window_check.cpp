// Host check of the Cholesky's launch geometry (chol_window.h): every pair of a window is
// taken exactly once by the strided CTAs of a launch whose dimensions the device accepts, and
// the groups hold every subdomain once, cover its window and keep idle CTAs bounded.
#include <cstdio>
#include <cstdlib>
#include <random>
#include <vector>

#include "../paper_2107_09006_gb300/csrc/chol_window.h"

namespace {

void require(bool ok, const char* what, long long v) {
  if (ok) return;
  std::printf("FAILED: %s (%lld)\n", what, v);
  std::exit(1);
}

void window(int below) {
  const unsigned gy = lsq::chol_grid_y(below);
  require(gy >= 1 && gy <= 65535, "gridDim.y", gy);
  std::vector<char> seen((size_t)lsq::chol_pairs(below), 0);
  for (unsigned y = 0; y < gy; ++y)
    for (int64_t e = y; e < lsq::chol_pairs(below); e += gy) {
      int b = -1, c = -1;
      lsq::chol_pair(e, b, c);
      require(0 <= c && c <= b && b < below, "pair in range", e);
      const size_t at = (size_t)b * (b + 1) / 2 + c;
      require(!seen[at], "pair taken twice", e);
      seen[at] = 1;
    }
  for (size_t k = 0; k < seen.size(); ++k) require(seen[k], "pair left out", (long long)k);
}

// Subdomains of nb[i] block rows whose block row b reaches back w[i] - 1 tiles.
void groups(const std::vector<int>& nb, const std::vector<int>& w, size_t most) {
  const int N = (int)nb.size();
  std::vector<int64_t> off{0};
  std::vector<int32_t> tf;
  for (int i = 0; i < N; ++i) {
    for (int b = 0; b < nb[i]; ++b) tf.push_back(std::max(0, b - w[i] + 1));
    off.push_back((int64_t)tf.size());
  }
  std::vector<int32_t> order;
  const auto g = lsq::chol_groups(N, off.data(), tf.data(), order);
  require(g.size() <= most, "number of groups", (long long)g.size());
  std::vector<char> seen((size_t)N, 0);
  int at = 0;
  for (const auto& q : g) {
    require(q.first == at && q.count > 0, "groups are consecutive", q.first);
    at += q.count;
    for (int k = q.first; k < at; ++k) {
      const int i = order[k], mine = std::min(w[i], nb[i]) - 1;
      require(!seen[i], "subdomain twice", i);
      seen[i] = 1;
      require(nb[i] <= q.max_nb && mine <= q.below, "window covered", i);
      require(4 * (mine + 1) >= q.below + 1, "idle CTAs bounded", i);
    }
  }
  require(at == N, "every subdomain", at);
}

}  // namespace

int main() {
  for (int below = 1; below <= 40; ++below) window(below);
  for (int below : {361, 362, 363, 500, 682, 683, 1072, 1073}) window(below);
  std::printf("windows\n");
  groups({363}, {363}, 1);
  groups(std::vector<int>(256, 145), std::vector<int>(256, 15), 1);
  groups(std::vector<int>(65536, 1), std::vector<int>(65536, 1), 1);
  std::vector<int> nb(4001, 6), w(4001, 4);
  nb[1234] = 700; w[1234] = 700;
  groups(nb, w, 2);
  std::mt19937 rng(7);
  for (int t = 0; t < 200; ++t) {
    const int N = 1 + (int)(rng() % 60);
    nb.assign((size_t)N, 0);
    w.assign((size_t)N, 0);
    for (int i = 0; i < N; ++i) {
      nb[i] = 1 + (int)(rng() % (1u << (rng() % 10)));
      w[i] = 1 + (int)(rng() % (unsigned)nb[i]);
    }
    groups(nb, w, 6);
  }
  std::printf("groups\nALL OK\n");
}
