// The partition of the double-layer sums (csrc/dlp_tree.cpp) for a star on an n x m grid with N
// nodes, grid points and free points, on threads and on one: whether all arrays are equal, whether
// every point's nodes are covered once, and the numbers of boxes and leaves.
#include <cmath>
#include <cstdio>
#include <cstdlib>
#include <cstring>

#include "../paper_2010_03901_gb300/csrc/dlp_tree.cpp"

using namespace fc2d;

template <typename T> static bool same(const std::vector<T>& a, const std::vector<T>& b) {
  return a.size() == b.size() && (a.empty() || !std::memcmp(a.data(), b.data(), a.size() * sizeof(T)));
}

int main(int argc, char** argv) {
  const int n = std::atoi(argv[1]), m = std::atoi(argv[2]), N = std::atoi(argv[3]), every = std::atoi(argv[4]);
  const double R = 0.34 * std::min(n, m);
  std::vector<double> x, y, px, py;
  auto at = [&](double t, double f, double& a, double& b) {
    a = 0.47 * n + f * R * (1 + 0.3 * std::cos(5 * t)) * std::cos(t);
    b = 0.52 * m + f * R * (1 + 0.3 * std::cos(5 * t)) * std::sin(t);
  };
  for (int k = 0; k < N; ++k) {
    double a, b;
    at(2 * M_PI * k / N, 1.0, a, b);
    x.push_back(a), y.push_back(b);
  }
  for (int k = 0; k < 4 * (n + m); ++k)
    for (int j = 1; every && j < 8; ++j) {
      double a, b;
      at(2 * M_PI * k / (4 * (n + m)), 1 - 0.01 * j, a, b);
      px.push_back(a), py.push_back(b);
    }
  std::vector<int32_t> lin;
  for (int j = 0; j < m; ++j)
    for (int i = 0; i < n; ++i) {
      const double t = std::atan2(j - 0.52 * m, i - 0.47 * n), r = std::hypot(j - 0.52 * m, i - 0.47 * n);
      const double d = R * (1 + 0.3 * std::cos(5 * t)) - r;
      if (every ? d > 0 && d < 0.2 * R : d > 0.05 * R) lin.push_back(j * n + i);
    }
  const DlpTree a = dlp_tree(x, y, lin, n, px, py, std::max(n, m), true);
  const DlpTree b = dlp_tree(x, y, lin, n, px, py, std::max(n, m), false);
  bool eq = a.shift == b.shift && same(a.nodes, b.nodes) && same(a.expand, b.expand) && same(a.near, b.near) &&
            same(a.chain, b.chain) && same(a.leaf, b.leaf) && same(a.grid_items, b.grid_items) &&
            same(a.free_items, b.free_items) && same(a.grid_order, b.grid_order) &&
            same(a.free_order, b.free_order) && same(a.box, b.box);
  bool covered = true;
  std::vector<int> grid_seen(n * m), free_seen(px.size());
  std::vector<std::vector<DlpSpan>> spans(a.box.size());
  for (const DlpSpan& s : a.expand) spans[s.box].push_back(s);
  for (int pass = 0; pass < 2; ++pass)
    for (const DlpItem& it : pass ? a.free_items : a.grid_items) {
      for (int p = it.p0; p < it.p0 + it.n; ++p) ++(pass ? free_seen[a.free_order[p]] : grid_seen[a.grid_order[p]]);
      const DlpLeaf& l = a.leaf[it.leaf];
      std::vector<int> c(N);
      for (int d = l.d0; d < l.d0 + l.nd; ++d)
        for (int k = 0; k < a.near[d].n; ++k) ++c[a.near[d].k0 + k];
      for (int q = l.c0; q < l.c0 + l.nc; ++q)
        for (const DlpSpan& s : spans[a.chain[q]])
          for (int k = 0; k < s.n; ++k) ++c[s.k0 + k];
      for (int v : c) covered &= v == 1;
    }
  for (int l : lin) covered &= grid_seen[l]-- == 1;
  for (int v : grid_seen) covered &= v == 0;
  for (int v : free_seen) covered &= v == 1;
  std::printf("%d %d %zu %zu %zu\n", (int)eq, (int)covered, a.box.size(), a.leaf.size(), lin.size() + px.size());
  return 0;
}
