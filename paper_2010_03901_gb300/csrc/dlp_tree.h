// Fast summation of the double-layer potential's trapezoidal sums: the partition of the
// point-node pairs (dlp_tree.cpp, host) and the sums over it (dlp_sum.cu).
//
// With z = x + i y and q_k = (x'_k + i y'_k) phi_k / N the sum at a point z is
// Im F(z), F(z) = sum_k q_k / (z - z_k): analytic away from the nodes.  In a box of points
// with centre c, the nodes at a distance of at least r/kTheta (r: the points' largest
// distance from c) enter through the first kOrder coefficients of F's Taylor series,
//   F(z) = -(1/R0) sum_j A_j ((z - c)/R0)^j,   A_j = sum_k q_k (R0/(z_k - c))^(j+1),
// the others term by term.  Left out: kTheta^kOrder = 2^-55.6 of sum |q_k|/|z_k - c|.
#pragma once
#include <cstdint>
#include <vector>

namespace fc2d {

constexpr int kDlpOrder = 32;       // coefficients per box: one per lane
constexpr double kDlpTheta = 0.3;
constexpr int kDlpNodes = 128;      // nodes per expansion work item (a warp), at most
constexpr int kDlpPoints = 64;      // points per evaluation work item (a block), at most

struct DlpBox {
  long long cx, cy;    // centre, grid units times 2^shift
  long long one, inv;  // R0 = m 2^lr, 1 <= m < 2, in the same unit; 2^62/m
  double rm;           // 1/m
  int lr, hb;          // 2^hb bounds 2^1.5 sum |R0/(z_k - c)|
};
struct DlpSpan {  // expansion item: nodes k0 .. k0 + n - 1 into a box; direct span (box unused)
  int box, k0, n, pad;
};
struct DlpLeaf {  // a leaf's expansions chain[c0 .. c0 + nc) and direct spans near[d0 .. d0 + nd)
  int c0, nc, d0, nd;
};
struct DlpItem {  // evaluation item: points p0 .. p0 + n - 1 of a leaf
  int leaf, p0, n, pad;
};

struct DlpTree {
  int shift = 0;
  std::vector<long long> nodes;       // [N][2] node positions, grid units times 2^shift
  std::vector<DlpBox> box;
  std::vector<DlpSpan> expand, near;
  std::vector<int32_t> chain;
  std::vector<DlpLeaf> leaf;
  std::vector<DlpItem> grid_items, free_items;
  // the points in leaf order: linear indices of grid points, indices of free points
  std::vector<int32_t> grid_order, free_order;
};

// nodes and free points in grid units, grid points as linear indices j stride + i; extent: bound
// of all coordinates.  The partition is the same with threads and without.
DlpTree dlp_tree(const std::vector<double>& nx, const std::vector<double>& ny,
                 const std::vector<int32_t>& lin, int stride, const std::vector<double>& px,
                 const std::vector<double>& py, int extent, bool threads = true);

}  // namespace fc2d
