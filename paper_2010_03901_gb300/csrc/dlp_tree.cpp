// Partition of the point-node pairs of a double-layer sum (see dlp_tree.h).
//
// Top down over squares of points: the nodes that are far from a square's points go into
// its expansion, the others to its four quarters, until summing them term by term is
// cheaper than another level.  The unit of the costs below is one issued instruction; what
// they decide is which path a pair takes, not the result (both are accurate to ~2^-48 of
// the terms' sizes).  Weights of 30 to 90 in place of the 45s below change the sums by 3%.
#include "dlp_tree.h"

#include <algorithm>
#include <cmath>

namespace fc2d {
namespace {

constexpr double kTerm = 130.0;           // one point-node term
constexpr double kExpand = 45.0 * kDlpOrder;  // one node into one box's coefficients
constexpr double kEval = 45.0 * kDlpOrder;    // one point from one box's coefficients
constexpr double kMinDist = 2.0;          // of an expanded node, grid units

struct Run {  // grid points (i0 .. i1 - 1, j), numbers id ..
  int i0, i1, j;
  int32_t id;
};
struct Point {
  double x, y;
  int32_t id;
};
struct Span {  // nodes k0 .. k1 - 1
  int k0, k1;
};

struct Builder {
  const std::vector<double>&nx, &ny;
  double step;  // largest distance of consecutive nodes
  DlpTree t;
  std::vector<int32_t> chain;

  static void append(std::vector<Span>& v, int k0, int k1) {
    if (!v.empty() && v.back().k1 == k0) v.back().k1 = k1;
    else v.push_back({k0, k1});
  }
  static void cut(const std::vector<Span>& v, int box, int n_max, std::vector<DlpSpan>& out) {
    for (const Span& s : v)
      for (int k = s.k0; k < s.k1; k += n_max) out.push_back({box, k, std::min(n_max, s.k1 - k), 0});
  }

  // the points in the square [x0, x0 + s) x [y0, y0 + s); cand: the nodes that no expansion
  // of the chain holds
  void build(double x0, double y0, double s, const std::vector<Run>& runs,
             const std::vector<Point>& free, const std::vector<Span>& cand) {
    if (runs.empty() && free.empty()) return;
    double xl = 1e300, xh = -1e300, yl = 1e300, yh = -1e300;  // the points' bounding box
    auto grow = [&](double a, double b, double y) {
      xl = std::min(xl, a), xh = std::max(xh, b), yl = std::min(yl, y), yh = std::max(yh, y);
    };
    int ng = 0;
    for (const Run& r : runs) {
      grow(r.i0, r.i1 - 1, r.j);
      ng += r.i1 - r.i0;
    }
    for (const Point& q : free) grow(q.x, q.x, q.y);
    const int n = ng + (int)free.size();
    const double cx = std::floor(xl + xh) * 0.5, cy = std::floor(yl + yh) * 0.5;
    const double rx = std::max(xh - cx, cx - xl), ry = std::max(yh - cy, cy - yl);
    const double r = std::sqrt(rx * rx + ry * ry);
    const double reach = std::max(r / kDlpTheta, kMinDist);
    // Along the curve: the next nodes are on the same side of the circle as long as the arc
    // between them is shorter than the distance to it; half of that is taken at once, which
    // keeps the bounds of the distances within a factor of 2.
    std::vector<Span> near, sep;
    double m = 0.0, ns = 0.0, inv = 0.0;  // inv: bound of sum 1/|z_k - c|
    for (const Span& q : cand)
      for (int k = q.k0; k < q.k1;) {
        const double dx = nx[k] - cx, dy = ny[k] - cy, d = std::sqrt(dx * dx + dy * dy);
        const double gap = std::fabs(d - reach) / (2.0 * step);
        const int c = gap < q.k1 - k ? 1 + (int)gap : q.k1 - k;
        if (d >= reach) {
          append(sep, k, k + c);
          const double low = std::max(reach, d - c * step);
          inv += c / low;
          ns += c;
        } else {
          append(near, k, k + c);
          m += c;
        }
        k += c;
      }
    // another level halves the terms, costs its expansions and their evaluation
    const bool split = s > 1.0 && 0.5 * kTerm * m * n > 2.0 * kExpand * m + kEval * n;
    // expanding here rather than in the four quarters; in a leaf, rather than term by term
    // (whose blocks have kDlpPoints threads, however few points there are)
    const double nb = (n + kDlpPoints - 1) / kDlpPoints * kDlpPoints;
    const bool expand = split ? 3.0 * kExpand * ns > kEval * n
                              : kExpand * ns + kEval * nb < kTerm * ns * nb;
    const size_t depth = chain.size();
    if (!sep.empty() && expand) {
      // R0: the circle itself, so that a point's (z - c)/R0 is at most kDlpTheta
      int lr;
      const double m = 2.0 * std::frexp(reach, &lr), w = inv * reach;
      --lr;
      const int id = (int)t.box.size();
      t.box.push_back({(long long)std::ldexp(cx, t.shift), (long long)std::ldexp(cy, t.shift),
                       (long long)std::ldexp(m, lr + t.shift), (long long)std::ldexp(1.0 / m, 62),
                       1.0 / m, lr, std::max(0, (int)std::ceil(std::log2(w) + 1.5))});
      cut(sep, id, kDlpNodes, t.expand);
      chain.push_back(id);
    } else if (!sep.empty()) {
      near = cand;
    }
    if (split) {
      const double hs = 0.5 * s, xm = x0 + hs, ym = y0 + hs;
      const int im = (int)std::ceil(xm);  // x < xm: i < im
      std::vector<Run> rq[4];
      std::vector<Point> fq[4];
      for (const Run& r : runs) {
        const int q = r.j < ym ? 0 : 2, cut = std::min(std::max(im, r.i0), r.i1);
        if (r.i0 < cut) rq[q].push_back({r.i0, cut, r.j, r.id});
        if (cut < r.i1) rq[q + 1].push_back({cut, r.i1, r.j, r.id + cut - r.i0});
      }
      for (const Point& f : free) fq[(f.y < ym ? 0 : 2) + (f.x < xm ? 0 : 1)].push_back(f);
      for (int q = 0; q < 4; ++q) build(q & 1 ? xm : x0, q < 2 ? y0 : ym, hs, rq[q], fq[q], near);
    } else {
      const int id = (int)t.leaf.size();
      DlpLeaf l = {(int)t.chain.size(), (int)chain.size(), (int)t.near.size(), 0};
      t.chain.insert(t.chain.end(), chain.begin(), chain.end());
      cut(near, 0, 1 << 30, t.near);
      l.nd = (int)t.near.size() - l.d0;
      t.leaf.push_back(l);
      int p = (int)t.grid_order.size();
      for (const Run& r : runs)
        for (int k = 0; k < r.i1 - r.i0; ++k) t.grid_order.push_back(r.id + k);
      for (const int e = p + ng; p < e; p += kDlpPoints)
        t.grid_items.push_back({id, p, std::min(kDlpPoints, e - p), 0});
      p = (int)t.free_order.size();
      for (const Point& f : free) t.free_order.push_back(f.id);
      for (const int e = (int)t.free_order.size(); p < e; p += kDlpPoints)
        t.free_items.push_back({id, p, std::min(kDlpPoints, e - p), 0});
    }
    chain.resize(depth);
  }
};

}  // namespace

DlpTree dlp_tree(const std::vector<double>& nx, const std::vector<double>& ny,
                 const std::vector<int32_t>& gi, const std::vector<int32_t>& gj,
                 const std::vector<double>& px, const std::vector<double>& py, int extent) {
  const int n = (int)nx.size();
  double step = 0.0;
  for (int k = 1; k < n; ++k) step = std::max(step, std::hypot(nx[k] - nx[k - 1], ny[k] - ny[k - 1]));
  Builder b{nx, ny, step * (1 + 1e-9) + 1e-9, {}, {}};
  int lg = 1;
  while ((1 << lg) < extent) ++lg;
  b.t.shift = 61 - lg;
  b.t.nodes.resize(2 * nx.size());
  for (int k = 0; k < n; ++k) {
    b.t.nodes[2 * k] = std::llrint(std::ldexp(nx[k], b.t.shift));
    b.t.nodes[2 * k + 1] = std::llrint(std::ldexp(ny[k], b.t.shift));
  }
  std::vector<Run> runs;
  for (size_t k = 0; k < gi.size(); ++k) {
    if (k && gj[k] == gj[k - 1] && gi[k] == gi[k - 1] + 1) ++runs.back().i1;
    else runs.push_back({gi[k], gi[k] + 1, gj[k], (int32_t)k});
  }
  std::vector<Point> free(px.size());
  for (size_t k = 0; k < px.size(); ++k) free[k] = {px[k], py[k], (int32_t)k};
  b.t.grid_order.reserve(gi.size());
  b.build(-0.5, -0.5, (double)(1 << lg), runs, free, {{0, n}});
  return std::move(b.t);
}

}  // namespace fc2d
