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
#include <future>

namespace fc2d {
namespace {

constexpr double kTerm = 130.0;           // one point-node term
constexpr double kExpand = 45.0 * kDlpOrder;  // one node into one box's coefficients
constexpr double kEval = 45.0 * kDlpOrder;    // one point from one box's coefficients
constexpr double kMinDist = 2.0;          // of an expanded node, grid units
// The root's quarters are built on threads of their own from so many points on: star at 1024^2
// with 1024 nodes, far sums 2.0 -> 0.9 ms, refined sums 6.5 -> 2.4; kite-sized point lists at 4096^2
// 21 -> 9 and 28 -> 10 ms (quarters of the quarters too: 11 and 11); at 128^2 0.8 -> 0.4 ms.
constexpr int kParallelPoints = 4096;

struct Run {  // grid points (i0 .. i1 - 1, j), linear indices id ..
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
  int32_t *grid_order, *free_order;  // of the whole tree
  int gp = 0, fp = 0;                // the next places in them
  int first = 0;  // number of t.box[0] (a quarter's boxes follow those of the squares around it)

  static void append(std::vector<Span>& v, int k0, int k1) {
    if (!v.empty() && v.back().k1 == k0) v.back().k1 = k1;
    else v.push_back({k0, k1});
  }
  static void cut(const std::vector<Span>& v, int box, int n_max, std::vector<DlpSpan>& out) {
    for (const Span& s : v)
      for (int k = s.k0; k < s.k1; k += n_max) out.push_back({box, k, std::min(n_max, s.k1 - k), 0});
  }

  // a quarter's tree behind this one's: as if it had been built here
  void add(const DlpTree& q, int q_first) {
    const int box = first + (int)t.box.size() - q_first, chain0 = (int)t.chain.size(),
              near0 = (int)t.near.size(), leaf0 = (int)t.leaf.size();
    auto join = [](auto& v, const auto& w, auto shift) {
      for (auto x : w) {
        shift(x);
        v.push_back(x);
      }
    };
    auto keep = [](auto&) {};
    join(t.box, q.box, keep);
    join(t.expand, q.expand, [&](DlpSpan& x) { x.box += box; });
    join(t.near, q.near, keep);
    join(t.chain, q.chain, [&](int32_t& x) { x += x >= q_first ? box : 0; });
    join(t.leaf, q.leaf, [&](DlpLeaf& x) { x.c0 += chain0, x.d0 += near0; });
    join(t.grid_items, q.grid_items, [&](DlpItem& x) { x.leaf += leaf0; });
    join(t.free_items, q.free_items, [&](DlpItem& x) { x.leaf += leaf0; });
  }

  // the points in the square [x0, x0 + s) x [y0, y0 + s); cand: the nodes that no expansion
  // of the chain holds; threads: one for each quarter
  void build(double x0, double y0, double s, const std::vector<Run>& runs,
             const std::vector<Point>& free, const std::vector<Span>& cand, bool threads) {
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
      const int id = first + (int)t.box.size();
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
      if (threads && n >= kParallelPoints) {
        const int q_first = first + (int)t.box.size();
        std::future<DlpTree> part[4];
        for (int q = 0; q < 4; ++q) {
          part[q] = std::async(std::launch::async | std::launch::deferred, [&, q, g0 = gp, f0 = fp] {
            Builder b{nx, ny, step, {}, chain, grid_order, free_order, g0, f0, q_first};
            b.t.shift = t.shift;
            b.build(q & 1 ? xm : x0, q < 2 ? y0 : ym, hs, rq[q], fq[q], near, false);
            return std::move(b.t);
          });
          for (const Run& r : rq[q]) gp += r.i1 - r.i0;
          fp += (int)fq[q].size();
        }
        for (auto& q : part) add(q.get(), q_first);
      } else {
        for (int q = 0; q < 4; ++q)
          build(q & 1 ? xm : x0, q < 2 ? y0 : ym, hs, rq[q], fq[q], near, false);
      }
    } else {
      const int id = (int)t.leaf.size();
      DlpLeaf l = {(int)t.chain.size(), (int)chain.size(), (int)t.near.size(), 0};
      t.chain.insert(t.chain.end(), chain.begin(), chain.end());
      cut(near, 0, 1 << 30, t.near);
      l.nd = (int)t.near.size() - l.d0;
      t.leaf.push_back(l);
      int p = gp;
      for (const Run& r : runs)
        for (int k = 0; k < r.i1 - r.i0; ++k) grid_order[gp++] = r.id + k;
      for (; p < gp; p += kDlpPoints) t.grid_items.push_back({id, p, std::min(kDlpPoints, gp - p), 0});
      p = fp;
      for (const Point& f : free) free_order[fp++] = f.id;
      for (; p < fp; p += kDlpPoints) t.free_items.push_back({id, p, std::min(kDlpPoints, fp - p), 0});
    }
    chain.resize(depth);
  }
};

}  // namespace

DlpTree dlp_tree(const std::vector<double>& nx, const std::vector<double>& ny,
                 const std::vector<int32_t>& lin, int stride, const std::vector<double>& px,
                 const std::vector<double>& py, int extent, bool threads) {
  const int n = (int)nx.size();
  double step = 0.0;
  for (int k = 1; k < n; ++k) step = std::max(step, std::hypot(nx[k] - nx[k - 1], ny[k] - ny[k - 1]));
  DlpTree orders;
  orders.grid_order.resize(lin.size());
  orders.free_order.resize(px.size());
  Builder b{nx, ny, step * (1 + 1e-9) + 1e-9, {}, {}, orders.grid_order.data(), orders.free_order.data(),
            0, 0, 0};
  int lg = 1;
  while ((1 << lg) < extent) ++lg;
  b.t.shift = 61 - lg;
  b.t.nodes.resize(2 * nx.size());
  for (int k = 0; k < n; ++k) {
    b.t.nodes[2 * k] = std::llrint(std::ldexp(nx[k], b.t.shift));
    b.t.nodes[2 * k + 1] = std::llrint(std::ldexp(ny[k], b.t.shift));
  }
  std::vector<Run> runs;
  for (size_t k = 0; k < lin.size();) {
    const int j = lin[k] / stride, l0 = lin[k], end = (j + 1) * stride;
    size_t e = k + 1;
    while (e < lin.size() && lin[e] == lin[e - 1] + 1 && lin[e] < end) ++e;
    runs.push_back({l0 - j * stride, l0 - j * stride + (int)(e - k), j, l0});
    k = e;
  }
  std::vector<Point> free(px.size());
  for (size_t k = 0; k < px.size(); ++k) free[k] = {px[k], py[k], (int32_t)k};
  b.build(-0.5, -0.5, (double)(1 << lg), runs, free, {{0, n}}, threads);
  b.t.grid_order.swap(orders.grid_order);
  b.t.free_order.swap(orders.free_order);
  return std::move(b.t);
}

}  // namespace fc2d
