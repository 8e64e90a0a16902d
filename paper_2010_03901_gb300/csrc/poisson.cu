// 2D-FC Poisson solver (Section 4.1, eqs. (4.1)-(4.6)), FP64 data; the double-layer
// sums on the grid by expansions in boxes of points (dlp_tree.h).
//
//   u = u_p + v.  u_p: the spectrum of the extension of f times the inverse Laplacian
//   symbol -1/((2 pi l/L_x)^2 + (2 pi m/L_y)^2) (0 at the origin), inverse DFT, plus
//   hat f_00 (x^2 + y^2)/4 (sign taken so that Delta u_p = f^c).
//   v: double-layer potential, -phi/2 + K phi = g - u_p on the curve, trapezoidal
//   Nystrom on N_b equispaced parameters, solved by GMRES (one cooperative
//   launch, gmres.cu).  v on the grid points inside: the
//   trapezoidal sum; within 5 s of the curve (s = (2 pi/N_b) max|q'|) the density is
//   refined R = 8 times by trigonometric interpolation and, closer than 5 s/R, v is
//   the degree M_P - 1 Lagrange interpolant along the normal through the boundary
//   value (trigonometric interpolation of g - u_p) and refined sums at 5s/R..(M_P+3)s/R.
//
// Kernels: the forward column DFT, k_symbol (multiplier), the same DFT on reversed rows as the
// inverse one, the inverse real rows + quadratic term (fx_wave.cu), k_up_nodes,
// GMRES (gmres.cu), k_density_dft / k_density_refine, the sums and the close points'
// values (dlp_sum.cu), k_zero_outside.
#include <cuda_runtime.h>

#include <algorithm>
#include <cmath>
#include <cstdint>
#include <cstring>
#include <future>
#include <string>
#include <vector>

#include "dd.h"
#include "dlp_sum.h"
#include "fc2d_kernels.cuh"
#include "fx.cuh"
#include "gmres.h"
#include "plan_internal.h"

namespace fc2d {

constexpr int kRefine = 8;

struct PoissonState {
  int Nb = 0, R = kRefine, MP = 8;
  double s = 0, delta = 0;
  double *bx = nullptr, *by = nullptr, *bx1 = nullptr, *by1 = nullptr;  // nodes [Nb]
  double* A = nullptr;                                                  // [Nb][Nb]
  double *rx = nullptr, *ry = nullptr, *rx1 = nullptr, *ry1 = nullptr;  // refined [R Nb]
  double* twb = nullptr;                                                // e^{-2 pi i t/Nb}
  double* twr = nullptr;                                                // e^{+2 pi i t/(R Nb)}
  int32_t *ui0 = nullptr, *uj0 = nullptr;                               // [Nb]
  double *uwx = nullptr, *uwy = nullptr;                                // [Nb][MP]
  int64_t n_far = 0, n_mid = 0, n_close = 0;
  DlpDev far, near;             // partitions of the far and the refined sums
  size_t sum_bytes = 0;         // their coefficients and magnitudes, zeroed per solution
  unsigned* mags = nullptr;     // magnitudes of the boundary values' and density's coefficients
  double2* spec = nullptr;      // [ny][pitch]: a function's spectrum, then its inverse columns
  int* exps = nullptr;          // of its two-pass columns
  double2 *qB = nullptr, *qR = nullptr;  // node coefficients [Nb], [R Nb]
  double* close_v = nullptr;    // [n_close][MP - 1] refined sums along the normals
  int32_t *far_lin = nullptr, *mid_lin = nullptr, *close_lin = nullptr;
  double* close_z = nullptr;    // [n_close][2]: cos, sin of the foot's parameter
  double* close_w = nullptr;    // [n_close][MP]
  std::vector<double> close_nodes;  // [MP] distances along the normal
  // per-solve workspace
  double *g = nullptr, *phi = nullptr;
  Gmres gm;
  double *ghat = nullptr, *phiR = nullptr, *c00 = nullptr;
  float4 *ab = nullptr, *abR = nullptr;        // double-float node coefficients [Nb], [R Nb]
  float4 *posB = nullptr, *posR = nullptr;     // nodes in grid units [Nb][2], [R Nb][2]
  std::vector<double> xy_host;  // node coordinates [Nb][2]
  int last_iters = 0;
  double last_resid = 0;
  std::vector<void*> allocs;
};

static void poisson_free(PoissonState* P) {
  if (!P) return;
  for (void* q : P->allocs) cudaFree(q);
  delete P;
}

void poisson_destroy(fc2d_plan_s* p) {
  poisson_free(static_cast<PoissonState*>(p->poisson));
  p->poisson = nullptr;
}

// ------------------------------------------------------------------------- //
// Kernels
// ------------------------------------------------------------------------- //
// hat f times the inverse Laplacian symbol; hat f_00 goes to c00.  Bound by the FP64 division
// (50% of that pipe at 1024^2, 18 us cold); with the two fixed-point column passes of 14 us
// the particular solution's columns take 43 us there, 187 us as FP64 transforms with the
// symbol in one kernel.  The rows are written in
// reversed order, ky at (ny - ky) mod ny: the forward column DFT of that is the inverse one of
// the spectrum.
constexpr int kSymbolRows = 8;
__global__ void __launch_bounds__(128) k_symbol(int nxh, int ny, int pitch, const double2* spec,
                                                double2* out, double* c00, double wx, double wy) {
  const int kx = blockIdx.x * blockDim.x + threadIdx.x;
  if (kx >= nxh) return;
  const double kxx = wx * kx, kx2 = kxx * kxx;
#pragma unroll
  for (int r = 0; r < kSymbolRows; ++r) {
    const int ky = blockIdx.y * kSymbolRows + r;
    if (ky >= ny) return;
    const double kyy = wy * (ky <= ny / 2 ? ky : ky - ny);
    const double2 v = spec[(size_t)ky * pitch + kx];
    double2 b{0.0, 0.0};
    if (kx == 0 && ky == 0) {
      *c00 = v.x;
    } else {
      const double s = -1.0 / fma(kyy, kyy, kx2);
      b = double2{v.x * s, v.y * s};
    }
    out[(size_t)(ky ? ny - ky : 0) * pitch + kx] = b;
  }
}

// u_p at the BIE nodes: iterated 1D interpolation (x on MP rows, a lane each, then y).  Latency
// bound: 6 us for 1024 nodes (22 with a thread per node).
__global__ void __launch_bounds__(128) k_up_nodes(int Nb, int MP, int nx, const int32_t* i0,
                                                  const int32_t* j0, const double* wx,
                                                  const double* wy, const double* up,
                                                  const double* g, double* ghom) {
  static_assert(kMaxM <= 16, "a lane per row");
  const int k = (blockIdx.x * blockDim.x + threadIdx.x) >> 4, a = threadIdx.x & 15;
  double acc = 0.0;
  if (k < Nb && a < MP) {
    const double* r = up + (size_t)(j0[k] + a) * nx + i0[k];
    double v = 0.0;
#pragma unroll 8
    for (int b = 0; b < MP; ++b) v = fma(wx[k * MP + b], r[b], v);
    acc = wy[k * MP + a] * v;
  }
  for (int o = 8; o; o >>= 1) acc += __shfl_xor_sync(0xFFFFFFFFu, acc, o);
  if (k < Nb && a == 0) ghom[k] = g[k] - acc;
}

__global__ void k_bie_matrix(int Nb, const double* x, const double* y, const double* x1,
                             const double* y1, const double* diag, double* A) {
  int i = blockIdx.y, k = blockIdx.x * blockDim.x + threadIdx.x;
  if (k >= Nb) return;
  const double w = 1.0 / Nb;  // (2 pi/Nb) * 1/(2 pi)
  double v;
  if (i == k) {
    v = -0.5 + diag[i];
  } else {
    double dx = x[i] - x[k], dy = y[i] - y[k];
    v = w * (y1[k] * dx - x1[k] * dy) / (dx * dx + dy * dy);
  }
  A[(size_t)i * Nb + k] = v;
}

// Coefficients of the trigonometric interpolant of phi: (1/Nb) sum_j phi_j e^{-2 pi i jk/Nb},
// k = 0..Nb/2, doubled for 0 < k < Nb/2 (the pairs k, Nb - k); a warp per k (12 us for 1024
// points, latency bound).  mag: the largest magnitude.
__global__ void __launch_bounds__(128) k_density_dft(int Nb, const double* phi, const double2* twb,
                                                     double2* ghat, unsigned* mag) {
  const int k = (blockIdx.x * blockDim.x + threadIdx.x) >> 5, lane = threadIdx.x & 31;
  if (k > Nb / 2) return;
  double re = 0.0, im = 0.0;
  int at = (int)(((int64_t)lane * k) % Nb);  // j k mod Nb
  const int step = (int)((32 * (int64_t)k) % Nb);
#pragma unroll 8
  for (int j = lane; j < Nb; j += 32) {
    const double2 w = twb[at];
    re = fma(phi[j], w.x, re);
    im = fma(phi[j], w.y, im);
    at += step;
    at -= at >= Nb ? Nb : 0;
  }
  for (int o = 16; o; o >>= 1) {
    re += __shfl_xor_sync(0xFFFFFFFFu, re, o);
    im += __shfl_xor_sync(0xFFFFFFFFu, im, o);
  }
  if (lane) return;
  const double fac = k == 0 || 2 * k == Nb ? 1.0 : 2.0;
  re = fac * re / Nb;
  im = fac * im / Nb;
  ghat[k] = double2{re, im};
  atomicMax(mag, max(fx::magnitude(re), fx::magnitude(im)));
}

// Trigonometric interpolant of the density at the NR = 8 Nb refined parameters: a warp per
// quadruple of parameters x, -x, pi - x, pi + x, whose sums are +- combinations of the cosine
// and sine sums over even and odd k (even and odd lanes): half an FP64 multiply-add per term
// and output.  11 us for 1024 nodes; 24 us with pairs x, -x and the doubling in the loop.
__global__ void __launch_bounds__(128) k_density_refine(int Nb, int NR, const double2* ghat,
                                                        const double2* twr, double* out) {
  const int m = (blockIdx.x * blockDim.x + threadIdx.x) >> 5, lane = threadIdx.x & 31;
  if (m > NR / 4) return;
  double C = 0.0, S = 0.0;
  int at = (int)(((int64_t)lane * m) % NR);  // k m mod NR
  const int step = (int)((32 * (int64_t)m) % NR);
#pragma unroll 4
  for (int k = lane; k <= Nb / 2; k += 32) {
    const double2 e = twr[at], g = ghat[k];
    C = fma(g.x, e.x, C);
    S = fma(g.y, e.y, S);
    at += step;
    at -= at >= NR ? NR : 0;
  }
  for (int o = 16; o > 1; o >>= 1) {
    C += __shfl_xor_sync(0xFFFFFFFFu, C, o);
    S += __shfl_xor_sync(0xFFFFFFFFu, S, o);
  }
  const double Co = __shfl_xor_sync(0xFFFFFFFFu, C, 1), So = __shfl_xor_sync(0xFFFFFFFFu, S, 1);
  if (lane) return;
  const double cp = C + Co, cm = C - Co, sp = S + So, sm = S - So;
  const int half = NR / 2;
  out[m] = cp - sp;
  out[half - m] = cm + sm;
  if (m == 0) return;
  out[half + m] = cm - sm;
  out[NR - m] = cp + sp;
}

__global__ void k_zero_outside(int nx, const int32_t* row_iv_off, const int32_t* row_iv,
                               double* u) {
  const int j = blockIdx.x;
  double* r = u + (size_t)j * nx;
  const int iv0 = row_iv_off[j], iv1 = row_iv_off[j + 1];
  for (int i = threadIdx.x; i < nx; i += blockDim.x) {
    bool in = false;
    for (int k = iv0; k < iv1; ++k) in |= (i >= row_iv[2 * k] && i <= row_iv[2 * k + 1]);
    if (!in) r[i] = 0.0;
  }
}

// ------------------------------------------------------------------------- //
// Setup
// ------------------------------------------------------------------------- //
template <typename T>
static fc2d_status up(PoissonState* P, T** dst, const std::vector<T>& src) {
  size_t bytes = std::max<size_t>(1, src.size()) * sizeof(T);
  if (cudaMalloc((void**)dst, bytes) != cudaSuccess)
    return set_error(FC2D_ERR_NOMEM, "Poisson setup: cudaMalloc failed");
  P->allocs.push_back(*dst);
  if (!src.empty() &&
      cudaMemcpy(*dst, src.data(), src.size() * sizeof(T), cudaMemcpyHostToDevice) != cudaSuccess)
    return set_error(FC2D_ERR_CUDA, "Poisson setup: cudaMemcpy failed");
  return FC2D_OK;
}

template <typename T>
static fc2d_status alloc(PoissonState* P, T** dst, size_t n) {
  if (cudaMalloc((void**)dst, std::max<size_t>(1, n) * sizeof(T)) != cudaSuccess)
    return set_error(FC2D_ERR_NOMEM, "Poisson setup: cudaMalloc failed");
  P->allocs.push_back(*dst);
  return FC2D_OK;
}

// Node positions in grid units for the double-float sums: per node (ix, iy, fx_hi,
// fx_lo), (fy_hi, fy_lo, 0, 0), with (x - a0)/h = ix + fx, 0 <= fx < 1 (the same in y).
static std::vector<float4> grid_units(const std::vector<double>& x, const std::vector<double>& y,
                                      double a0, double b0, double h) {
  std::vector<float4> out(2 * x.size());
  for (size_t k = 0; k < x.size(); ++k) {
    const double ux = (x[k] - a0) / h, uy = (y[k] - b0) / h;
    const double ix = std::floor(ux), iy = std::floor(uy), fx = ux - ix, fy = uy - iy;
    const float fxh = (float)fx, fyh = (float)fy;
    out[2 * k] = make_float4((float)ix, (float)iy, fxh, (float)(fx - (double)fxh));
    out[2 * k + 1] = make_float4(fyh, (float)(fy - (double)fyh), 0.f, 0.f);
  }
  return out;
}

static void lagr(const double* nodes, int n, double t, double* w) {
  for (int k = 0; k < n; ++k) {
    double v = 1.0;
    for (int m = 0; m < n; ++m)
      if (m != k) v *= (t - nodes[m]) / (nodes[k] - nodes[m]);
    w[k] = v;
  }
}

// A partition's arrays on the device (coefficients and magnitude word are placed by the
// caller).  pts: the free points.
static fc2d_status up_tree(PoissonState* P, DlpDev* d, const DlpTree& t,
                           const std::vector<double>& px, const std::vector<double>& py) {
  std::vector<long long> pts(2 * px.size());
  for (size_t k = 0; k < px.size(); ++k) {
    pts[2 * k] = std::llrint(std::ldexp(px[t.free_order[k]], t.shift));
    pts[2 * k + 1] = std::llrint(std::ldexp(py[t.free_order[k]], t.shift));
  }
  auto put = [&](auto** dst, const auto& v) {
    typename std::remove_const<typename std::remove_reference<decltype(**dst)>::type>::type* q =
        nullptr;
    const fc2d_status st = up(P, &q, v);
    *dst = q;
    return st;
  };
  d->shift = t.shift;
  d->n_expand = (int)t.expand.size();
  d->n_grid = (int)t.grid_items.size();
  d->n_free = (int)t.free_items.size();
  fc2d_status st;
  if ((st = put(&d->nodes, t.nodes)) || (st = put(&d->box, t.box)) ||
      (st = put(&d->expand, t.expand)) || (st = put(&d->near, t.near)) ||
      (st = put(&d->chain, t.chain)) || (st = put(&d->leaf, t.leaf)) ||
      (st = put(&d->grid_items, t.grid_items)) || (st = put(&d->free_items, t.free_items)) ||
      (st = put(&d->points, pts)) || (st = put(&d->points_idx, t.free_order)))
    return st;
  return FC2D_OK;
}

fc2d_status poisson_setup(fc2d_plan_s* p, int Nb) {
  if (p->prm.precision != FC2D_FP64)
    return set_error(FC2D_ERR_UNSUPPORTED, "fc2d_poisson_plan: the Poisson solver needs an FP64 plan");
  const int nx = p->grid.nx, ny = p->grid.ny, MP = p->prm.M;
  if (Nb <= 0) Nb = nx;
  if (Nb < 16 || Nb > 65536) return set_error(FC2D_ERR_ARG, "fc2d_poisson_plan: bad n_b");
  poisson_destroy(p);
  auto* P = new PoissonState();
  P->Nb = Nb;
  P->MP = MP;
  const Curve& cv = p->curve;
  const double a0 = p->grid.a0, b0 = p->grid.b0, h = p->grid.h;
  const double two_pi = 2.0 * M_PI;
  auto fail = [&](fc2d_status s) {
    poisson_free(P);
    return s;
  };
  // nodes
  std::vector<double> x(Nb), y(Nb), x1(Nb), y1(Nb), diag(Nb);
  P->xy_host.assign(2 * (size_t)Nb, 0.0);
  for (int k = 0; k < Nb; ++k) {
    double t = two_pi * k / Nb, xx, yy, xd, yd, x2, y2;
    cv.eval(t, xx, yy);
    cv.eval_d(t, 1, xd, yd);
    cv.eval_d(t, 2, x2, y2);
    x[k] = xx;
    y[k] = yy;
    x1[k] = xd;
    y1[k] = yd;
    diag[k] = (x2 * yd - xd * y2) / (4.0 * M_PI * (xd * xd + yd * yd)) * (two_pi / Nb);
    P->xy_host[2 * k] = xx;
    P->xy_host[2 * k + 1] = yy;
  }
  // largest node spacing and the near bands
  double smax = 0.0;
  for (int k = 0; k < 4096; ++k) {
    double xd, yd;
    cv.eval_d(two_pi * k / 4096, 1, xd, yd);
    smax = std::max(smax, std::hypot(xd, yd));
  }
  P->s = two_pi / Nb * smax;
  P->delta = 5.0 * P->s;
  const int R = P->R, NR = R * Nb;
  std::vector<double> rx(NR), ry(NR), rx1(NR), ry1(NR);
  for (int m = 0; m < NR; ++m) {
    double t = two_pi * m / NR;
    cv.eval(t, rx[m], ry[m]);
    cv.eval_d(t, 1, rx1[m], ry1[m]);
  }
  std::vector<double> twb(2 * (size_t)Nb), twr(2 * (size_t)NR);
  for (int t = 0; t < Nb; ++t) {
    double ang = two_pi * t / Nb;
    twb[2 * t] = std::cos(ang);
    twb[2 * t + 1] = -std::sin(ang);
  }
  for (int t = 0; t < NR; ++t) {
    double ang = two_pi * t / NR;
    twr[2 * t] = std::cos(ang);
    twr[2 * t + 1] = std::sin(ang);
  }
  // u_p interpolation stencils at the nodes
  std::vector<int32_t> ui0(Nb), uj0(Nb);
  std::vector<double> uwx((size_t)Nb * MP), uwy((size_t)Nb * MP);
  const int off = (MP + 1) / 2 - 1;
  for (int k = 0; k < Nb; ++k) {
    int i0 = (int)std::floor((x[k] - a0) / h) - off;
    int j0 = (int)std::floor((y[k] - b0) / h) - off;
    i0 = std::min(std::max(i0, 0), nx - MP);
    j0 = std::min(std::max(j0, 0), ny - MP);
    ui0[k] = i0;
    uj0[k] = j0;
    double nxs[kMaxM], nys[kMaxM];
    for (int e = 0; e < MP; ++e) {
      nxs[e] = a0 + h * double(i0 + e);
      nys[e] = b0 + h * double(j0 + e);
    }
    lagr(nxs, MP, x[k], &uwx[(size_t)k * MP]);
    lagr(nys, MP, y[k], &uwy[(size_t)k * MP]);
  }
  // near points: inside points closer than delta; seeds from the nearest node of a
  // fine sampling of the curve (boxes around each sample)
  std::vector<uint8_t> inside((size_t)nx * ny, 0);
  for (int j = 0; j < ny; ++j)
    for (int k = p->row_iv_off[j]; k < p->row_iv_off[j + 1]; ++k)
      for (int i = p->row_iv[2 * k]; i <= p->row_iv[2 * k + 1]; ++i) inside[(size_t)j * nx + i] = 1;
  const int ns = std::max(p->prm.B, 4 * Nb);
  std::vector<double> seed((size_t)nx * ny, -1.0), best((size_t)nx * ny, 1e300);
  const double reach = P->delta + 2.0 * h;
  for (int q = 0; q < ns; ++q) {
    double t = two_pi * q / ns, cx, cy;
    cv.eval(t, cx, cy);
    int i0 = std::max(0, (int)std::floor((cx - reach - a0) / h));
    int i1 = std::min(nx - 1, (int)std::ceil((cx + reach - a0) / h));
    int j0 = std::max(0, (int)std::floor((cy - reach - b0) / h));
    int j1 = std::min(ny - 1, (int)std::ceil((cy + reach - b0) / h));
    for (int j = j0; j <= j1; ++j)
      for (int i = i0; i <= i1; ++i) {
        size_t l = (size_t)j * nx + i;
        if (!inside[l]) continue;
        double dx = a0 + h * double(i) - cx, dy = b0 + h * double(j) - cy;
        double d2 = dx * dx + dy * dy;
        if (d2 < best[l] && d2 <= reach * reach) {
          best[l] = d2;
          seed[l] = t;
        }
      }
  }
  std::vector<int32_t> cl;
  std::vector<double> qx, qy, tq;
  for (size_t l = 0; l < seed.size(); ++l)
    if (seed[l] >= 0) {
      cl.push_back((int32_t)l);
      qx.push_back(a0 + h * double(l % nx));
      qy.push_back(b0 + h * double(l / nx));
      tq.push_back(seed[l]);
    }
  std::vector<int> conv;
  fc2d_status st = foot_newton_gpu(cv, qx, qy, tq, conv, two_pi / ns);
  if (st) return fail(st);
  std::vector<uint8_t> near((size_t)nx * ny, 0);
  std::vector<int32_t> mid, close;
  std::vector<double> cgeo, cz, cw;  // foot and normal, e^{i theta}, Lagrange weights
  P->close_nodes.assign(MP, 0.0);
  for (int j = 1; j < MP; ++j) P->close_nodes[j] = (P->delta + P->s * (j - 1)) / R;
  for (size_t n = 0; n < cl.size(); ++n) {
    double fx, fy;
    cv.eval(tq[n], fx, fy);
    double eta = std::hypot(qx[n] - fx, qy[n] - fy);
    if (!(eta < P->delta)) continue;
    if (!conv[n]) return fail(set_error(FC2D_ERR_NOT_CONVERGED, "Poisson setup: foot search"));
    near[cl[n]] = 1;
    if (eta >= P->delta / R) {
      mid.push_back(cl[n]);
    } else {
      double t = std::fmod(tq[n], two_pi);
      if (t < 0) t += two_pi;
      double xd, yd;
      cv.eval_d(t, 1, xd, yd);
      double sp = std::hypot(xd, yd);
      close.push_back(cl[n]);
      cgeo.insert(cgeo.end(), {fx, fy, yd / sp, -xd / sp});
      cz.insert(cz.end(), {std::cos(t), std::sin(t)});
      double w[kMaxM];
      lagr(P->close_nodes.data(), MP, eta, w);
      cw.insert(cw.end(), w, w + MP);
    }
  }
  std::vector<int32_t> far;
  for (size_t l = 0; l < inside.size(); ++l)
    if (inside[l] && !near[l]) far.push_back((int32_t)l);
  // partitions of the sums, in grid units; the point lists in their leaves' order
  auto grid = [&](const std::vector<double>& v, double o) {
    std::vector<double> r(v.size());
    for (size_t k = 0; k < v.size(); ++k) r[k] = (v[k] - o) / h;
    return r;
  };
  std::vector<double> px, py;
  for (size_t n = 0; n < close.size(); ++n)
    for (int j = 1; j < MP; ++j) {
      px.push_back((cgeo[4 * n] - P->close_nodes[j] * cgeo[4 * n + 2] - a0) / h);
      py.push_back((cgeo[4 * n + 1] - P->close_nodes[j] * cgeo[4 * n + 3] - b0) / h);
    }
  auto partition = [&](std::vector<int32_t>& lin, const std::vector<double>& X,
                       const std::vector<double>& Y, const std::vector<double>& fx,
                       const std::vector<double>& fy) {
    DlpTree t = dlp_tree(grid(X, a0), grid(Y, b0), lin, nx, fx, fy, std::max(nx, ny));
    lin.swap(t.grid_order);
    return t;
  };
  // the two side by side
  auto far_tree = std::async(std::launch::async | std::launch::deferred,
                             [&] { return partition(far, x, y, {}, {}); });
  const DlpTree tn = partition(mid, rx, ry, px, py);
  const DlpTree tf = far_tree.get();
  P->n_far = (int64_t)far.size();
  P->n_mid = (int64_t)mid.size();
  P->n_close = (int64_t)close.size();
  if ((st = up(P, &P->bx, x)) || (st = up(P, &P->by, y)) || (st = up(P, &P->bx1, x1)) ||
      (st = up(P, &P->by1, y1)) || (st = up(P, &P->rx, rx)) || (st = up(P, &P->ry, ry)) ||
      (st = up(P, &P->rx1, rx1)) || (st = up(P, &P->ry1, ry1)) || (st = up(P, &P->twb, twb)) ||
      (st = up(P, &P->twr, twr)) || (st = up(P, &P->ui0, ui0)) || (st = up(P, &P->uj0, uj0)) ||
      (st = up(P, &P->uwx, uwx)) || (st = up(P, &P->uwy, uwy)) ||
      (st = up(P, &P->far_lin, far)) || (st = up(P, &P->mid_lin, mid)) ||
      (st = up(P, &P->close_lin, close)) || (st = up(P, &P->close_z, cz)) ||
      (st = up(P, &P->close_w, cw)) || (st = up_tree(P, &P->far, tf, {}, {})) ||
      (st = up_tree(P, &P->near, tn, px, py)) || (st = alloc(P, &P->close_v, px.size())) ||
      (st = alloc(P, &P->spec, (size_t)ny * row_pitch(p))) ||
      (st = alloc(P, &P->exps, fx_exps(nx, ny, 1))) || (st = alloc(P, &P->qB, Nb)) || (st = alloc(P, &P->qR, NR)) ||
      (st = up(P, &P->posB, grid_units(x, y, a0, b0, h))) ||
      (st = up(P, &P->posR, grid_units(rx, ry, a0, b0, h))))
    return fail(st);
  double* ddiag = nullptr;
  int n_sm = 1;
  cudaDeviceGetAttribute(&n_sm, cudaDevAttrMultiProcessorCount, p->device);
  P->gm.n = Nb;
  P->gm.rows = gmres_rows(Nb, n_sm);
  P->gm.n_blk = (Nb + P->gm.rows - 1) / P->gm.rows;
  const size_t n_blk = P->gm.n_blk;
  if ((st = up(P, &ddiag, diag)) || (st = alloc(P, &P->A, (size_t)Nb * Nb)) ||
      (st = alloc(P, &P->gm.V, (size_t)(kGmresMax + 1) * Nb)) ||
      (st = alloc(P, &P->gm.w, Nb)) || (st = alloc(P, &P->gm.dev, 1)) || (st = alloc(P, &P->gm.norm, n_blk)) ||
      (st = alloc(P, &P->gm.part[0], n_blk * (kGmresMax + 1))) ||
      (st = alloc(P, &P->gm.part[1], n_blk * (kGmresMax + 1))) ||
      (st = alloc(P, &P->g, Nb)) ||
      (st = alloc(P, &P->phi, Nb)) || (st = alloc(P, &P->ghat, 2 * (Nb / 2 + 1))) ||
      (st = alloc(P, &P->phiR, NR)) || (st = alloc(P, &P->ab, (size_t)Nb)) ||
      (st = alloc(P, &P->abR, (size_t)NR)) || (st = alloc(P, &P->c00, 1024)))
    return fail(st);
  const size_t cf = tf.box.size() * 2 * kDlpOrder, cn = tn.box.size() * 2 * kDlpOrder;
  unsigned long long* sums = nullptr;
  if ((st = alloc(P, &sums, cf + cn + 4))) return fail(st);
  P->sum_bytes = (cf + cn + 4) * sizeof(*sums);
  P->far.coef = sums;
  P->near.coef = sums + cf;
  P->far.mag = reinterpret_cast<unsigned*>(sums + cf + cn);
  P->near.mag = reinterpret_cast<unsigned*>(sums + cf + cn + 1);
  P->mags = reinterpret_cast<unsigned*>(sums + cf + cn + 2);
  k_bie_matrix<<<dim3((Nb + 255) / 256, Nb), 256>>>(Nb, P->bx, P->by, P->bx1, P->by1, ddiag,
                                                    P->A);
  P->gm.A = P->A;
  if ((st = cuda_check(cudaDeviceSynchronize(), "BIE matrix"))) return fail(st);
  p->poisson = P;
  return FC2D_OK;
}

fc2d_status poisson_solve(fc2d_plan_s* p, int n_f, const double* fg, const double* fb,
                          const double* gn, double* u, double* phi_out, void* inter,
                          cudaStream_t s) {
  auto* P = static_cast<PoissonState*>(p->poisson);
  const int nx = p->grid.nx, ny = p->grid.ny, Nb = P->Nb, MP = P->MP, NR = P->R * Nb;
  const double a0 = p->grid.a0, b0 = p->grid.b0, h = p->grid.h;
  if (n_f > 1024) return set_error(FC2D_ERR_ARG, "fc2d_poisson: n_f <= 1024");
  // u_p (forward rows already in `inter` from the caller): the forward columns, the symbol,
  // the inverse columns and rows, one function at a time
  FftArgs fa = fft_args(p);
  const size_t slab = (size_t)ny * fa.pitch;
  auto* in = static_cast<double2*>(inter);
  FftArgs inv = fa;
  fa.exps = inv.exps = P->exps;
  fa.opitch = inv.opitch = fa.pitch;
  inv.fxs = FxFactor{0, 0, 0};
  for (int f = 0; f < n_f; ++f) {
    {
      ProfScope ps(p, "poisson_cols", s);
      launch_fft_cols(fa, 1, true, in + f * slab, P->spec, s);
      k_symbol<<<dim3((nx / 2 + 128) / 128, (ny + kSymbolRows - 1) / kSymbolRows), 128, 0, s>>>(
          nx / 2 + 1, ny, fa.pitch, P->spec, in + f * slab, P->c00 + f, 2.0 * M_PI / (nx * h),
          2.0 * M_PI / (ny * h));
      launch_fft_cols(inv, 1, true, in + f * slab, P->spec, s);
    }
    {
      ProfScope ps(p, "poisson_rows", s);
      launch_inverse_rows(fa, 1, P->spec, P->c00 + f, a0, b0, h, u + (size_t)f * nx * ny, s);
    }
  }
  fc2d_status st = cuda_check(cudaGetLastError(), "Poisson particular solution");
  if (st) return st;
  const unsigned gb = (unsigned)((Nb + 255) / 256);
  for (int f = 0; f < n_f; ++f) {
    double* uf = u + (size_t)f * nx * ny;
    k_up_nodes<<<(unsigned)((Nb + 7) / 8), 128, 0, s>>>(Nb, MP, nx, P->ui0, P->uj0, P->uwx, P->uwy, uf,
                                  gn + (size_t)f * Nb, P->g);
    {
      ProfScope ps(p, "bie_gmres", s);
      if ((st = gmres_solve(P->gm, P->g, P->phi, 1e-14, &P->last_iters, &P->last_resid, s)))
        return st;
    }
    if (phi_out) cudaMemcpyAsync(phi_out + (size_t)f * Nb, P->phi, Nb * 8, cudaMemcpyDeviceToDevice, s);
    // density refinement and node coefficients
    cudaMemsetAsync(P->far.coef, 0, P->sum_bytes, s);
    auto dft = [&](const double* v, unsigned* mag) {
      k_density_dft<<<(unsigned)((Nb / 2 + 4) / 4), 128, 0, s>>>(Nb, v, (const double2*)P->twb,
                                                                 (double2*)P->ghat, mag);
    };
    dft(P->phi, P->mags + 1);
    k_density_refine<<<(unsigned)((NR / 4 + 4) / 4), 128, 0, s>>>(
        Nb, NR, (const double2*)P->ghat, (const double2*)P->twr, P->phiR);
    launch_node_coef(Nb, P->bx1, P->by1, P->phi, P->qB, P->ab, P->far.mag, s);
    launch_node_coef(NR, P->rx1, P->ry1, P->phiR, P->qR, P->abR, P->near.mag, s);
    {
      ProfScope ps(p, "dlp_far", s);
      if (P->n_far) {
        launch_dlp_expand(P->far, P->qB, s);
        launch_dlp_grid(P->far, P->far_lin, nx, h, P->posB, P->ab, uf, s);
      }
    }
    {
      ProfScope ps(p, "dlp_near", s);
      if (P->n_mid || P->n_close) {
        launch_dlp_expand(P->near, P->qR, s);
        launch_dlp_grid(P->near, P->mid_lin, nx, h, P->posR, P->abR, uf, s);
      }
      if (P->n_close) {
        launch_dlp_free(P->near, h, P->posR, P->abR, P->close_v, s);
        // boundary values g - u_p: reuse ghat for their coefficients
        dft(P->g, P->mags);
        launch_close((int)P->n_close, P->close_lin, (const double2*)P->close_z, P->close_w, MP,
                     P->close_v, Nb, (const double2*)P->ghat, P->mags, uf, s);
      }
    }
    k_zero_outside<<<ny, 256, 0, s>>>(nx, p->dev.row_iv_off, p->dev.row_iv, uf);
  }
  return cuda_check(cudaGetLastError(), "Poisson solve");
}

// inverse real 2D-DFT rows (after an inverse column pass)
bool launch_inverse_rows_fx(const FftArgs& fa, int n_f, const void* inter, const double* c00,
                            double a0, double b0, double h, double* out, const int32_t* off,
                            const int32_t* points, int ld, cudaStream_t s);
void launch_inverse_rows_mixed(const FftArgs& fa, int n_f, const void* inter, const double* c00,
                               double a0, double b0, double h, double* out, const int32_t* off,
                               const int32_t* points, int ld, cudaStream_t s);

void launch_inverse_rows(const FftArgs& fa, int n_f, const void* inter, const double* c00,
                         double a0, double b0, double h, double* out, cudaStream_t s) {
  if (!launch_inverse_rows_fx(fa, n_f, inter, c00, a0, b0, h, out, nullptr, nullptr, 0, s))
    launch_inverse_rows_mixed(fa, n_f, inter, c00, a0, b0, h, out, nullptr, nullptr, 0, s);
}

int poisson_nb(const fc2d_plan_s* p) {
  return p->poisson ? static_cast<const PoissonState*>(p->poisson)->Nb : 0;
}

const double* poisson_nodes(const fc2d_plan_s* p) {
  return p->poisson ? static_cast<const PoissonState*>(p->poisson)->xy_host.data() : nullptr;
}

void poisson_stats(const fc2d_plan_s* p, int* iters, double* resid, int64_t* n_near) {
  auto* P = static_cast<const PoissonState*>(p->poisson);
  if (iters) *iters = P ? P->last_iters : 0;
  if (resid) *resid = P ? P->last_resid : 0.0;
  if (n_near) *n_near = P ? P->n_mid + P->n_close : 0;
}

}  // namespace fc2d
