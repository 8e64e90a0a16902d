// Fourier Forwarding (Section 4.2): the interior propagator U_FC combined with the
// near-boundary solver U_B by eq. (4.9), large step after large step (U_B in FP64, U_FC and the
// squares in 64-bit fixed point).
//
// Large step j (T_j = j Delta T, Delta T = n_c h / c, S = 8 n_c small steps of
// Delta t = Delta T / S, i.e. c Delta t = h/8, CFL 0.125 as in Section 4.2.1):
//   1. the 2D-FC spectra of u(T_j) and u_t(T_j) (eq. (4.10)) with the Dirichlet data
//      g(T_j) and its time derivative (capi.cu wave_spectra);
//   2. for each small step s: the modal solution a(s Delta t) (eq. (4.12), w the square
//      root of the paper's alpha) and its inverse DFT at U_B's interface points
//      (fx_wave.cu; with squares fx_squares.cu), which feed the step;
//   3. the U_B small step (k_ub_advance, on u and its increment): u^{n+1} = 2u^n - u^{n-1} + (h/8)^2 L(u^n)
//      - 0.3 D(u^n - u^{n-1}), the first step of the solve by the Taylor start
//      u^1 = u^0 + dt u_t^0 + (h/8)^2/2 L(u^0); L and D are the plan-time operators of
//      wave_band.cpp (rows per unknown, columns keyed unknown / interface grid point /
//      boundary point);
//   4. U_FC(T_{j+1}) and dU_FC/dt on the grid, one further U_B step for the time
//      derivative (u^{N+1} - u^{N-1})/(2 dt), and the merge: at the band points nearer
//      than delta = n_c h to the curve the grid takes U_B's values (slaved points by their
//      boundary polynomial).
// The U_B state is function-minor ([unknown][n_f]), so that a warp reads one operator
// row for 32 functions with coalesced loads.
#include <cuda_runtime.h>

#include <algorithm>
#include <cmath>
#include <cstdint>
#include <cstring>
#include <map>
#include <memory>
#include <string>
#include <type_traits>

#include "fc2d_kernels.cuh"
#include "fx_squares.h"
#include "plan_internal.h"
#include "wave_band.h"

namespace fc2d {

fc2d_status wave_spectra(fc2d_plan_s* p, int n_f, const double* u, const double* ub,
                         const double* ut, const double* utb, void* spec, cudaStream_t s);
namespace {

struct DevCsr {
  int32_t* off = nullptr;
  uint32_t* col = nullptr;
  double* w = nullptr;
  int64_t rows = 0, nnz = 0;
};

struct DevSquares {
  SquareSet host;
  int32_t* origin = nullptr;        // [n_sq][2] (row, column) of the first grid point
  int32_t* served_off = nullptr;    // [n_sq + 1]
  int32_t* served_at = nullptr;     // the served interface point (index into iface_lin)
  int32_t* served_local = nullptr;
  double* A = nullptr;              // [C][d]
  double* Q = nullptr;              // [d][d]
  int32_t* tw = nullptr;            // exp(-2 pi i t / P) 2^60 in limbs, t < P (fx.cuh)
  int32_t* rows = nullptr;          // [n_sq][2]: first and last box row holding served points
  int n = 0, max_rows = 0;          // squares; the most rows any of them needs
  SquareArgs args() const {
    return {n, origin, A, Q, reinterpret_cast<const int4*>(tw), served_off, served_at, served_local, rows};
  }
};

// An operator entry of the solve: the weight and the row of the state it multiplies
struct __align__(16) UbEntry {
  double w;
  int32_t col, pad;
};
struct DevOp {
  int2* row = nullptr;   // [rows + 1] (x: the row's first entry, y: its first outer one)
  UbEntry* e = nullptr;
};

struct DevBand {
  WaveBand host;
  DevCsr S;                         // with keys (the merge)
  DevOp L, D;                       // with state rows (the small step)
  int32_t* unknown_lin = nullptr;
  int32_t* near_lin = nullptr;
  int32_t* near_src = nullptr;
  int32_t* iface_off = nullptr;     // [ny + 1]: the interface points of each grid row
  int32_t* iface_lin = nullptr;     // their linear indices, ascending
  std::unique_ptr<DevSquares> sq;   // the small-square procedure's squares (mode 1)
};

struct Scratch {
  int n_f = 0;
  size_t bytes = 0;
  void* base = nullptr;
};

struct WaveState {
  std::map<std::pair<int, int>, std::unique_ptr<DevBand>> bands;  // by (n_c, interface mode)
  Scratch scr;
};

template <typename T>
fc2d_status upload(T** dst, const std::vector<T>& src) {
  *dst = nullptr;
  const size_t n = std::max<size_t>(1, src.size());
  if (cudaMalloc(dst, n * sizeof(T)) != cudaSuccess)
    return set_error(FC2D_ERR_NOMEM, "wave band: cudaMalloc failed");
  if (!src.empty() && cudaMemcpy(*dst, src.data(), src.size() * sizeof(T), cudaMemcpyHostToDevice) != cudaSuccess)
    return set_error(FC2D_ERR_CUDA, "wave band: upload failed");
  return FC2D_OK;
}

fc2d_status upload_csr(DevCsr& d, const Csr& h) {
  d.rows = (int64_t)h.off.size() - 1;
  d.nnz = (int64_t)h.w.size();
  fc2d_status st;
  if ((st = upload(&d.off, h.off)) || (st = upload(&d.col, h.col)) || (st = upload(&d.w, h.w)))
    return st;
  return FC2D_OK;
}

// position of a grid point in the band's interface list
int32_t iface_index(const WaveBand& b, int32_t lin) {
  return (int32_t)(std::lower_bound(b.iface_lin.begin(), b.iface_lin.end(), lin) - b.iface_lin.begin());
}

// The operator with its columns as rows of the state (unknowns, interface points, boundary
// points); each row's entries from column `outer` on come last
fc2d_status upload_op(DevOp& d, const Csr& h, const WaveBand& b, int32_t outer) {
  const int32_t n = (int32_t)b.unknown_lin.size(), ni = (int32_t)b.iface_lin.size();
  std::vector<UbEntry> e(h.w.size());
  std::vector<int2> row(h.off.size());
  for (size_t r = 0; r < h.off.size(); ++r) {
    row[r] = {h.off[r], h.off[r]};
    if (r + 1 == h.off.size()) break;
    for (int k = h.off[r]; k < h.off[r + 1]; ++k) {
      const uint32_t kind = h.col[k] & kKeyKind;
      const int32_t idx = (int32_t)(h.col[k] & kKeyIndex);
      e[k] = {h.w[k], kind == kKeyUnknown ? idx : kind == kKeyGrid ? n + iface_index(b, idx) : n + ni + idx, 0};
    }
    row[r].y = (int)(std::stable_partition(e.begin() + h.off[r], e.begin() + h.off[r + 1],
                                           [&](const UbEntry& v) { return v.col < outer; }) - e.begin());
  }
  fc2d_status st = upload(&d.row, row);
  return st ? st : upload(&d.e, e);
}

void free_csr(DevCsr& d) {
  cudaFree(d.off);
  cudaFree(d.col);
  cudaFree(d.w);
}

WaveState* state(fc2d_plan_s* p) {
  if (!p->wave) p->wave = new WaveState();
  return static_cast<WaveState*>(p->wave);
}

// The band reach (grid units) for an interface mode: 0 full U_FC at every small step,
// 1 the small squares (whose service needs interface points at sqrt(2) n_c h or more).
int reach_cells(int n_c, int mode) {
  return mode ? (int)std::ceil(std::sqrt(2.0) * n_c) + 2 : n_c + kUbBandExtra;
}

fc2d_status upload_squares(const fc2d_plan_s* p, DevBand& b, int n_c) {
  auto q = std::make_unique<DevSquares>();
  fc2d_status st = build_wave_squares(p, b.host, n_c, q->host);
  if (st) return st;
  const SquareSet& h = q->host;
  q->n = (int)h.origin_j.size();
  std::vector<int32_t> origin(2 * (size_t)q->n);
  for (int k = 0; k < q->n; ++k) {
    origin[2 * k] = h.origin_j[k];
    origin[2 * k + 1] = h.origin_i[k];
  }
  std::vector<int32_t> rows(2 * (size_t)q->n);
  for (int k = 0; k < q->n; ++k) {
    int lo = h.P, hi = -1;
    for (int i = h.served_off[k]; i < h.served_off[k + 1]; ++i) {
      lo = std::min(lo, h.served_local[i] / h.P);
      hi = std::max(hi, h.served_local[i] / h.P);
    }
    rows[2 * k] = lo;
    rows[2 * k + 1] = hi;
    q->max_rows = std::max(q->max_rows, hi - lo + 1);
  }
  std::vector<int32_t> at;
  for (int32_t lin : h.served_lin) at.push_back(iface_index(b.host, lin));
  if ((st = upload(&q->origin, origin)) || (st = upload(&q->served_off, h.served_off)) ||
      (st = upload(&q->served_at, at)) || (st = upload(&q->served_local, h.served_local)) ||
      (st = upload(&q->A, h.A)) || (st = upload(&q->Q, h.Q)) || (st = upload(&q->tw, fx_twiddle_table(h.P))) ||
      (st = upload(&q->rows, rows)))
    return st;
  b.sq = std::move(q);
  return FC2D_OK;
}

fc2d_status get_band(fc2d_plan_s* p, int n_c, int mode, DevBand** out) {
  WaveState* W = state(p);
  auto it = W->bands.find({n_c, mode});
  if (it != W->bands.end()) {
    *out = it->second.get();
    return FC2D_OK;
  }
  auto b = std::make_unique<DevBand>();
  fc2d_status st = build_wave_band(p, n_c, reach_cells(n_c, mode), b->host);
  if (st) return st;
  if (mode && (st = upload_squares(p, *b, n_c))) return st;
  // operator entries of a grid kind must index the grid (30 bits), boundary data too
  if ((int64_t)p->grid.nx * p->grid.ny > (int64_t)kKeyIndex || p->n_bdry > (int64_t)kKeyIndex)
    return set_error(FC2D_ERR_UNSUPPORTED, "wave band: grid too large for the operator keys");
  if ((st = upload_csr(b->S, b->host.S)) || (st = upload(&b->unknown_lin, b->host.unknown_lin)) ||
      (st = upload(&b->near_lin, b->host.near_lin)) || (st = upload(&b->near_src, b->host.near_src)))
    return st;
  const std::vector<int32_t>& q = b->host.iface_lin;
  std::vector<int32_t> off(p->grid.ny + 1);
  for (int j = 0; j <= p->grid.ny; ++j)
    off[j] = (int32_t)(std::lower_bound(q.begin(), q.end(), (int64_t)j * p->grid.nx) - q.begin());
  if ((st = upload(&b->iface_off, off)) || (st = upload(&b->iface_lin, q)) ||
      (st = upload_op(b->L, b->host.L, b->host, (int32_t)(b->host.unknown_lin.size() + q.size()))) ||
      (st = upload_op(b->D, b->host.D, b->host, (int32_t)b->host.unknown_lin.size())))
    return st;
  *out = b.get();
  W->bands[{n_c, mode}] = std::move(b);
  return FC2D_OK;
}

// ------------------------------------------------------------------------- //
// Kernels
// ------------------------------------------------------------------------- //

// U_B state from grids: out[r][f] = grid[f][lin[r]]
__global__ void k_ub_gather(int64_t n, int n_f, int64_t grid_stride, const int32_t* __restrict__ lin,
                            const double* __restrict__ grid, double* __restrict__ out) {
  const int64_t t = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
  if (t >= n * n_f) return;
  const int64_t r = t / n_f;
  const int f = (int)(t - r * n_f);
  out[t] = grid[(size_t)f * grid_stride + lin[r]];
}

// value of an operator column for function f
__device__ __forceinline__ double ub_value(uint32_t key, int f, int n_f, int64_t grid_stride,
                                           int64_t n_b, const double* __restrict__ u,
                                           const double* __restrict__ grid,
                                           const double* __restrict__ g) {
  const uint32_t kind = key & kKeyKind, idx = key & kKeyIndex;
  if (kind == kKeyUnknown) return u[(size_t)idx * n_f + f];
  if (kind == kKeyGrid) return grid[(size_t)f * grid_stride + idx];
  return g ? g[(size_t)f * n_b + idx] : 0.0;
}

// One U_B small step for every (unknown r, function f), thread t = r n_f + f, on u and
// w = u^n - u^{n-1}.  The columns of the operators are rows of the state: the N unknowns, the n_i
// interface points (U_FC at u's time), then boundary points (g: Dirichlet data [n_f][n_b] at u's
// time, NULL: zero).
//   mode 0: w' = dt u_t + cdt2/2 L(u)     (Taylor start; W holds u_t)
//   mode 1: w' = w + cdt2 L(u) - sigma D(w)
//   mode 2: (w' + w)/(2 dt), w' of mode 1, to Uout (the time derivative at u's time)
// and u' = u + w'.  The FP64 pipe bounds it: w saves the difference u - u_prev of every
// D entry (38 multiply-adds and 33 additions per value before), and does not cancel.
// UbRows (the solve): function-minor rows, U [N + n_i][n_f] and Uold the step before (only its
// interface rows are read), W [N][n_f]; Wout receives w'.  UbGrids (a caller's own arrays): U and
// Uold are u^n and u^{n-1} of the unknowns, the interface points iface[n_i] lie in grid and
// grid_prev [n_f][stride], W is u_t (mode 0 only).
struct UbRows {};
struct UbGrids {
  const double *grid, *grid_prev;
  int64_t stride;
  const int32_t* iface;
};
template <typename State>
__global__ void __launch_bounds__(256) k_ub_advance(
    int mode, int n, int n_i, int n_f, int64_t n_b, const int2* __restrict__ Lrow,
    const UbEntry* __restrict__ Le, const int2* __restrict__ Drow, const UbEntry* __restrict__ De,
    const double* __restrict__ U, const double* __restrict__ Uold, const double* __restrict__ W,
    const double* __restrict__ g, double cdt2, double dt, double sigma, double* __restrict__ Uout,
    double* __restrict__ Wout, State state) {
  constexpr bool GRIDS = std::is_same<State, UbGrids>::value;
  const int64_t t = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
  if (t >= (int64_t)n * n_f) return;
  const int r = (int)(t / n_f), f = (int)(t - (int64_t)r * n_f);
  const double u = U[t], w = GRIDS && mode ? u - Uold[t] : W[t];
  double lap = 0.0, dis = 0.0;
  const double *Uf = U + f, *Wf = W + f;
  // GRIDS: the interface point of a column in a grid
  auto face = [&](int col) -> size_t {
    if constexpr (GRIDS) return (size_t)f * state.stride + __ldg(state.iface + (col - n));
    else return 0;
  };
  // u at a column, D's difference at a column of each kind
  auto value = [&](int col) {
    if constexpr (GRIDS) return col >= n ? state.grid[face(col)] : Uf[(size_t)col * n_f];
    else return Uf[(size_t)col * n_f];
  };
  auto step = [&](int col) {
    const size_t o = (size_t)col * n_f;
    if constexpr (GRIDS) return Uf[o] - Uold[o + f];
    else return Wf[o];
  };
  auto face_step = [&](int col) {
    if constexpr (GRIDS) return state.grid[face(col)] - state.grid_prev[face(col)];
    else return U[(size_t)col * n_f + f] - Uold[(size_t)col * n_f + f];
  };
  const int2 l0 = __ldg(Lrow + r);
  const int l1 = __ldg(&Lrow[r + 1].x);
#pragma unroll 4
  for (int k = l0.x; k < l0.y; ++k) {
    const UbEntry e = Le[k];
    lap += e.w * value(e.col);
  }
  if (g)  // boundary points
    for (int k = l0.y; k < l1; ++k) {
      const UbEntry e = Le[k];
      lap += e.w * __ldg(g + (size_t)f * n_b + (e.col - n - n_i));
    }
  double wn;
  if (mode == 0) {
    wn = dt * w + 0.5 * cdt2 * lap;
  } else {
    const int2 d0 = __ldg(Drow + r);
    const int d1 = __ldg(&Drow[r + 1].x);
#pragma unroll 4
    for (int k = d0.x; k < d0.y; ++k) {
      const UbEntry e = De[k];
      dis += e.w * step(e.col);
    }
    for (int k = d0.y; k < d1; ++k) {  // interface points
      const UbEntry e = De[k];
      dis += e.w * face_step(e.col);
    }
    wn = w + cdt2 * lap - sigma * dis;
    if (mode == 2) {
      Uout[t] = (wn + w) / (2.0 * dt);
      return;
    }
  }
  if (!GRIDS) Wout[t] = wn;
  Uout[t] = u + wn;
}

// The merge of eq. (4.9) at the band points nearer than delta to the curve: unknowns
// copy U_B's value and time derivative, slaved points evaluate their boundary
// polynomial on (U_B values, the grid's U_FC values at interface points, Dirichlet data)
// and on the time derivatives of the same.
__global__ void k_ff_merge(int64_t n_near, int n_f, int64_t grid_stride, int64_t n_b,
                           const int32_t* __restrict__ near_lin, const int32_t* __restrict__ near_src,
                           const int32_t* __restrict__ Soff, const uint32_t* __restrict__ Scol,
                           const double* __restrict__ Sw, const double* __restrict__ uB,
                           const double* __restrict__ utB, const double* __restrict__ g,
                           const double* __restrict__ gt, double* __restrict__ u,
                           double* __restrict__ ut) {
  const int64_t t = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
  if (t >= n_near * n_f) return;
  const int64_t q = t / n_f;
  const int f = (int)(t - q * n_f);
  const int32_t src = near_src[q];
  double v, vt;
  if (src >= 0) {
    v = uB[(size_t)src * n_f + f];
    vt = utB[(size_t)src * n_f + f];
  } else {
    const int s = -1 - src;
    v = 0.0;
    vt = 0.0;
    for (int k = Soff[s]; k < Soff[s + 1]; ++k) {
      v += Sw[k] * ub_value(Scol[k], f, n_f, grid_stride, n_b, uB, u, g);
      vt += Sw[k] * ub_value(Scol[k], f, n_f, grid_stride, n_b, utB, ut, gt);
    }
  }
  const size_t o = (size_t)f * grid_stride + near_lin[q];
  u[o] = v;
  ut[o] = vt;
}

// Zero the grid points outside the domain (row intervals of the inside points).
__global__ void k_zero_outside(int nx, int ny, int n_f, const int32_t* __restrict__ iv_off,
                               const int32_t* __restrict__ iv, double* __restrict__ a,
                               double* __restrict__ b) {
  const int j = blockIdx.x, f = blockIdx.y;
  double* ra = a + ((size_t)f * ny + j) * nx;
  double* rb = b + ((size_t)f * ny + j) * nx;
  for (int i = threadIdx.x; i < nx; i += blockDim.x) {
    bool in = false;
    for (int k = iv_off[j]; k < iv_off[j + 1]; ++k) in |= (i >= iv[2 * k] && i <= iv[2 * k + 1]);
    if (!in) {
      ra[i] = 0.0;
      rb[i] = 0.0;
    }
  }
}

unsigned blocks(int64_t n, int t) { return (unsigned)((n + t - 1) / t); }

}  // namespace

void wave_destroy(fc2d_plan_s* p) {
  wave_modes_destroy(p);
  if (!p->wave) return;
  auto* W = static_cast<WaveState*>(p->wave);
  for (auto& kv : W->bands) {
    DevBand& b = *kv.second;
    free_csr(b.S);
    for (DevOp* o : {&b.L, &b.D}) {
      cudaFree(o->row);
      cudaFree(o->e);
    }
    cudaFree(b.unknown_lin);
    cudaFree(b.near_lin);
    cudaFree(b.near_src);
    cudaFree(b.iface_off);
    cudaFree(b.iface_lin);
    if (b.sq) {
      DevSquares& q = *b.sq;
      for (void* ptr : {(void*)q.origin, (void*)q.served_off, (void*)q.served_at,
                        (void*)q.served_local, (void*)q.A, (void*)q.Q, (void*)q.tw, (void*)q.rows})
        cudaFree(ptr);
    }
  }
  cudaFree(W->scr.base);
  delete W;
  p->wave = nullptr;
}

}  // namespace fc2d

using namespace fc2d;

namespace {

fc2d_status wave_checks(fc2d_plan_t p, int n_c, const char* who) {
  if (!p) return set_error(FC2D_ERR_ARG, std::string(who) + ": null plan");
  if (n_c < 1 || n_c > 256) return set_error(FC2D_ERR_ARG, std::string(who) + ": n_c in 1..256");
  if (p->prm.precision != FC2D_FP64)
    return set_error(FC2D_ERR_UNSUPPORTED, std::string(who) + ": FP64 plans only");
  return FC2D_OK;
}

}  // namespace

extern "C" fc2d_status fc2d_wave_band_info(fc2d_plan_t p, int n_c, int interface_mode,
                                           int64_t* counts) {
  fc2d_status st = wave_checks(p, n_c, "fc2d_wave_band_info");
  if (st) return st;
  if (!counts) return set_error(FC2D_ERR_ARG, "fc2d_wave_band_info: null argument");
  if (interface_mode < 0 || interface_mode > 1)
    return set_error(FC2D_ERR_ARG, "fc2d_wave_band_info: interface_mode 0 or 1");
  cudaSetDevice(p->device);
  DevBand* b;
  if ((st = get_band(p, n_c, interface_mode, &b))) return st;
  counts[0] = (int64_t)b->host.unknown_lin.size();
  counts[1] = (int64_t)b->host.slaved_lin.size();
  counts[2] = (int64_t)b->host.iface_lin.size();
  counts[3] = (int64_t)b->host.near_lin.size();
  counts[4] = b->sq ? (int64_t)b->sq->n : 0;
  return FC2D_OK;
}

extern "C" fc2d_status fc2d_wave_band_points(fc2d_plan_t p, int n_c, int interface_mode,
                                             int32_t* unknown_lin,
                                             int32_t* slaved_lin, int32_t* iface_lin,
                                             int32_t* near_lin) {
  fc2d_status st = wave_checks(p, n_c, "fc2d_wave_band_points");
  if (st) return st;
  if (interface_mode < 0 || interface_mode > 1)
    return set_error(FC2D_ERR_ARG, "fc2d_wave_band_points: interface_mode 0 or 1");
  cudaSetDevice(p->device);
  DevBand* b;
  if ((st = get_band(p, n_c, interface_mode, &b))) return st;
  const WaveBand& w = b->host;
  auto cp = [](int32_t* dst, const std::vector<int32_t>& v) {
    if (dst && !v.empty()) std::memcpy(dst, v.data(), v.size() * sizeof(int32_t));
  };
  cp(unknown_lin, w.unknown_lin);
  cp(slaved_lin, w.slaved_lin);
  cp(iface_lin, w.iface_lin);
  cp(near_lin, w.near_lin);
  return FC2D_OK;
}

extern "C" fc2d_status fc2d_wave_ub_step(fc2d_plan_t p, int n_c, int n_f, int mode, double c,
                                         const double* u, const double* u_prev, const double* ut,
                                         const double* grid, const double* grid_prev,
                                         const double* g, double* out, void* stream) {
  fc2d_status st = wave_checks(p, n_c, "fc2d_wave_ub_step");
  if (st) return st;
  if ((st = check_nf(p, n_f))) return st;
  if (mode < 0 || mode > 2 || !u || !grid || !out || (mode == 0 && !ut) ||
      (mode > 0 && (!u_prev || !grid_prev)) || !(c > 0))
    return set_error(FC2D_ERR_ARG, "fc2d_wave_ub_step: bad mode, c or null pointer");
  cudaSetDevice(p->device);
  DevBand* b;
  if ((st = get_band(p, n_c, 0, &b))) return st;
  const double h = p->grid.h, cdt2 = (kUbCfl * h) * (kUbCfl * h);
  const double dt = kUbCfl * h / c;
  const int64_t n = (int64_t)b->host.unknown_lin.size();
  if (n > 0)
    k_ub_advance<<<blocks(n * n_f, 256), 256, 0, (cudaStream_t)stream>>>(
        mode, (int)n, (int)b->host.iface_lin.size(), n_f, p->n_bdry, b->L.row, b->L.e, b->D.row, b->D.e,
        u, u_prev, ut, g, cdt2, dt, kUbSigma, out, nullptr,
        UbGrids{grid, grid_prev, (int64_t)p->grid.nx * p->grid.ny, b->iface_lin});
  return cuda_check(cudaGetLastError(), "fc2d_wave_ub_step");
}

extern "C" fc2d_status fc2d_forward_wave(fc2d_plan_t p, int n_f, double c, int n_c, int n_large,
                                         int interface_mode, double* u, double* ut,
                                         const double* g_dir, const double* gt_dir,
                                         void* stream) {
  fc2d_status st = wave_checks(p, n_c, "fc2d_forward_wave");
  if (st) return st;
  if ((st = check_nf(p, n_f))) return st;
  if (!u || !ut) return set_error(FC2D_ERR_ARG, "fc2d_forward_wave: null pointer");
  if (!(c > 0) || n_large < 0)
    return set_error(FC2D_ERR_ARG, "fc2d_forward_wave: c > 0 and n_large >= 0 required");
  if (interface_mode < 0 || interface_mode > 2)
    return set_error(FC2D_ERR_ARG, "fc2d_forward_wave: interface_mode 0, 1 or 2");
  if (p->grid.ny > kWaveMaxRows)
    return set_error(FC2D_ERR_UNSUPPORTED, "fc2d_forward_wave: ny <= 4842");
  if (n_large == 0) return FC2D_OK;
  cudaSetDevice(p->device);
  cudaStream_t s = (cudaStream_t)stream;
  DevBand* b;
  // mode 2 (once the squares in double-float arithmetic) runs the fixed-point squares of
  // mode 1, which are both faster and more accurate
  if ((st = get_band(p, n_c, interface_mode ? 1 : 0, &b))) return st;
  const int nx = p->grid.nx, ny = p->grid.ny, nxh = nx / 2 + 1;
  const int64_t NN = (int64_t)nx * ny, nb = p->n_bdry, Nu = b->host.unknown_lin.size();
  const int64_t Ni = (int64_t)b->host.iface_lin.size();
  const size_t pitch = row_pitch(p);
  const int S = 8 * n_c;
  const double h = p->grid.h, dT = n_c * h / c, dt = dT / S, cdt2 = (c * dt) * (c * dt);
  const DevSquares* sq = b->sq.get();
  // scratch: spectra [2 n_f][ny][nxh], row-pass layout [2 n_f][ny][pitch], four U_B arrays (u and w, twice), zero boundary data
  auto al = [](size_t x) { return (x + 255) / 256 * 256; };
  const size_t b_spec = al((size_t)2 * n_f * ny * nxh * 16), b_inter = al((size_t)2 * n_f * ny * pitch * 16),
               b_ub = al((size_t)std::max<int64_t>(1, Nu + Ni) * n_f * 8),
               b_zero = al((size_t)n_f * nb * 8);
  const int n_sq = sq ? sq->n : 0;
  const size_t b_sqz = al(squares_spectrum_bytes(n_sq, n_f)), b_sqt = sq ? al(squares_factor_bytes(S)) : 0;
  const size_t b_sqe = al((size_t)n_sq * n_f * sizeof(int));
  const size_t b_ut = al((size_t)std::max<int64_t>(1, Nu) * n_f * 8);
  const size_t b_exps = al(wave_fx_exps(nx, ny, n_f) * sizeof(int));
  const size_t need = b_spec + b_inter + 4 * b_ub + b_zero + b_sqz + b_sqt + b_sqe + b_ut + b_exps;
  WaveState* W = state(p);
  if (W->scr.bytes < need) {
    cudaDeviceSynchronize();
    cudaFree(W->scr.base);
    W->scr = Scratch();
    if (cudaMalloc(&W->scr.base, need) != cudaSuccess)
      return set_error(FC2D_ERR_NOMEM, "fc2d_forward_wave: scratch cudaMalloc failed");
    W->scr.bytes = need;
  }
  char* base = static_cast<char*>(W->scr.base);
  double2* spec = reinterpret_cast<double2*>(base);
  double2* inter = reinterpret_cast<double2*>(base + b_spec);
  double* ub[4];
  for (int k = 0; k < 4; ++k)
    ub[k] = reinterpret_cast<double*>(base + b_spec + b_inter + k * b_ub);
  double* zero = reinterpret_cast<double*>(base + b_spec + b_inter + 4 * b_ub);
  char* sqZ = base + b_spec + b_inter + 4 * b_ub + b_zero;
  char* sqT = sqZ + b_sqz;
  int* sqE = reinterpret_cast<int*>(sqT + b_sqt);
  int* exps = reinterpret_cast<int*>(base + need - b_exps);
  cudaMemsetAsync(zero, 0, (size_t)n_f * nb * 8, s);
  // the spectra of u_t are scaled by 2^eT >= dT in the fixed-point solutions
  const int eT = wave_fx_time(dT, h, c);
  if (sq) squares_factors(S, c, h, dt, eT, sqT, s);
  auto gat = [&](int64_t m) { return g_dir ? g_dir + (size_t)m * n_f * nb : nullptr; };
  auto gtat = [&](int64_t j) { return gt_dir ? gt_dir + (size_t)j * n_f * nb : nullptr; };
  FftArgs fa = fft_args(p);
  if ((st = wave_fx_prepare(p))) return st;
  // U_FC at tau = cells h / c: u, or (deriv) its time derivative, on the grid or at the
  // interface points
  auto eval_ufc = [&](double tau, double cells, bool deriv, double* out, bool points) {
    return wave_fx_eval(p, fa, n_f, deriv, c, tau, cells, 0.0, eT, spec, exps, inter, out,
                        points ? b->iface_off : nullptr, points ? b->iface_lin : nullptr, s);
  };
  // U_B: u and w in (U[a], V[a]), the next ones into the other pair
  double* utB = reinterpret_cast<double*>(base + need - b_exps - b_ut);
  double *U[2] = {ub[0], ub[1]}, *V[2] = {ub[2], ub[3]};
  int a = 0;
  auto gather = [&](int64_t n, const int32_t* lin, const double* grid, double* out) {
    if (n > 0) k_ub_gather<<<blocks(n * n_f, 256), 256, 0, s>>>(n, n_f, NN, lin, grid, out);
  };
  auto ub_step = [&](int mode, const double* g, double* uo, double* wo) {
    if (Nu == 0) return;
    ProfScope ps(p, "ub_step", s);
    k_ub_advance<<<blocks(Nu * n_f, 256), 256, 0, s>>>(
        mode, (int)Nu, (int)Ni, n_f, nb, b->L.row, b->L.e, b->D.row, b->D.e, U[a], U[1 - a], V[a],
        g, cdt2, dt, kUbSigma, uo, wo, UbRows{});
  };
  // U_B at t = 0: u^0, and u_t^0 in the place of w
  gather(Nu, b->unknown_lin, u, U[a]);
  gather(Nu, b->unknown_lin, ut, V[a]);
  for (int j = 0; j < n_large; ++j) {
    const int64_t m0 = (int64_t)j * S;
    if (sq) {  // the squares' expansions of u(T_j), u_t(T_j), before u and ut change
      ProfScope ps(p, "sq_forward", s);
      const SquareSet& H = sq->host;
      squares_expand(sq->args(), 2 * H.a + 1, H.C, H.d, nx, NN, n_f, eT, u, ut, sqZ, sqE, s);
    }
    if ((st = wave_spectra(p, n_f, u, g_dir ? gat(m0) : zero, ut, gt_dir ? gtat(j) : zero, spec, s)))
      return st;
    wave_fx_spectra(fa, n_f, eT, spec, exps, s);
    for (int sidx = 0; sidx < S; ++sidx) {
      const int64_t m = m0 + sidx;
      double* face = U[a] + Nu * n_f;  // U_FC at the interface points
      if (sq) {
        ProfScope ps(p, "sq_eval", s);
        squares_solve(sq->args(), sq->max_rows, n_f, sqZ, sqE, sqT, sidx, face, s);
      } else {
        if ((st = eval_ufc(sidx * dt, sidx * kUbCfl, false, face, true))) return st;
      }
      ub_step(m == 0 ? 0 : 1, gat(m), U[1 - a], V[1 - a]);
      a = 1 - a;
    }
    // T_{j+1}: U_FC and its time derivative on the grid (into u, ut), then U_B's time
    // derivative from one further step and the merge of eq. (4.9)
    if ((st = eval_ufc(dT, n_c, false, u, false)) || (st = eval_ufc(dT, n_c, true, ut, false))) return st;
    const int64_t mN = m0 + S;
    gather(Ni, b->iface_lin, u, U[a] + Nu * n_f);
    ub_step(2, gat(mN), utB, nullptr);
    const int64_t n_near = (int64_t)b->host.near_lin.size();
    if (n_near > 0) {
      ProfScope ps(p, "ff_merge", s);
      k_ff_merge<<<blocks(n_near * n_f, 256), 256, 0, s>>>(
          n_near, n_f, NN, nb, b->near_lin, b->near_src, b->S.off, b->S.col, b->S.w, U[a],
          utB, g_dir ? gat(mN) : zero, gt_dir ? gtat(j + 1) : zero, u, ut);
    }
  }
  k_zero_outside<<<dim3(ny, n_f), 256, 0, s>>>(nx, ny, n_f, p->dev.row_iv_off, p->dev.row_iv, u, ut);
  return cuda_check(cudaGetLastError(), "fc2d_forward_wave");
}
