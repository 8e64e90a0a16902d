// The double-precision DFT of sizes 2^a 3^b 5^c in block fixed point (fx_mixed.cuh): rows
// whose half length is not a power of two, columns in two passes, their inverses for the
// Fourier Forwarding and Poisson solutions.
#include <cuda_runtime.h>

#include <algorithm>

#include "fc2d_kernels.cuh"
#include "fx_mixed.cuh"
#include "plan_internal.h"

namespace fc2d {
namespace fx {

// Rows: one block per (row, function), as k_rows_fx
__global__ void __launch_bounds__(256, 2)
k_rows_mixed(FftArgs fa, RowArgs ra, int mode, const double* __restrict__ ext,
             const double* __restrict__ f_grid, const double* __restrict__ vals,
             double2* __restrict__ inter) {
  extern __shared__ __align__(16) unsigned char smem_raw[];
  __shared__ unsigned st[kMixedSlots];
  const int nx = fa.nx, NH = nx / 2, j = blockIdx.x, f = blockIdx.y, t = threadIdx.x, nt = blockDim.x;
  double2* row = reinterpret_cast<double2*>(smem_raw);
  c64* buf = reinterpret_cast<c64*>(smem_raw);
  if (t < kMixedSlots) st[t] = 0;
  pdl_wait();
  pdl_trigger();
  if (mode == 0) {
    const double* src = ext + (size_t)f * ra.grid_stride + (size_t)j * nx;
    for (int i = t; i < nx; i += nt) reinterpret_cast<double*>(row)[i] = src[i];
  } else {
    load_row<double>(ra, j, f, f_grid + (size_t)f * ra.grid_stride, mode == 2, vals,
                     reinterpret_cast<double*>(row));
  }
  __syncthreads();
  unsigned mag = 0;
  for (int i = t; i < NH; i += nt) mag = max(mag, max(magnitude(row[i].x), magnitude(row[i].y)));
  block_max(mag, st);
  __syncthreads();
  const int E = block_exp(st[0]);
  int e = E - 1080;
  // the doubles lie in buffer 1, which the second stage overwrites
  c64* b0 = buf + NH;
  mixed_dft<FORWARD>(fa.mix.row, NH, t, nt, [&](int i) { return from_double(row[i], E); },
            [&](int b, int i) { return b ? buf[i] : b0[i]; },
            [&](int b, int i, c64 v) { (b ? buf : b0)[i] = v; }, fa.fxwx, 1, st, e);
  const c64* z = (fa.mix.row.n - 1) & 1 ? buf : b0;
  const int L = max(headroom(st[fa.mix.row.n]) - 1, 0);  // |z| <= 2^61
  e += kDrop - 1 - L;
  if (E >= 0x7FF) e = kNaN;
  const bool plain = plain_exp(e);
  double2* out = inter + ((size_t)f * fa.ny + j) * fa.pitch;
  for (int k = t; k <= NH / 2; k += nt) {
    const c64 zk = z[k], zl = z[k ? NH - k : 0];
    c64 xk, xl;
    split_pair(c64{zk.x << L, zk.y << L}, c64{zl.x << L, zl.y << L}, __ldg(fa.fxr + k), xk, xl);
    out[k] = to_double(xk, e, plain);
    if (k != NH - k) out[NH - k] = to_double(xl, e, plain);
  }
}

// Inverse rows, as k_inverse_rows_fx (fx_wave.cu)
__global__ void __launch_bounds__(256, 2)
k_inverse_rows_mixed(FftArgs fa, const double2* __restrict__ inter, const double* __restrict__ c00,
                     double a0, double b0, double h, double* __restrict__ out,
                     const int32_t* __restrict__ point_off, const int32_t* __restrict__ points, int ld) {
  extern __shared__ __align__(16) unsigned char smem_raw[];
  __shared__ unsigned st[kMixedSlots];
  const int NH = fa.nx / 2, j = blockIdx.x, f = blockIdx.y, t = threadIdx.x, nt = blockDim.x;
  c64 *b1 = reinterpret_cast<c64*>(smem_raw), *bz = b1 + NH;
  int p0 = 0, p1 = 0;
  if (point_off) {
    p0 = point_off[j];
    p1 = point_off[j + 1];
    if (p0 == p1) return;
  }
  if (t < kMixedSlots) st[t] = 0;
  __syncthreads();
  pdl_wait();
  pdl_trigger();
  const double2* row = inter + ((size_t)f * fa.ny + j) * fa.pitch;
  unsigned mag = 0;
  for (int k = t; k <= NH; k += nt) mag = max(mag, max(magnitude(row[k].x), magnitude(row[k].y)));
  block_max(mag, st);
  __syncthreads();
  const int E = block_exp(st[0]);
  int e = E - 1082 + kDrop;
  for (int k = t; k <= NH / 2; k += nt) {
    const c64 x = from_double<7>(row[k], E), y = from_double<7>(row[NH - k], E);
    const c64 s = drop(c64{x.x + y.x, x.y - y.y});
    const c64 q = mulw_conj(c64{x.x - y.x, x.y + y.y}, __ldg(fa.fxr + k));
    b1[k] = {s.x - q.y, -s.y - q.x};
    if (k && k != NH - k) b1[NH - k] = {s.x + q.y, s.y - q.x};
  }
  __syncthreads();
  mixed_dft<INVERSE>(fa.mix.row, NH, t, nt, [&](int i) { return b1[i]; },
            [&](int b, int i) { return b ? b1[i] : bz[i]; },
            [&](int b, int i, c64 v) { (b ? b1 : bz)[i] = v; }, fa.fxwx, 1, st, e);
  const c64* z = (fa.mix.row.n - 1) & 1 ? b1 : bz;
  if (E >= 0x7FF) e = kNaN;
  const bool plain = plain_exp(e);
  if (point_off) {
    for (int p = p0 + t; p < p1; p += nt) {
      const int x = points[p] - j * (2 * NH);
      const c64 v = z[x >> 1];
      out[(size_t)p * ld + f] = (x & 1) ? to_double(-v.y, e, plain) : to_double(v.x, e, plain);
    }
    return;
  }
  const double q = c00 ? c00[f] * 0.25 : 0.0, y = b0 + h * double(j);
  double* dst = out + ((size_t)f * fa.ny + j) * (2 * NH);
  for (int m = t; m < NH; m += nt) {
    const double2 v = to_double(z[m], e, plain);
    double2 o = {v.x, -v.y};
    if (c00) {
      const double x0 = a0 + h * double(2 * m), x1 = a0 + h * double(2 * m + 1);
      o.x += q * (x0 * x0 + y * y);
      o.y += q * (x1 * x1 + y * y);
    }
    dst[2 * m] = o.x;
    dst[2 * m + 1] = o.y;
  }
}

// Columns, N = n1 n2: a block of kCols columns, ct threads per column.  Pass A for the rows
// n2 j1 + j2 of one j2: in(row, kx) are the inputs' doubles, or (ADV) integers |z| <= 2^58.5 in
// units of 2^e.  Leaves its integers at rows n2 m1 + j2 of mid.
template <bool ADV, typename In>
__device__ __forceinline__ void mixed_pass_a(const FxMixed& mx, unsigned char* smem, unsigned* st, In in,
                                             c64* __restrict__ mid, unsigned pitch, int j2, int kx,
                                             bool live, const int4* __restrict__ w, int e, int* exp_out) {
  const int c = threadIdx.x & (kCols - 1), t = threadIdx.x / kCols, ct = blockDim.x / kCols;
  const int n1 = mx.n1, n2 = mx.n2;
  double2* raw = reinterpret_cast<double2*>(smem) + c;
  c64 *b1 = reinterpret_cast<c64*>(smem) + c, *b0 = b1 + n1 * kCols;
  int E = 1;
  if constexpr (!ADV) {
    unsigned mag = 0;
    for (int i = t; i < n1; i += ct) {
      const double2 u = live ? in(n2 * i + j2, kx) : double2{0.0, 0.0};
      raw[i * kCols] = u;
      mag = max(mag, max(magnitude(u.x), magnitude(u.y)));
    }
    block_max(mag, st);
    __syncthreads();
    E = block_exp(st[0]);
    e = E - 1080;
  }
  auto first = [&](int i) {
    if constexpr (ADV) return live ? in(n2 * i + j2, kx) : c64{0, 0};
    else return from_double(raw[i * kCols], E);
  };
  mixed_dft<ADV ? INVERSE : FORWARD>(mx.a, n1, t, ct, first, [&](int b, int i) { return (b ? b1 : b0)[i * kCols]; },
            [&](int b, int i, c64 v) { (b ? b1 : b0)[i * kCols] = v; }, w, n2, st, e);
  const c64* z = (mx.a.n - 1) & 1 ? b1 : b0;
  if (live)
    for (int i = t; i < n1; i += ct) mid[(unsigned)(n2 * i + j2) * pitch + kx] = z[i * kCols];
  if (threadIdx.x == 0) *exp_out = E >= 0x7FF ? kNaN : e;
}

// Pass B for one m1: out(row, v, e, plain) for the rows m1 + n1 m2 of the transform
template <Order O, typename Out>
__device__ __forceinline__ void mixed_pass_b(const FxMixed& mx, unsigned char* smem, unsigned* st,
                                             const c64* __restrict__ mid, unsigned pitch, int m1, int kx,
                                             bool live, const int4* __restrict__ w,
                                             const int* __restrict__ exps, int estride, int eadd, Out out) {
  const int c = threadIdx.x & (kCols - 1), t = threadIdx.x / kCols, ct = blockDim.x / kCols;
  const int n1 = mx.n1, n2 = mx.n2;
  c64 *b1 = reinterpret_cast<c64*>(smem) + c, *b0 = b1 + n2 * kCols;
  int top = -2048;
  for (int i = t; i < n2; i += ct) {
    const c64 v = live ? mid[(unsigned)(n2 * m1 + i) * pitch + kx] : c64{0, 0};
    b1[i * kCols] = v;
    top = max(top, exps[i * estride] + 63 - __clz((int)(spread(v) | 1u)));
  }
  block_max((unsigned)(top + 4096), st);
  __syncthreads();
  const int e0 = (int)st[0] - 4096 - 62;
  int e = e0 + kDrop;
  auto first = [&](int i) {
    const int s = exps[i * estride] - e0, up = max(s, 0), dn = min(max(-s, 0), 63);
    const i64 rnd = (i64)((1ull << dn) >> 1);
    const c64 v = b1[i * kCols];
    return mulw(c64{((v.x << up) + rnd) >> dn, ((v.y << up) + rnd) >> dn}, __ldg(w + i * m1));
  };
  mixed_dft<O>(mx.b, n2, t, ct, first, [&](int b, int i) { return (b ? b1 : b0)[i * kCols]; },
            [&](int b, int i, c64 v) { (b ? b1 : b0)[i * kCols] = v; }, w, n1, st, e);
  const c64* z = (mx.b.n - 1) & 1 ? b1 : b0;
  e += eadd;
  const bool plain = plain_exp(e);
  if (live)
    for (int i = t; i < n2; i += ct) out(m1 + n1 * i, z[i * kCols], e, plain);
}

__global__ void __launch_bounds__(160, 4)
k_cols_mixed_a(FftArgs fa, double2* __restrict__ inter, int* __restrict__ exps) {
  extern __shared__ __align__(16) unsigned char smem_raw[];
  __shared__ unsigned st[kMixedSlots];
  if (threadIdx.x < kMixedSlots) st[threadIdx.x] = 0;
  const int kx = blockIdx.x * kCols + (threadIdx.x & (kCols - 1)), j2 = blockIdx.y, f = blockIdx.z;
  const unsigned pitch = fa.pitch;
  double2* slab = inter + (size_t)f * fa.ny * pitch;
  __syncthreads();
  pdl_wait();
  pdl_trigger();
  mixed_pass_a<false>(fa.mix, smem_raw, st, [&](int row, int k) { return slab[(unsigned)row * pitch + k]; },
                      reinterpret_cast<c64*>(slab), pitch, j2, kx, kx < fa.nx / 2 + 1, fa.fxwy, 0,
                      exps + ((size_t)f * fa.mix.n2 + j2) * gridDim.x + blockIdx.x);
}

__global__ void __launch_bounds__(160, 4)
k_cols_mixed_b(FftArgs fa, const double2* __restrict__ inter, const int* __restrict__ exps,
               double2* __restrict__ fhat) {
  extern __shared__ __align__(16) unsigned char smem_raw[];
  __shared__ unsigned st[kMixedSlots];
  if (threadIdx.x < kMixedSlots) st[threadIdx.x] = 0;
  const int ncol = fa.nx / 2 + 1, kx = blockIdx.x * kCols + (threadIdx.x & (kCols - 1)), f = blockIdx.z;
  const c64* slab = reinterpret_cast<const c64*>(inter) + (size_t)f * fa.ny * fa.pitch;
  double2* dst = fhat + (size_t)f * fa.ny * fa.opitch + kx;
  __syncthreads();
  pdl_wait();
  pdl_trigger();
  mixed_pass_b<FORWARD>(fa.mix, smem_raw, st, slab, fa.pitch, blockIdx.y, kx, kx < ncol, fa.fxwy,
               exps + (size_t)f * fa.mix.n2 * gridDim.x + blockIdx.x, gridDim.x, fa.fxs.exp,
               [&](int row, c64 v, int e, bool plain) {
                 dst[(unsigned)row * (unsigned)fa.opitch] = to_double(scaled(v, fa.fxs), e, plain);
               });
}

// Modal advance and inverse columns (fx_wave.cu: k_adv_a, k_adv_b), spectra in place to
// integers (k_spec_fix)
__global__ void __launch_bounds__(160)
k_spec_fix_mixed(FxMixed mx, int ny, int nxh, int n_f, int eT, double2* __restrict__ spec,
                 int* __restrict__ exps) {
  __shared__ unsigned st[2];
  if (threadIdx.x < 2) st[threadIdx.x] = 0;
  const int kx = blockIdx.x * kCols + (threadIdx.x & (kCols - 1)), t = threadIdx.x / kCols;
  const int ct = blockDim.x / kCols, j2 = blockIdx.y, f = blockIdx.z;
  const bool live = kx < nxh;
  double2* F = spec + (size_t)f * ny * nxh + kx;
  double2* G = spec + (size_t)(n_f + f) * ny * nxh + kx;
  __syncthreads();
  pdl_wait();
  pdl_trigger();
  unsigned mu = 0, mv = 0;
  if (live)
    for (int i = t; i < mx.n1; i += ct) {
      const unsigned o = (unsigned)(mx.n2 * i + j2) * (unsigned)nxh;
      mu = max(mu, max(magnitude(F[o].x), magnitude(F[o].y)));
      mv = max(mv, max(magnitude(G[o].x), magnitude(G[o].y)));
    }
  block_max(mu, st);
  block_max(mv, st + 1);
  __syncthreads();
  const int EF = block_exp(st[0]), EG = block_exp(st[1]), E = max(EF, EG + eT);
  if (live)
    for (int i = t; i < mx.n1; i += ct) {
      const unsigned o = (unsigned)(mx.n2 * i + j2) * (unsigned)nxh;
      reinterpret_cast<c64*>(F)[o] = from_double<8>(F[o], E);
      reinterpret_cast<c64*>(G)[o] = from_double<8>(G[o], E - eT);
    }
  if (threadIdx.x == 0)
    exps[((size_t)f * mx.n2 + j2) * gridDim.x + blockIdx.x] = max(EF, EG) >= 0x7FF ? kNaN : E - 1083;
}

template <bool DERIV>
__global__ void __launch_bounds__(160, 4)
k_adv_mixed_a(FxMixed mx, int ny, int nxh, unsigned pitch, int n_f, int f0, int eS,
              const int4* __restrict__ fac, const c64* __restrict__ spec, const int* __restrict__ exps,
              const int4* __restrict__ tw, c64* __restrict__ mid, int* __restrict__ mexps) {
  extern __shared__ __align__(16) unsigned char smem_raw[];
  __shared__ unsigned st[kMixedSlots], sp[1];
  if (threadIdx.x < kMixedSlots) st[threadIdx.x] = 0;
  if (threadIdx.x == 0) sp[0] = 0;
  const int kx = blockIdx.x * kCols + (threadIdx.x & (kCols - 1)), j2 = blockIdx.y, f = blockIdx.z;
  const bool live = kx < nxh;
  __syncthreads();
  pdl_wait();
  pdl_trigger();
  const c64* F = spec + (size_t)(f0 + f) * ny * nxh + kx;
  const c64* G = spec + (size_t)(n_f + f0 + f) * ny * nxh + kx;
  auto factor = [&](int row) { return __ldg(fac + (unsigned)(row <= ny / 2 ? row : ny - row) * (unsigned)nxh + kx); };
  int up = 0;
  if constexpr (DERIV) {  // the bits that the block's largest value leaves unused
    unsigned h = 0;
    if (live)
      for (int i = threadIdx.x / kCols; i < mx.n1; i += blockDim.x / kCols) {
        const int row = mx.n2 * i + j2;
        const unsigned o = (unsigned)row * (unsigned)nxh;
        const int4 t = factor(row);
        h |= spread(dot(F[o].x, G[o].x, t)) | spread(dot(F[o].y, G[o].y, t));
      }
    block_or(h, sp);
    __syncthreads();
    up = min(max(headroom(sp[0]) - 4, 0), 28);
  }
  auto in = [&](int row, int) {
    const unsigned o = (unsigned)row * (unsigned)nxh;
    const c64 a = F[o], b = G[o];
    const int4 t = factor(row);
    if constexpr (DERIV) {
      const Wide x = dot_wide(a.x, b.x, t), y = dot_wide(a.y, b.y, t);
      return c64{(x.hi << up) + (x.mid >> (32 - up)), -(y.hi << up) - (y.mid >> (32 - up))};
    } else {
      return c64{dot(a.x, b.x, t), -dot(a.y, b.y, t)};
    }
  };
  const int e = exps[((size_t)(f0 + f) * mx.n2 + j2) * gridDim.x + blockIdx.x] + kDrop + eS - up;
  mixed_pass_a<true>(mx, smem_raw, st, in, mid + (size_t)f * ny * pitch, pitch, j2, kx, live, tw, e,
                     mexps + ((size_t)f * mx.n2 + j2) * gridDim.x + blockIdx.x);
}

__global__ void __launch_bounds__(160, 4)
k_adv_mixed_b(FxMixed mx, int ny, int nxh, unsigned pitch, const c64* __restrict__ mid,
              const int* __restrict__ mexps, const int4* __restrict__ tw, double2* __restrict__ out) {
  extern __shared__ __align__(16) unsigned char smem_raw[];
  __shared__ unsigned st[kMixedSlots];
  if (threadIdx.x < kMixedSlots) st[threadIdx.x] = 0;
  const int kx = blockIdx.x * kCols + (threadIdx.x & (kCols - 1)), f = blockIdx.z;
  double2* dst = out + (size_t)f * ny * pitch + kx;
  __syncthreads();
  pdl_wait();
  pdl_trigger();
  mixed_pass_b<INVERSE>(mx, smem_raw, st, mid + (size_t)f * ny * pitch, pitch, blockIdx.y, kx, kx < nxh, tw,
               mexps + (size_t)f * mx.n2 * gridDim.x + blockIdx.x, gridDim.x, 0,
               [&](int row, c64 v, int e, bool plain) {
                 const double2 z = to_double(v, e, plain);
                 dst[(unsigned)row * pitch] = double2{z.x, -z.y};
               });
}

template <typename K> static size_t allow(K k, size_t sm) {
  cudaFuncSetAttribute(k, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)sm);
  return sm;
}
static int row_threads_for(int NH) { return NH <= 1024 ? 128 : 256; }
static size_t col_smem(int n) { return (size_t)2 * n * kCols * sizeof(c64); }

}  // namespace fx

void launch_fft_rows_mixed(const FftArgs& fa, const RowArgs& ra, int n_f, int mode, const void* ext,
                           const double* f_grid, const void* vals, void* inter, cudaStream_t s) {
  const size_t sm = fx::allow(fx::k_rows_mixed, (size_t)fa.nx * 16);
  launch_pdl(fx::k_rows_mixed, dim3(fa.ny, n_f), dim3(fx::row_threads_for(fa.nx / 2)), sm, s, fa, ra, mode,
             (const double*)ext, f_grid, (const double*)vals, (double2*)inter);
}

void launch_inverse_rows_mixed(const FftArgs& fa, int n_f, const void* inter, const double* c00,
                               double a0, double b0, double h, double* out, const int32_t* off,
                               const int32_t* points, int ld, cudaStream_t s) {
  const size_t sm = fx::allow(fx::k_inverse_rows_mixed, (size_t)fa.nx * 16);
  launch_pdl(fx::k_inverse_rows_mixed, dim3(fa.ny, n_f), dim3(fx::row_threads_for(fa.nx / 2)), sm, s, fa,
             (const double2*)inter, c00, a0, b0, h, out, off, points, ld);
}

void launch_fft_cols_mixed(const FftArgs& fa, int n_f, void* inter, void* fhat, cudaStream_t s) {
  const int groups = fa.nx / 32 + 1;
  launch_pdl(fx::k_cols_mixed_a, dim3(groups, fa.mix.n2, n_f), dim3(16 * fa.mix.ta),
             fx::allow(fx::k_cols_mixed_a, fx::col_smem(fa.mix.n1)), s, fa, (double2*)inter, fa.exps);
  launch_pdl(fx::k_cols_mixed_b, dim3(groups, fa.mix.n1, n_f), dim3(16 * fa.mix.tb),
             fx::allow(fx::k_cols_mixed_b, fx::col_smem(fa.mix.n2)), s, fa, (const double2*)inter,
             (const int*)fa.exps, (double2*)fhat);
}

void launch_spec_fix_mixed(const FftArgs& fa, int n_f, int eT, void* spec, int* exps, cudaStream_t s) {
  launch_pdl(fx::k_spec_fix_mixed, dim3(fa.nx / 32 + 1, fa.mix.n2, n_f), dim3(16 * fa.mix.ta), 0, s, fa.mix,
             fa.ny, fa.nx / 2 + 1, n_f, eT, (double2*)spec, exps);
}

void launch_adv_mixed(const FftArgs& fa, int n_f, int f0, int nf, bool deriv, int eS, const int4* fac,
                      const void* spec, const int* exps, void* mid, int* mexps, void* res, cudaStream_t s) {
  const int groups = fa.nx / 32 + 1, nxh = fa.nx / 2 + 1;
  auto ka = deriv ? fx::k_adv_mixed_a<true> : fx::k_adv_mixed_a<false>;
  launch_pdl(ka, dim3(groups, fa.mix.n2, nf), dim3(16 * fa.mix.ta), fx::allow(ka, fx::col_smem(fa.mix.n1)), s,
             fa.mix, fa.ny, nxh, (unsigned)fa.pitch, n_f, f0, eS, fac, (const fx::c64*)spec, exps, fa.fxwy,
             (fx::c64*)mid, mexps);
  launch_pdl(fx::k_adv_mixed_b, dim3(groups, fa.mix.n1, nf), dim3(16 * fa.mix.tb),
             fx::allow(fx::k_adv_mixed_b, fx::col_smem(fa.mix.n2)), s, fa.mix, fa.ny, nxh, (unsigned)fa.pitch,
             (const fx::c64*)mid, (const int*)mexps, fa.fxwy, (double2*)res);
}

}  // namespace fc2d
