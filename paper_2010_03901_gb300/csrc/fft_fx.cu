// The double-precision DFT (eq. (3.1)) of power-of-two sizes in block fixed point (fx.cuh).
//
// k_rows_fx: one block per (row, function): the extended row (assembled from f and the
// strip values, or a row of an extended grid) as nx/2 complex pairs, the length-nx/2
// transform, the even/odd split to X_k, k = 0..nx/2, to the intermediate.
// k_cols_fx: one block per (CB columns, function): length-ny transforms, scaled by
// 1/(nx ny), to the half spectrum [ny][nx/2+1].
#include <cuda_runtime.h>

#include <algorithm>

#include "fc2d_kernels.cuh"
#include "fx.cuh"
#include "p2_rows.cuh"
#include "plan_internal.h"

namespace fc2d {
namespace fx {

template <int LOGNH> __host__ __device__ constexpr int row_threads() {
  return (1 << LOGNH) / 8 < 32 ? 32 : (1 << LOGNH) / 8;
}

// resident blocks asked of the compiler: 64 registers per thread, within shared memory
__host__ __device__ constexpr int blocks_for(int threads, int bytes) {
  const int r = 1024 / threads, m = 220 * 1024 / (bytes + 1024);
  return r < m ? (r < 1 ? 1 : r) : (m < 1 ? 1 : m);
}

template <int LOGNH>
__global__ void __launch_bounds__(row_threads<LOGNH>(), blocks_for(row_threads<LOGNH>(), 16 * padded(1 << LOGNH)))
k_rows_fx(FftArgs fa, RowArgs ra, int mode, const double* __restrict__ ext,
          const double* __restrict__ f_grid, const double* __restrict__ vals,
          double2* __restrict__ inter) {
  constexpr int NH = 1 << LOGNH, NT = NH / 8;
  extern __shared__ __align__(16) unsigned char smem_raw[];
  __shared__ unsigned st[kSlots];
  double2* row = reinterpret_cast<double2*>(smem_raw);
  c64* buf = reinterpret_cast<c64*>(smem_raw);
  const int j = blockIdx.x, f = blockIdx.y, t = threadIdx.x;
  const bool active = t < NT;
  if (t < kSlots) st[t] = 0;
  p2::assemble_row<double, double, row_threads<LOGNH>()>(ra, mode, NH, j, f, ext, f_grid, vals, row);
  double2 u[8];
  c64 v[8];
  if (active) {
#pragma unroll
    for (int r = 0; r < 8; ++r) u[r] = row[pad(t + r * NT)];
  }
  int e;
  transform<LOGNH>(u, v, buf, t, active, st, fa.fxx, e);
  __syncthreads();
  unsigned h = 0;
  if (active) {
    constexpr int R = last_radix<LOGNH>();
#pragma unroll
    for (int m = 0; m < 8 / R; ++m)
#pragma unroll
      for (int r = 0; r < R; ++r) {
        buf[pad(out_index<LOGNH>(t, m, r))] = v[m * R + r];
        h |= spread(v[m * R + r]);
      }
  }
  block_or(h, st + kSlots - 1);
  __syncthreads();
  const int L = max(headroom(st[kSlots - 1]) - 1, 0);  // |z| <= 2^61
  e += kDrop - 1 - L;
  const bool plain = plain_exp(e);
  double2* out = inter + ((size_t)f * fa.ny + j) * fa.pitch;
  for (int k = t; k <= NH / 2; k += row_threads<LOGNH>()) {
    c64 xk, xl;
    const c64 zk = buf[pad(k)], zl = buf[pad(k ? NH - k : 0)];
    split_pair(c64{zk.x << L, zk.y << L}, c64{zl.x << L, zl.y << L}, __ldg(fa.fxr + k), xk, xl);
    out[k] = to_double(xk, e, plain);
    if (k != NH - k) out[NH - k] = to_double(xl, e, plain);
  }
}

template <int LOGNY, int CB>
__global__ void __launch_bounds__(CB * (1 << LOGNY) / 8, blocks_for(CB * (1 << LOGNY) / 8, 16 * CB * padded(1 << LOGNY)))
k_cols_fx(FftArgs fa, const double2* __restrict__ inter, double2* __restrict__ fhat) {
  constexpr int N = 1 << LOGNY, NT = N / 8, R = last_radix<LOGNY>();
  extern __shared__ __align__(16) unsigned char smem_raw[];
  __shared__ unsigned st[kSlots];
  const int ncol = fa.nx / 2 + 1;
  const int c = threadIdx.x % CB, t = threadIdx.x / CB;
  const int kx = blockIdx.x * CB + c, f = blockIdx.y;
  if (threadIdx.x < kSlots) st[threadIdx.x] = 0;
  // column c of the block's CB, offset so that the columns served by one shared-memory
  // wavefront (8 lanes) fall in disjoint banks
  c64* col = reinterpret_cast<c64*>(smem_raw) + c * padded(N) + c * (8 / CB);
  const double2* src = inter + (size_t)f * N * fa.pitch + kx;
  __syncthreads();
  pdl_wait();
  pdl_trigger();
  double2 u[8];
  c64 v[8];
  // kx < pitch always (the pitch is a multiple of 16 and CB divides 16); the pad columns
  // may hold anything and are left out of the block exponent
  const bool live = kx < ncol;
#pragma unroll
  for (int r = 0; r < 8; ++r)
    u[r] = live ? __ldg(src + (size_t)(t + r * NT) * fa.pitch) : double2{0.0, 0.0};
  int e;
  transform<LOGNY>(u, v, col, t, true, st, fa.fxy, e);
  e += fa.fxs.exp;
  const bool plain = plain_exp(e);
  double2* dst = fhat + (size_t)f * N * fa.opitch + kx;
  if (live) {
#pragma unroll
    for (int m = 0; m < 8 / R; ++m)
#pragma unroll
      for (int r = 0; r < R; ++r)
        dst[(size_t)out_index<LOGNY>(t, m, r) * fa.opitch] = to_double(scaled(v[m * R + r], fa.fxs), e, plain);
  }
}

// The two passes of columns of 64 N2 points from the row pass's intermediate (whose rows
// pass A overwrites with its integers) to the spectrum.
template <int N2>
__global__ void __launch_bounds__(kColThreads, 8)
k_cols2_a(FftArgs fa, double2* __restrict__ inter, int* __restrict__ exps) {
  __shared__ c64 ex[64 * kCols];
  __shared__ unsigned st[1];
  if (threadIdx.x == 0) st[0] = 0;
  const int ncol = fa.nx / 2 + 1, kx = blockIdx.x * kCols + (threadIdx.x & (kCols - 1));
  const int j2 = blockIdx.y, f = blockIdx.z;
  double2* slab = inter + (size_t)f * (64 * N2) * fa.pitch;
  const unsigned pitch = fa.pitch;
  __syncthreads();
  pdl_wait();
  pdl_trigger();
  cols_pass_a<N2>([&](int row, int k) { return slab[(unsigned)row * pitch + k]; },
                  reinterpret_cast<c64*>(slab), pitch, j2, kx, kx < ncol, ex, st, fa.fxwy,
                  exps + ((size_t)f * N2 + j2) * gridDim.x + blockIdx.x);
}

template <int N2>
__global__ void __launch_bounds__(kColThreads, 8)
k_cols2_b(FftArgs fa, const double2* __restrict__ inter, const int* __restrict__ exps,
          double2* __restrict__ fhat) {
  constexpr int R2 = N2 / 8, G = 8 / R2;  // G values of m1 per block
  __shared__ c64 ex[64 * kCols];
  __shared__ unsigned st[1];
  if (threadIdx.x == 0) st[0] = 0;
  const int ncol = fa.nx / 2 + 1, c = threadIdx.x & (kCols - 1), kx = blockIdx.x * kCols + c;
  const int l = (threadIdx.x / kCols) % R2, g = threadIdx.x / (kCols * R2), f = blockIdx.z;
  const int m1 = blockIdx.y * G + g;
  const c64* slab = reinterpret_cast<const c64*>(inter) + (size_t)f * (64 * N2) * fa.pitch;
  const bool live = kx < ncol;
  __syncthreads();
  pdl_wait();
  pdl_trigger();
  c64 v[8];
  int e = cols_pass_b<N2>(v, slab, fa.pitch, m1, l, kx, live, ex + g * 8 * R2 * kCols, st, fa.fxwy,
                          exps + (size_t)f * N2 * gridDim.x + blockIdx.x, gridDim.x);
  e += fa.fxs.exp;
  const bool plain = plain_exp(e);
  if (live) {
    const unsigned opitch = fa.opitch;
    double2* dst = fhat + (size_t)f * (64 * N2) * opitch + kx;
#pragma unroll
    for (int mm = 0; mm < 8 / R2; ++mm)
#pragma unroll
      for (int q = 0; q < R2; ++q)
        dst[(unsigned)(m1 + 64 * (l * (8 / R2) + mm + 8 * q)) * opitch] =
            to_double(scaled(v[mm * R2 + q], fa.fxs), e, plain);
  }
}

template <int N2>
static void cols2_launch(const FftArgs& fa, int n_f, void* inter, void* fhat, cudaStream_t s) {
  const int groups = (fa.nx / 2 + kCols) / kCols;
  launch_pdl(k_cols2_a<N2>, dim3(groups, N2, n_f), dim3(kColThreads), 0, s, fa, (double2*)inter, fa.exps);
  launch_pdl(k_cols2_b<N2>, dim3(groups, N2, n_f), dim3(kColThreads), 0, s, fa, (const double2*)inter,
             (const int*)fa.exps, (double2*)fhat);
}

template <int L>
static void rows_launch(const FftArgs& fa, const RowArgs& ra, int n_f, int mode, const void* ext,
                        const double* fg, const void* vals, void* inter, cudaStream_t s) {
  const size_t sm = (size_t)padded(1 << L) * sizeof(c64);
  cudaFuncSetAttribute(k_rows_fx<L>, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)sm);
  launch_pdl(k_rows_fx<L>, dim3(fa.ny, n_f), dim3(row_threads<L>()), sm, s, fa, ra, mode,
             (const double*)ext, fg, (const double*)vals, (double2*)inter);
}

template <int L, int CB>
static void cols_launch(const FftArgs& fa, int n_f, const void* inter, void* fhat, cudaStream_t s) {
  const size_t sm = ((size_t)CB * padded(1 << L) + 8) * sizeof(c64);
  cudaFuncSetAttribute(k_cols_fx<L, CB>, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)sm);
  const int ncol = fa.nx / 2 + 1;
  launch_pdl(k_cols_fx<L, CB>, dim3((ncol + CB - 1) / CB, n_f), dim3(CB * (1 << L) / 8), sm, s, fa,
             (const double2*)inter, (double2*)fhat);
}

static int ilog2_exact(int n) {
  if (n <= 0 || (n & (n - 1))) return -1;
  int l = 0;
  while ((1 << l) < n) ++l;
  return l;
}

}  // namespace fx

// The double-precision power-of-two DFT passes.  Return false (nothing launched) for other
// sizes.
bool launch_fft_rows_fx(const FftArgs& fa, const RowArgs& ra, int n_f, int mode, const void* ext,
                        const double* f_grid, const void* vals, void* inter, cudaStream_t s) {
#define FC2D_ROWS(L) \
  case L: fx::rows_launch<L>(fa, ra, n_f, mode, ext, f_grid, vals, inter, s); return true;
  switch (fx::ilog2_exact(fa.nx / 2)) {
    FC2D_ROWS(5) FC2D_ROWS(6) FC2D_ROWS(7) FC2D_ROWS(8)
    FC2D_ROWS(9) FC2D_ROWS(10) FC2D_ROWS(11) FC2D_ROWS(12)
    default: return false;
  }
#undef FC2D_ROWS
}

bool launch_fft_cols_fx(const FftArgs& fa, int n_f, void* inter, void* fhat, cudaStream_t s) {
  switch (fx::ilog2_exact(fa.ny)) {
    case 6: fx::cols_launch<6, 8>(fa, n_f, inter, fhat, s); return true;
    case 7: fx::cols_launch<7, 8>(fa, n_f, inter, fhat, s); return true;
    case 8: fx::cols_launch<8, 4>(fa, n_f, inter, fhat, s); return true;
    case 9: fx::cols_launch<9, 4>(fa, n_f, inter, fhat, s); return true;
    case 10: fx::cols_launch<10, 2>(fa, n_f, inter, fhat, s); return true;
    case 11: fx::cols2_launch<32>(fa, n_f, inter, fhat, s); return true;
    case 12: fx::cols2_launch<64>(fa, n_f, inter, fhat, s); return true;
    default: return false;
  }
}

}  // namespace fc2d
