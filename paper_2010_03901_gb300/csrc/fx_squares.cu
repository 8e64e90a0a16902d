// The small squares of Fourier Forwarding (Section 4.2; wave_band.cpp places them) in block
// fixed point (fx.cuh): each square's expansion once per large step, its modal solution at
// the served interface points every small step.
//
// The 64 x 64 transforms of a square run as 64-point DFTs by groups of 8 lanes, 8 values
// each, that exchange through shared memory within their warp.  In FP64 the evaluation was
// bound by the 2 FP64 operations per clock and SM (3.3 ms per small step for 576 squares and
// 32 functions; 0.69 ms in double-float on the FP32 pipe).
#include <cuda_runtime.h>

#include <algorithm>
#include <cstdint>

#include "fc2d_kernels.cuh"
#include "fx.cuh"
#include "fx_squares.h"

namespace fc2d {
namespace fx {

constexpr int kP = 64;          // the box
constexpr int kHalf = kP / 2 + 1;  // kept x frequencies l = 0 .. 32
constexpr int kThreads = 256;   // 32 groups of 8
constexpr int kRow = 73;        // stride of the expansion's rows (odd: no bank conflicts either way)

// 64-point DFT by the 8 lanes q of a group: in v[r] = x[q + 8 r] (|z| <= 2^59), out
// v[k] = X[q + 8 k], times 2^-kDrop; buf: the sequence's padded shared storage, element e at
// pad(e) ST.  Warp-wide barriers only.
template <int ST>
__device__ __forceinline__ void dft64_group(c64 (&v)[8], c64* buf, int q, const int4* __restrict__ tw) {
  dft<8>(v);
  v[0] = drop(v[0]);
#pragma unroll
  for (int k = 1; k < 8; ++k) v[k] = mulw(v[k], __ldg(tw + q * k));
#pragma unroll
  for (int k = 0; k < 8; ++k) buf[pad(q + 8 * k) * ST] = v[k];
  __syncwarp();
#pragma unroll
  for (int r = 0; r < 8; ++r) v[r] = buf[pad(8 * q + r) * ST];
  dft<8>(v);
  __syncwarp();
}

// shift left by n (n < 0: right, rounded)
__device__ __forceinline__ i64 shift(i64 v, int n) {
  return n >= 0 ? v << n : (v + ((1ll << -n) >> 1)) >> -n;
}

// Once per large step, block (square, function): the square's u and u_t 2^eT as one complex
// field, continued by 1D-FC (eq. (2.7)) along rows, then columns, to 64 x 64; its normalised
// 2D DFT, separated into the spectra F of u and G of u_t 2^eT: out[square][function][l][m] =
// (F, G), l <= 32, |values| <= 2^61 in units of 2^exps[square][function].
__global__ void __launch_bounds__(kThreads, 2)
k_sq_expand(int n_side, int C, int d, int nx, int64_t grid_stride, int n_f, int eT,
            const int32_t* __restrict__ origin, const double* __restrict__ A,
            const double* __restrict__ Q, const int4* __restrict__ tw, const double* __restrict__ u,
            const double* __restrict__ ut, c64* __restrict__ out, int* __restrict__ exps) {
  extern __shared__ __align__(16) unsigned char smem_raw[];
  double2* field = reinterpret_cast<double2*>(smem_raw);
  c64* buf = reinterpret_cast<c64*>(smem_raw);
  double2* gram = field + (kP + kP / 8 - 1) * kRow;  // [line][end][d]
  __shared__ unsigned st[4];
  const int sq = blockIdx.x, f = blockIdx.y, tid = threadIdx.x;
  const int j0 = __ldg(origin + 2 * sq), i0 = __ldg(origin + 2 * sq + 1);
  const double* uf = u + (size_t)f * grid_stride;
  const double* tf = ut + (size_t)f * grid_stride;
  const double up = __hiloint2double((1023 + eT) << 20, 0);  // 2^eT
  if (tid < 4) st[tid] = 0;
  for (int t = tid; t < n_side * n_side; t += kThreads) {
    const int y = t / n_side, x = t - y * n_side;
    const size_t g = (size_t)(j0 + y) * nx + (i0 + x);
    field[pad(y) * kRow + pad(x)] = double2{uf[g], tf[g] * up};
  }
  __syncthreads();
  // lines: rows y < n_side, then columns x < 64; the Gram coefficients Q^T f of both ends of
  // every line first (right: the last d values; left: the first d in reverse order)
#pragma unroll 1
  for (int dir = 0; dir < 2; ++dir) {
    const int lines = dir ? kP : n_side;
    auto at = [&](int line, int i) { return dir ? pad(i) * kRow + pad(line) : pad(line) * kRow + pad(i); };
    for (int t = tid; t < lines * 2 * d; t += kThreads) {
      const int line = t / (2 * d), e = (t / d) & 1, i = t % d;
      double2 s = {0.0, 0.0};
      for (int m = 0; m < d; ++m) {
        const double qm = __ldg(Q + m * d + i);
        const double2 v = field[at(line, e ? d - 1 - m : n_side - d + m)];
        s.x += qm * v.x;
        s.y += qm * v.y;
      }
      gram[(line * 2 + e) * d + i] = s;
    }
    __syncthreads();
    for (int t = tid; t < lines * C; t += kThreads) {
      const int line = t / C, k = t - line * C;
      const double2* g = gram + line * 2 * d;
      double2 vr = {0.0, 0.0}, vl = {0.0, 0.0};
      for (int i = 0; i < d; ++i) {
        const double ar = __ldg(A + k * d + i), al = __ldg(A + (C - 1 - k) * d + i);
        vr.x += ar * g[i].x;
        vr.y += ar * g[i].y;
        vl.x += al * g[d + i].x;
        vl.y += al * g[d + i].y;
      }
      field[at(line, n_side + k)] = double2{vl.x + vr.x, vl.y + vr.y};
    }
    __syncthreads();
  }
  const int g = tid >> 3, q = tid & 7;
  unsigned mag = 0;
#pragma unroll 1
  for (int y = g; y < kP; y += kThreads / 8)
#pragma unroll
    for (int r = 0; r < 8; ++r) {
      const double2 v = field[pad(y) * kRow + pad(q + 8 * r)];
      mag = max(mag, max(magnitude(v.x), magnitude(v.y)));
    }
  block_max(mag, st);
  __syncthreads();
  const int E = block_exp(st[0]);
  int e = E - 1080 + kDrop;
  unsigned h = 0;
  c64 v[8];
#pragma unroll 1
  for (int y = g; y < kP; y += kThreads / 8) {  // along x
    c64* row = buf + pad(y) * kRow;
#pragma unroll
    for (int r = 0; r < 8; ++r) v[r] = from_double(field[pad(y) * kRow + pad(q + 8 * r)], E);
    __syncwarp();
    dft64_group<1>(v, row, q, tw);
#pragma unroll
    for (int k = 0; k < 8; ++k) {
      row[pad(q + 8 * k)] = v[k];
      h |= spread(v[k]);
    }
  }
  block_or(h, st + 1);
  __syncthreads();
  int L = headroom(st[1]) - kDrop;  // to 2^58
  e += kDrop - L;
  h = 0;
#pragma unroll 1
  for (int l = g; l < kP; l += kThreads / 8) {  // along y
    c64* col = buf + pad(l);
#pragma unroll
    for (int r = 0; r < 8; ++r) {
      const c64 a = col[pad(q + 8 * r) * kRow];
      v[r] = {shift(a.x, L), shift(a.y, L)};
    }
    __syncwarp();
    dft64_group<kRow>(v, col, q, tw);
#pragma unroll
    for (int k = 0; k < 8; ++k) {
      col[pad(q + 8 * k) * kRow] = v[k];
      h |= spread(v[k]);
    }
  }
  block_or(h, st + 2);
  __syncthreads();
  // F = (Z_k + conj Z_-k)/2, G = (Z_k - conj Z_-k)/(2i), |Z| below 2^62 before the shift
  L = headroom(st[2]) - 2;
  c64* dst = out + ((size_t)sq * n_f + f) * (2 * kHalf * kP);
  for (int t = tid; t < kHalf * kP; t += kThreads) {
    const int l = t >> 6, m = t & 63;
    const c64 a = buf[pad(m) * kRow + pad(l)];
    const c64 b = buf[pad((kP - m) & 63) * kRow + pad((kP - l) & 63)];
    dst[2 * t] = {shift(a.x + b.x, L), shift(a.y - b.y, L)};
    dst[2 * t + 1] = {shift(a.y + b.y, L), shift(b.x - a.x, L)};
  }
  // 1/64^2 of the normalisation and the 1/2 above in the exponent
  if (tid == 0) exps[(size_t)sq * n_f + f] = E >= 0x7FF ? kNaN : e - L - 13;
}

// Every small step, block (square, function): the modal solution a = F t0 + G t1 at the time
// of `fac` ([l][m], limbs of (cos w t, 2^-eT sin(w t)/w)), its inverse 2D DFT (forward
// transforms of conj(a)), the values at the served points, function-minor.  Along m: 31
// complex sequences l = 1 .. 31 and the packed pair l = 0, 32, whose transforms are real
// (the field is).  Along l only the rows r0 .. r1 that hold served points (at most 21 of 64:
// they lie within 10 cells of the centre), two real rows per complex transform: with 16
// groups to a block most have one.
// 128 x 5: 107 us for 576 squares and 8 functions (256 x 3: 129, 128 x 6: 111, 64 x 10: 113)
constexpr int kSolveThreads = 128;
__global__ void __launch_bounds__(kSolveThreads, 5)
k_sq_solve(int n_f, const c64* __restrict__ spec, const int* __restrict__ exps,
           const int4* __restrict__ fac, const int4* __restrict__ tw,
           const int32_t* __restrict__ served_off, const int32_t* __restrict__ served_at,
           const int32_t* __restrict__ served_local, const int32_t* __restrict__ rows,
           double* __restrict__ out) {
  constexpr int kT = kHalf, kG = kSolveThreads / 8;  // kT: row stride of T (odd); groups
  extern __shared__ __align__(16) unsigned char smem_raw[];
  c64* ex = reinterpret_cast<c64*>(smem_raw);  // per group: an exchange sequence of 72
  c64* T = ex + kG * 72;                       // [rows][33]
  __shared__ unsigned st[1];
  const int sq = blockIdx.x, f = blockIdx.y, tid = threadIdx.x, g = tid >> 3, q = tid & 7;
  if (tid == 0) st[0] = 0;
  const c64* Z = spec + ((size_t)sq * n_f + f) * (2 * kHalf * kP);
  const int r0 = __ldg(rows + 2 * sq), nr = __ldg(rows + 2 * sq + 1) - r0 + 1;
  auto value = [&](int l, int m) {  // conj(a)
    const int t = l * kP + m;
    const c64 F = Z[2 * t], G = Z[2 * t + 1];
    const int4 w = __ldg(fac + t);
    return c64{dot(F.x, G.x, w), -dot(F.y, G.y, w)};
  };
  c64 v[8];
  c64* mine = ex + g * 72;
  unsigned h = 0;
  __syncthreads();  // st is zero
#pragma unroll 1
  for (int l = g; l < kP / 2; l += kG) {
#pragma unroll
    for (int r = 0; r < 8; ++r) v[r] = value(l, q + 8 * r);
    if (l == 0) {  // + i times the sequence l = 32
#pragma unroll
      for (int r = 0; r < 8; ++r) {
        const c64 b = value(kP / 2, q + 8 * r);
        v[r].x -= b.y;
        v[r].y += b.x;
      }
    }
    __syncwarp();
    dft64_group<1>(v, mine, q, tw);  // v[k]: y = q + 8 k
#pragma unroll
    for (int k = 0; k < 8; ++k) {
      const int y = q + 8 * k - r0;
      if (y >= 0 && y < nr) {
        h |= spread(v[k]);
        if (l == 0) {
          T[y * kT] = {v[k].x, 0};
          T[y * kT + kP / 2] = {v[k].y, 0};
        } else {
          T[y * kT + l] = v[k];
        }
      }
    }
  }
  block_or(h, st);
  __syncthreads();
  // two rows X_l = T(l, y1) + i T(l, y2): to |X| <= 2^58.5
  const int L = headroom(st[0]) - kDrop - 1;
  const int e = exps[(size_t)sq * n_f + f] + 3 * kDrop - L;
  const bool plain = plain_exp(e);
  const int s0 = __ldg(served_off + sq), s1 = __ldg(served_off + sq + 1);
#pragma unroll 1
  for (int p0 = 0; 2 * p0 < nr; p0 += kG) {
    const int p = p0 + g;
    if (2 * p < nr) {
      const c64 *a = T + 2 * p * kT, *b = a + kT;
      const bool two = 2 * p + 1 < nr;
#pragma unroll
      for (int r = 0; r < 8; ++r) {
        const int l = q + 8 * r, k = l <= kP / 2 ? l : kP - l;
        c64 x = a[k], y = two ? b[k] : c64{0, 0};
        if (l > kP / 2) {
          x.y = -x.y;
          y.y = -y.y;
        }
        v[r] = {shift(x.x, L) - shift(y.y, L), shift(x.y, L) + shift(y.x, L)};
      }
    }
    if (__any_sync(0xFFFFFFFFu, 2 * p < nr)) {
      dft64_group<1>(v, mine, q, tw);
#pragma unroll
      for (int k = 0; k < 8; ++k) mine[pad(q + 8 * k)] = v[k];
    }
    __syncthreads();
    for (int k = s0 + tid; k < s1; k += kSolveThreads) {
      const int loc = __ldg(served_local + k), y = (loc >> 6) - r0, x = loc & 63, r = (y >> 1) - p0;
      if (r >= 0 && r < kG) {
        const c64 z = ex[r * 72 + pad(x)];
        out[(size_t)__ldg(served_at + k) * n_f + f] = to_double((y & 1) ? z.y : z.x, e, plain);
      }
    }
    __syncthreads();
  }
}

// The factors of the small steps s < S: fac[s][l][m], l <= 32, at s dt (dt = h/(8 c) here
// enters as its own argument): limbs of (cos w t, 2^-eT sin(w t)/w), (1, 2^-eT t) at w = 0.
__global__ void k_sq_factors(int S, double c, double h, double dt, int eT, int4* __restrict__ fac) {
  const int64_t t = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
  if (t >= (int64_t)S * kHalf * kP) return;
  const int s = (int)(t / (kHalf * kP)), lm = (int)(t - (int64_t)s * kHalf * kP);
  const int l = lm >> 6, m = lm & 63, ms = m <= kP / 2 ? m : kP - m;
  const double box = kP * h, tau = s * dt, fl = l / box, fm = ms / box;
  const double w = 6.283185307179586476925286766559 * c * sqrt(fl * fl + fm * fm);
  double co = 1.0, si = tau;
  if (w > 0.0) {
    sincos(w * tau, &si, &co);
    si /= w;
  }
  const i64 p = __double2ll_rn(ldexp(co, 60)), q = __double2ll_rn(ldexp(si, 60 - eT));
  fac[t] = {hi32(p), lo32(p), hi32(q), lo32(q)};
}

}  // namespace fx

size_t squares_spectrum_bytes(int n_sq, int n_f) {
  return (size_t)n_sq * n_f * 2 * fx::kHalf * fx::kP * sizeof(fx::c64);
}
size_t squares_factor_bytes(int S) { return (size_t)S * fx::kHalf * fx::kP * sizeof(int4); }

void squares_factors(int S, double c, double h, double dt, int eT, void* fac, cudaStream_t s) {
  const int64_t n = (int64_t)S * fx::kHalf * fx::kP;
  fx::k_sq_factors<<<(unsigned)((n + 255) / 256), 256, 0, s>>>(S, c, h, dt, eT, (int4*)fac);
}

void squares_expand(const SquareArgs& q, int n_side, int C, int d, int nx, int64_t grid_stride,
                    int n_f, int eT, const double* u, const double* ut, void* spec, int* exps,
                    cudaStream_t s) {
  const size_t sm = ((size_t)(fx::kP + fx::kP / 8 - 1) * fx::kRow + (size_t)fx::kP * 2 * d) * 16;
  cudaFuncSetAttribute(fx::k_sq_expand, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)sm);
  fx::k_sq_expand<<<dim3(q.n, n_f), fx::kThreads, sm, s>>>(n_side, C, d, nx, grid_stride, n_f, eT,
                                                          q.origin, q.A, q.Q, q.tw, u, ut,
                                                          (fx::c64*)spec, exps);
}

void squares_solve(const SquareArgs& q, int max_rows, int n_f, const void* spec, const int* exps,
                   const void* fac, int step, double* out, cudaStream_t s) {
  const size_t sm = ((size_t)(fx::kSolveThreads / 8) * 72 + (size_t)max_rows * fx::kHalf) * 16;
  cudaFuncSetAttribute(fx::k_sq_solve, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)sm);
  fx::k_sq_solve<<<dim3(q.n, n_f), fx::kSolveThreads, sm, s>>>(
      n_f, (const fx::c64*)spec, exps, (const int4*)fac + (size_t)step * fx::kHalf * fx::kP, q.tw,
      q.served_off, q.served_at, q.served_local, q.rows, out);
}

}  // namespace fc2d
