// Fourier Forwarding's modal solutions in block fixed point (fx.cuh): the time factors,
// the modal advance fused into the inverse column transform, and the inverse real rows.
//
// A mode (l, m) of the box turns at w = 2 pi c kappa / h with kappa = |(l/nx, m/ny)|, so at
// time t its phase is the fraction of kappa (c t / h) turns, a 64-bit integer product.  Its
// cosine and sine come from a table of 512 directions and short Taylor series in the rest,
// all in integers: FP64 sincos costs about 40 FP64 instructions, at 2 per clock and SM
// more than the transform of the column itself.
//
// With F, G the spectra of u and u_t, a = F cos(w t) + G sin(w t)/w and a' = -F w sin(w t) +
// G cos(w t).  F and G 2^eT (2^eT >= t) are kept as integers with a common exponent per
// block of the column pass A (64 rows x 16 columns), made from the doubles once per large
// step (k_spec_fix), so the factors are at most 1 and pass A starts without a block maximum.
#include <cuda_runtime.h>

#include <algorithm>
#include <cmath>
#include <cstdint>
#include <vector>

#include "fc2d_kernels.cuh"
#include "fx.cuh"
#include "plan_internal.h"

namespace fc2d {
namespace fx {

constexpr int kTurn = 512;  // directions of the table

// kappa and 1/(2 pi kappa) of the modes m <= ny/2, l <= nx/2
struct Mode {
  unsigned long long kappa;  // kappa 2^64
  i64 inv;                   // 1/(2 pi kappa) = (inv >> 8) 2^-55 2^(inv & 255), inv >> 8 in [2^54, 2^55)
};

struct Modes {
  Mode* tab = nullptr;     // [ny/2 + 1][nx/2 + 1]
  longlong2* turn = nullptr;  // (cos, sin)(2 pi i/512) 2^62
  int4* fac = nullptr;        // the factors at the current time (k_factors)
};

__global__ void k_modes(int nx, int ny, Mode* __restrict__ tab) {
  const int l = blockIdx.x * blockDim.x + threadIdx.x, m = blockIdx.y;
  if (l > nx / 2) return;
  // kappa = sqrt(D)/(nx ny) with the integer D = (l ny)^2 + (m nx)^2 < 2^53 exact; the root
  // and the quotient in two doubles each
  const double a = (double)l * ny, b = (double)m * nx, D = a * a + b * b, n = (double)nx * ny;
  const double s = sqrt(D), ds = s > 0 ? fma(-s, s, D) / (2 * s) : 0.0;
  const double q = s / n, dq = (fma(-q, n, s) + ds) / n;
  const double hi = q * 18446744073709551616.0, fl = floor(hi);
  Mode o;
  o.kappa = (unsigned long long)fl + (unsigned long long)__double2ll_rn((hi - fl) + dq * 18446744073709551616.0);
  o.inv = 0;
  if (s > 0) {  // 1/(2 pi (q + dq)) = r + dr
    const double two_pi = 6.283185307179586476925286766559, two_pi_lo = 2.4492935982947064e-16;
    const double p = two_pi * q, dp = fma(two_pi, q, -p) + fma(two_pi_lo, q, two_pi * dq);
    const double r = 1.0 / p, dr = r * (fma(-r, p, 1.0) - r * dp);
    int e;
    const double f = frexp(r, &e);  // [1/2, 1)
    o.inv = (((i64)(f * 36028797018963968.0) + __double2ll_rn(ldexp(dr, 55 - e))) << 8) | (i64)(e & 255);  // 2^55
  }
  tab[(size_t)m * (nx / 2 + 1) + l] = o;
}

// Everything of a time that its factors need
struct When {
  unsigned long long cells, frac;  // c t / h = cells + frac 2^-64
  i64 tau;                         // t 2^-eT 2^62 (in [2^61, 2^62])
  i64 hc;                          // (h/c) 2^-eT = hc 2^-62 2^ehc, hc in [2^61, 2^62)
  int ehc;
  i64 nu;                          // 8 (c/h) 2^-eS 2^62
  int down;                        // eT + eS >= 0
  int eS;
  int eT;
};

// cos and sin of phase 2^-64 turns, times 2^62; `small`: the phase is within 1/1024 turn of
// 0, and then sinc = (sin x)/x 2^62 (x the angle)
__device__ __forceinline__ void cos_sin(unsigned long long phase, const longlong2* __restrict__ turn,
                                        i64& co, i64& si, bool& small, i64& sinc) {
  const unsigned long long r = phase + (1ull << 54);
  const int idx = (int)(r >> 55);
  const i64 d = (i64)(r & ((1ull << 55) - 1)) - (1ll << 54);  // |d| <= 2^54, angle 2 pi d 2^-64
  // angle x 2^69 = d 2^8 (pi/4), pi/4 - 1 = m 2^-32 + r 2^-64
  const i64 x = mulc(d << 8, -921707870, 560513589);
  const i64 x2 = mulh(x, x);  // x^2 2^74 < 2^60
  constexpr i64 k62 = 1ll << 62;
  // 1 - cos x = x^2 (1/2 - x^2 (1/24 - x^2/720)), sin x = x (1 - x^2 (1/6 - x^2/120)); the
  // polynomials times 2^62 (x^2 2^74 times y 2^62 is 2^72: shift by 10)
  const i64 p1 = k62 / 24 - (mulh(x2, k62 / 720) >> 10);
  const i64 p2 = k62 / 2 - (mulh(x2, p1) >> 10);
  const i64 vers = mulh(x2, p2);  // (1 - cos x) 2^72
  const i64 s1 = k62 / 6 - (mulh(x2, k62 / 120) >> 10);
  const i64 sc = k62 - (mulh(x2, s1) >> 10);  // sinc 2^62
  const i64 sx = mulh(x, sc);                 // sin x 2^67
  const longlong2 t = __ldg(turn + idx);
  // cos(a + x) = C - C vers - S sin x, sin(a + x) = S - S vers + C sin x
  const i64 cv = mulh(vers, t.x), sv = mulh(vers, t.y);  // 2^70
  const i64 cs = mulh(sx, t.x), ss = mulh(sx, t.y);      // 2^65
  co = t.x - ((cv + (ss << 5) + 128) >> 8);
  si = t.y - ((sv - (cs << 5) + 128) >> 8);
  small = idx == 0;
  sinc = sc;
}

__device__ __forceinline__ int4 limbs(i64 p, i64 q) { return {hi32(p), lo32(p), hi32(q), lo32(q)}; }

// The factors (t0, t1) of F and G 2^eT, as limbs of t 2^60: of a (deriv false) or a' 2^-eS
__device__ __forceinline__ int4 factors(const Mode& md, const When& w, const longlong2* __restrict__ turn,
                                        bool deriv) {
  const unsigned long long lo = md.kappa * w.cells, phase = lo + __umul64hi(md.kappa, w.frac);
  i64 co, si, sinc;
  bool small;
  cos_sin(phase, turn, co, si, small, sinc);
  if (deriv) {  // -w sin(w t) 2^-eS = -sin (2 pi kappa/8) nu
    const i64 kp = mulc((i64)(md.kappa >> 2), -921707870, 560513589);  // kappa (pi/4) 2^62
    return limbs(-mulh(mulh(si, kp) << 2, w.nu), (co >> 2) >> min(w.down, 62));
  }
  // an angle below 1/1024 turn in all: t1 = t sinc, which keeps its relative precision
  small = small && phase < (1ull << 54) && __umul64hi(md.kappa, w.cells) == 0 && phase >= lo;
  i64 t1;
  if (small) {
    t1 = mulh(w.tau, sinc);
  } else {  // sin (h/c) 2^-eT / (2 pi kappa)
    const i64 q = mulh(mulh(si, w.hc) << 2, (md.inv >> 8) << 7);
    const int up = (int)(signed char)(md.inv & 255) + w.ehc;
    t1 = up >= 0 ? q << up : q >> min(-up, 63);
  }
  return limbs(co >> 2, t1);
}

// The spectra F (spec[f]) and G (spec[n_f + f]), [ny][nx/2+1] doubles, into integers in
// place: F and G 2^eT in units of 2^exps[f][j2][column group], |values| < 2^61.
template <int N2>
__global__ void __launch_bounds__(kColThreads)
k_spec_fix(int nxh, int n_f, int eT, double2* __restrict__ spec, int* __restrict__ exps) {
  __shared__ unsigned st[2];
  if (threadIdx.x < 2) st[threadIdx.x] = 0;
  const int c = threadIdx.x & (kCols - 1), l = threadIdx.x / kCols, kx = blockIdx.x * kCols + c;
  const int j2 = blockIdx.y, f = blockIdx.z;
  const bool live = kx < nxh;
  double2* F = spec + (size_t)f * (64 * N2) * nxh + kx;
  double2* G = spec + (size_t)(n_f + f) * (64 * N2) * nxh + kx;
  __syncthreads();
  pdl_wait();
  pdl_trigger();
  double2 u[8], v[8];
  unsigned mu = 0, mv = 0;
#pragma unroll
  for (int i = 0; i < 8; ++i) {
    const unsigned o = (unsigned)(N2 * (l + 8 * i) + j2) * (unsigned)nxh;
    u[i] = live ? F[o] : double2{0.0, 0.0};
    v[i] = live ? G[o] : double2{0.0, 0.0};
    mu = max(mu, max(magnitude(u[i].x), magnitude(u[i].y)));
    mv = max(mv, max(magnitude(v[i].x), magnitude(v[i].y)));
  }
  block_max(mu, st);
  block_max(mv, st + 1);
  __syncthreads();
  const int EF = block_exp(st[0]), EG = block_exp(st[1]), E = max(EF, EG + eT);
  if (live) {
#pragma unroll
    for (int i = 0; i < 8; ++i) {
      const unsigned o = (unsigned)(N2 * (l + 8 * i) + j2) * (unsigned)nxh;
      reinterpret_cast<c64*>(F)[o] = from_double<8>(u[i], E);
      reinterpret_cast<c64*>(G)[o] = from_double<8>(v[i], E - eT);
    }
  }
  if (threadIdx.x == 0)
    exps[((size_t)f * N2 + j2) * gridDim.x + blockIdx.x] = max(EF, EG) >= 0x7FF ? kNaN : E - 1083;
}

// The factors of all modes m <= ny/2 at one time, [ny/2 + 1][nx/2 + 1]
__global__ void __launch_bounds__(256)
k_factors(int nxh, bool deriv, When w, const Mode* __restrict__ modes,
          const longlong2* __restrict__ turn, int4* __restrict__ fac) {
  const int l = blockIdx.x * blockDim.x + threadIdx.x;
  const size_t at = (size_t)blockIdx.y * nxh + l;
  int4 v{};
  if (l < nxh) v = factors(modes[at], w, turn, deriv);
  pdl_wait();
  pdl_trigger();
  if (l < nxh) fac[at] = v;
}

// The modal solutions in FP64: a into F and a' into the first half of `deriv`, whose other half
// and G become zero.  For times in which a wave crosses less than an eighth of a cell (or
// times that no fixed-point phase holds): F and G t, or F w^2 t and G, then differ by
// more orders of magnitude than their common exponent leaves bits for.  A thread per mode for all
// functions, bound by the FP64 pipe: the call at 2048^2 takes 725 us with it and 418 with the
// fixed-point factors.
__global__ void __launch_bounds__(128)
k_modal_double(int nxh, int ny, int n_f, double c, double t, double Lx, double Ly,
               double2* __restrict__ spec, double2* __restrict__ deriv) {
  const int kx = blockIdx.x * blockDim.x + threadIdx.x, ky = blockIdx.y;
  pdl_wait();
  pdl_trigger();
  if (kx >= nxh) return;
  const double fl = kx / Lx, fm = (ky <= ny / 2 ? ky : ky - ny) / Ly;
  const double w = 6.283185307179586476925286766559 * c * sqrt(fl * fl + fm * fm);
  double si = 0.0, co = 1.0, sw = t;
  if (w != 0.0) {
    sincos(w * t, &si, &co);
    sw = si / w;
  }
  const size_t slab = (size_t)ny * nxh;
  for (int f = 0; f < n_f; ++f) {
    const size_t o = f * slab + (size_t)ky * nxh + kx, g = o + n_f * slab;
    const double2 F = spec[o], G = spec[g];
    spec[o] = {F.x * co + G.x * sw, F.y * co + G.y * sw};
    deriv[o] = {G.x * co - F.x * w * si, G.y * co - F.y * w * si};
    spec[g] = deriv[g] = {0.0, 0.0};
  }
}

// Modal advance and pass A of the inverse column transform (a forward transform of the
// conjugate) for the functions f0 <= f < f0 + gridDim.z: spec, exps as k_spec_fix leaves
// them; mid [nf][ny][pitch] integers with exponents mexps[nf][N2][column group].
// DERIV: a', whose factor w sin(w t) spans the orders of magnitude of w: the products keep 31
// bits more, and the block takes those that its largest value allows.  The block is rescaled between
// the halves of the transform (27.5 -> 28.3 us at 2048^2, see shifts() in fx.cuh).
template <int N2, bool DERIV>
__global__ void __launch_bounds__(kColThreads, DERIV ? 4 : 8)
k_adv_a(int nxh, unsigned pitch, int n_f, int f0, int eS, const int4* __restrict__ fac,
        const c64* __restrict__ spec, const int* __restrict__ exps, const int4* __restrict__ tw,
        c64* __restrict__ mid, int* __restrict__ mexps) {
  constexpr int ny = 64 * N2;
  __shared__ c64 ex[64 * kCols];
  __shared__ unsigned st[2];
  if (threadIdx.x < 2) st[threadIdx.x] = 0;
  const int c = threadIdx.x & (kCols - 1), l = threadIdx.x / kCols, kx = blockIdx.x * kCols + c;
  const int j2 = blockIdx.y, f = blockIdx.z;
  const bool live = kx < nxh;
  __syncthreads();
  pdl_wait();
  pdl_trigger();
  const c64* F = spec + (size_t)(f0 + f) * ny * nxh + kx;
  const c64* G = spec + (size_t)(n_f + f0 + f) * ny * nxh + kx;
  c64 v[8];
  int up = 0;
  auto factor = [&](int row) { return __ldg(fac + (unsigned)(row <= ny / 2 ? row : ny - row) * (unsigned)nxh + kx); };
  if constexpr (DERIV) {
    Wide x[8], y[8];
    unsigned h = 0;
#pragma unroll
    for (int i = 0; i < 8; ++i) {
      const int row = N2 * (l + 8 * i) + j2;
      const unsigned o = (unsigned)row * (unsigned)nxh;
      x[i] = y[i] = Wide{0, 0};
      if (live) {
        const c64 a = F[o], b = G[o];
        const int4 t = factor(row);
        x[i] = dot_wide(a.x, b.x, t);
        y[i] = dot_wide(a.y, b.y, t);
        h |= spread(x[i].hi + (x[i].mid >> 32)) | spread(y[i].hi + (y[i].mid >> 32));
      }
    }
    block_or(h, st);
    __syncthreads();
    up = min(max(headroom(st[0]) - 4, 0), 28);  // values below 2^58
#pragma unroll
    for (int i = 0; i < 8; ++i)
      v[i] = {(x[i].hi << up) + (x[i].mid >> (32 - up)), -(y[i].hi << up) - (y[i].mid >> (32 - up))};
  } else {
#pragma unroll
    for (int i = 0; i < 8; ++i) {
      const int row = N2 * (l + 8 * i) + j2;
      const unsigned o = (unsigned)row * (unsigned)nxh;
      v[i] = {0, 0};
      if (live) {
        const c64 a = F[o], b = G[o];
        const int4 t = factor(row);
        v[i] = {dot(a.x, b.x, t), -dot(a.y, b.y, t)};
      }
    }
  }
  const int L = dft_group<8, true>(v, c, l, ex, tw, N2, st + 1);
  if (live) {
    c64* out = mid + (size_t)f * ny * pitch + kx;
#pragma unroll
    for (int q = 0; q < 8; ++q) out[(unsigned)(N2 * (l + 8 * q) + j2) * pitch] = v[q];
  }
  if (threadIdx.x == 0)
    mexps[((size_t)f * N2 + j2) * gridDim.x + blockIdx.x] =
        exps[((size_t)(f0 + f) * N2 + j2) * gridDim.x + blockIdx.x] + 2 * kDrop + eS - up - L;
}

// Pass B of the inverse column transform: its conjugate, as doubles, [nf][ny][pitch]
template <int N2>
__global__ void __launch_bounds__(kColThreads, 8)
k_adv_b(int nxh, unsigned pitch, const c64* __restrict__ mid, const int* __restrict__ mexps,
        const int4* __restrict__ tw, double2* __restrict__ out) {
  constexpr int R2 = N2 / 8, G = 8 / R2;
  __shared__ c64 ex[64 * kCols];
  __shared__ unsigned st[1];
  if (threadIdx.x == 0) st[0] = 0;
  const int c = threadIdx.x & (kCols - 1), kx = blockIdx.x * kCols + c;
  const int l = (threadIdx.x / kCols) % R2, g = threadIdx.x / (kCols * R2), f = blockIdx.z;
  const int m1 = blockIdx.y * G + g;
  const bool live = kx < nxh;
  __syncthreads();
  pdl_wait();
  pdl_trigger();
  c64 v[8];
  const int e = cols_pass_b<N2>(v, mid + (size_t)f * (64 * N2) * pitch, pitch, m1, l, kx, live,
                                ex + g * 8 * R2 * kCols, st, tw,
                                mexps + (size_t)f * N2 * gridDim.x + blockIdx.x, gridDim.x);
  const bool plain = plain_exp(e);
  if (live) {
    double2* dst = out + (size_t)f * (64 * N2) * pitch + kx;
#pragma unroll
    for (int mm = 0; mm < 8 / R2; ++mm)
#pragma unroll
      for (int q = 0; q < R2; ++q) {
        const double2 z = to_double(v[mm * R2 + q], e, plain);
        dst[(unsigned)(m1 + 64 * (l * (8 / R2) + mm + 8 * q)) * pitch] = double2{z.x, -z.y};
      }
  }
}

// Inverse real row DFT: Z_k = S_k + i conj(w^k) D_k with S_k, D_k = X_k +- conj(X_{NH-k});
// the length-NH transform runs as a forward transform of conj(Z), and x_{2m} + i x_{2m+1} is
// the conjugate of its result; plus c00[f] (x^2 + y^2)/4 when c00 is given.  One block per
// (row, function).  With point_off only the values at the row's listed points (point_off[j] ..
// point_off[j+1], linear grid indices) are written, to out[point][ld] at column f, and rows
// without any are skipped.
template <int LOGNH>
__global__ void __launch_bounds__((1 << LOGNH) / 8 < 32 ? 32 : (1 << LOGNH) / 8,
                                  (1 << LOGNH) / 8 >= 128 ? 1024 / ((1 << LOGNH) / 8) : 8)
k_inverse_rows_fx(FftArgs fa, const double2* __restrict__ inter, const double* __restrict__ c00,
                  double a0, double b0, double h, double* __restrict__ out,
                  const int32_t* __restrict__ point_off, const int32_t* __restrict__ points, int ld) {
  constexpr int NH = 1 << LOGNH, NT = NH / 8, R = last_radix<LOGNH>();
  extern __shared__ __align__(16) unsigned char smem_raw[];
  __shared__ unsigned st[kSlots];
  c64* buf = reinterpret_cast<c64*>(smem_raw);
  const int j = blockIdx.x, f = blockIdx.y, t = threadIdx.x;
  const bool active = t < NT;
  int p0 = 0, p1 = 0;
  if (point_off) {
    p0 = point_off[j];
    p1 = point_off[j + 1];
    if (p0 == p1) return;
  }
  if (t < kSlots) st[t] = 0;
  __syncthreads();
  pdl_wait();
  pdl_trigger();
  // X_k and X_{NH-k}, k = t + i NT < NH/2, and X_{NH/2}
  const double2* row = inter + ((size_t)f * fa.ny + j) * fa.pitch;
  double2 a[4], b[4], mid{0.0, 0.0};
  unsigned mag = 0;
  if (active) {
#pragma unroll
    for (int i = 0; i < 4; ++i) {
      a[i] = row[t + i * NT];
      b[i] = row[NH - t - i * NT];
      mag = max(mag, max(max(magnitude(a[i].x), magnitude(a[i].y)), max(magnitude(b[i].x), magnitude(b[i].y))));
    }
    if (t == 0) {
      mid = row[NH / 2];
      mag = max(mag, max(magnitude(mid.x), magnitude(mid.y)));
    }
  }
  block_max(mag, st);
  __syncthreads();
  // |X| < 2^60.5, |S|, |D| < 2^61.5, |Z| < 2^58.5
  const int E = block_exp(st[0]);
  int e = E - 1082 + kDrop;
  if (active) {
#pragma unroll
    for (int i = 0; i < 4; ++i) {
      const int k = t + i * NT;
      const c64 x = from_double<7>(a[i], E), y = from_double<7>(b[i], E);
      const c64 s = drop(c64{x.x + y.x, x.y - y.y});
      const c64 q = mulw_conj(c64{x.x - y.x, x.y + y.y}, __ldg(fa.fxr + k));  // i q = T
      buf[pad(k)] = {s.x - q.y, -s.y - q.x};                     // conj(S + T)
      if (k) buf[pad(NH - k)] = {s.x + q.y, s.y - q.x};          // S - T
    }
    if (t == 0) {  // Z = 2 conj(X): S = 2 re X, T = i i (2 i im X)
      const c64 x = from_double<7>(mid, E);
      buf[pad(NH / 2)] = drop(c64{x.x + x.x, x.y + x.y});
    }
  }
  __syncthreads();
  c64 v[8];
  if (active) {
#pragma unroll
    for (int r = 0; r < 8; ++r) v[r] = buf[pad(t + r * NT)];
  }
  transform<LOGNH>(v, buf, t, active, st, fa.fxx, e);
  if (E >= 0x7FF) e = kNaN;
  const bool plain = plain_exp(e);
  if (point_off) {
    __syncthreads();
    if (active) {
#pragma unroll
      for (int m = 0; m < 8 / R; ++m)
#pragma unroll
        for (int r = 0; r < R; ++r) buf[pad(out_index<LOGNH>(t, m, r))] = v[m * R + r];
    }
    __syncthreads();
    for (int p = p0 + t; p < p1; p += blockDim.x) {
      const int x = points[p] - j * (2 * NH);
      const c64 z = buf[pad(x >> 1)];
      out[(size_t)p * ld + f] = (x & 1) ? to_double(-z.y, e, plain) : to_double(z.x, e, plain);
    }
    return;
  }
  if (!active) return;
  double* dst = out + (size_t)f * fa.ny * (2 * NH);
  const double q = c00 ? c00[f] * 0.25 : 0.0, y = b0 + h * double(j);
#pragma unroll
  for (int m = 0; m < 8 / R; ++m)
#pragma unroll
    for (int r = 0; r < R; ++r) {
      const int k = out_index<LOGNH>(t, m, r);
      const double2 z = to_double(v[m * R + r], e, plain);
      double2 o = {z.x, -z.y};
      if (c00) {
        const double x0 = a0 + h * double(2 * k), x1 = a0 + h * double(2 * k + 1);
        o.x += q * (x0 * x0 + y * y);
        o.y += q * (x1 * x1 + y * y);
      }
      dst[(size_t)j * (2 * NH) + 2 * k] = o.x;
      dst[(size_t)j * (2 * NH) + 2 * k + 1] = o.y;
    }
}

template <int L>
static void inverse_rows_launch(const FftArgs& fa, int n_f, const void* inter, const double* c00,
                                double a0, double b0, double h, double* out, const int32_t* off,
                                const int32_t* points, int ld, cudaStream_t s) {
  const size_t sm = (size_t)padded(1 << L) * sizeof(c64);
  cudaFuncSetAttribute(k_inverse_rows_fx<L>, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)sm);
  launch_pdl(k_inverse_rows_fx<L>, dim3(fa.ny, n_f), dim3(std::max(32, (1 << L) / 8)), sm, s, fa,
             (const double2*)inter, c00, a0, b0, h, out, off, points, ld);
}

static int ilog2_exact(int n) {
  if (n <= 0 || (n & (n - 1))) return -1;
  int l = 0;
  while ((1 << l) < n) ++l;
  return l;
}

// v + lo times 2^k, rounded
static i64 scaled_pair(double v, double lo, int k) {
  return (i64)std::ldexp(v, k) + (i64)std::nearbyint(std::ldexp(lo, k));
}

// (t, eT): t <= 2^eT; cells + cells_lo = c t / h.  Quotients in two doubles each: a factor rounded to
// 53 bits is off by the same relative amount at every mode.
static When when(double t, double cells, double cells_lo, double c, double h, int eT) {
  When w{};
  const double x = std::min(cells, 9.0e18), fl = std::floor(x);
  const __int128 n = ((__int128)(i64)fl << 64) + (__int128)std::ldexp(x - fl, 64) +
                     (__int128)std::nearbyint(std::ldexp(cells_lo, 64));
  w.cells = n < 0 ? 0 : (unsigned long long)(n >> 64);
  w.frac = n < 0 ? 0 : (unsigned long long)n;
  w.tau = (i64)std::ldexp(t, 62 - eT);
  const double hc = h / c, hc_lo = std::fma(-hc, c, h) / c;
  std::frexp(hc, &w.ehc);
  w.hc = scaled_pair(hc, hc_lo, 62 - w.ehc);
  w.ehc -= eT;
  const double nu = 8 * c / h, nu_lo = std::fma(-nu, h, 8 * c) / h;
  int k;
  std::frexp(nu, &k);
  w.eT = eT;
  w.eS = std::max(k, -eT);
  w.nu = scaled_pair(nu, nu_lo, 62 - w.eS);
  w.down = eT + w.eS;
  return w;
}

}  // namespace fx

// Inverse real rows of power-of-two length (nx/2 = 2^5 .. 2^12), to the whole grid or, with
// off, at the listed points (out[point][ld]); false (nothing launched) for other sizes.
bool launch_inverse_rows_fx(const FftArgs& fa, int n_f, const void* inter, const double* c00,
                            double a0, double b0, double h, double* out, const int32_t* off,
                            const int32_t* points, int ld, cudaStream_t s) {
  switch (fx::ilog2_exact(fa.nx / 2)) {
#define FC2D_INV(L) \
  case L: fx::inverse_rows_launch<L>(fa, n_f, inter, c00, a0, b0, h, out, off, points, ld, s); return true;
    FC2D_INV(5) FC2D_INV(6) FC2D_INV(7) FC2D_INV(8)
    FC2D_INV(9) FC2D_INV(10) FC2D_INV(11) FC2D_INV(12)
#undef FC2D_INV
    default: return false;
  }
}

void launch_inverse_rows_mixed(const FftArgs& fa, int n_f, const void* inter, const double* c00,
                               double a0, double b0, double h, double* out, const int32_t* off,
                               const int32_t* points, int ld, cudaStream_t s);
void launch_spec_fix_mixed(const FftArgs& fa, int n_f, int eT, void* spec, int* exps, cudaStream_t s);
void launch_adv_mixed(const FftArgs& fa, int n_f, int f0, int nf, bool deriv, int eS, const int4* fac,
                      const void* spec, const int* exps, void* mid, int* mexps, void* res, cudaStream_t s);

// columns of 64 x 8, 16, 32 or 64 points
static bool wave_cols64(int ny) { return ny == 512 || ny == 1024 || ny == 2048 || ny == 4096; }

// The exponent eT of the times up to t: 2^eT >= t, and at least the time h/(8 c) in which a
// wave crosses an eighth of a cell (u_t is of the size of w u, w up to 4.4 c/h)
int wave_fx_time(double t, double h, double c) {
  const double x = std::max(t, h / (8 * c));
  int e = 0;
  if (std::isfinite(x)) std::frexp(x, &e);
  return e;
}

// The plan's mode table, built on first use: on a stream of its own and in the relaxed capture
// mode, so that the first call may come while streams are captured and waits for nothing else
static fc2d_status build_modes(fc2d_plan_s* p, fx::Modes* m) {
  const int nx = p->grid.nx, ny = p->grid.ny;
  const std::vector<int64_t> turn = fx_turn_table(fx::kTurn);
  const size_t modes = (size_t)(ny / 2 + 1) * (nx / 2 + 1);
  fx::Mode* tab = nullptr;
  if ((!m->turn && cudaMalloc(&m->turn, turn.size() * 8) != cudaSuccess) ||
      (!m->fac && cudaMalloc(&m->fac, modes * sizeof(int4)) != cudaSuccess) ||
      cudaMalloc(&tab, modes * sizeof(fx::Mode)) != cudaSuccess) {
    cudaGetLastError();
    return set_error(FC2D_ERR_NOMEM, "wave modes: device allocation failed");
  }
  cudaStream_t s = nullptr;
  fc2d_status st = cuda_check(cudaStreamCreateWithFlags(&s, cudaStreamNonBlocking), "wave modes");
  if (!st) {
    st = cuda_check(cudaMemcpyAsync(m->turn, turn.data(), turn.size() * 8, cudaMemcpyHostToDevice, s),
                    "wave modes");
    fx::k_modes<<<dim3((nx / 2 + 256) / 256, ny / 2 + 1), 256, 0, s>>>(nx, ny, tab);
    const fc2d_status done = cuda_check(cudaStreamSynchronize(s), "wave modes");
    if (!st) st = done;
    cudaStreamDestroy(s);
  }
  if (st) cudaFree(tab);
  else m->tab = tab;
  return st;
}

static fc2d_status wave_modes(fc2d_plan_s* p, fx::Modes** out) {
  auto* m = static_cast<fx::Modes*>(p->modes);
  if (!m) {
    m = new fx::Modes();
    p->modes = m;  // freed with the plan, whatever happens below
  }
  if (!m->tab) {
    cudaStreamCaptureMode mode = cudaStreamCaptureModeRelaxed;
    cudaThreadExchangeStreamCaptureMode(&mode);
    const fc2d_status st = build_modes(p, m);
    cudaThreadExchangeStreamCaptureMode(&mode);
    if (st) return st;
  }
  *out = m;
  return FC2D_OK;
}

void wave_modes_destroy(fc2d_plan_s* p) {
  auto* m = static_cast<fx::Modes*>(p->modes);
  if (!m) return;
  cudaFree(m->tab);
  cudaFree(m->turn);
  cudaFree(m->fac);
  delete m;
  p->modes = nullptr;
}

// Functions per launch: 160 MB of intermediate.  Smaller launches would keep it in L2, but
// their last waves cost more (8 solutions at 1024^2, one large step: 12.0 ms with 40 MB, 11.2
// with 80 MB or more)
static int wave_chunk(const FftArgs& fa, int n_f) {
  const size_t one = (size_t)fa.ny * fa.pitch * 16;
  return (int)std::min<size_t>(n_f, std::max<size_t>(1, (size_t(160) << 20) / one));
}

size_t wave_fx_exps(int nx, int ny, int n_f) { return 2 * fx_exps(nx, ny, n_f); }

fc2d_status wave_fx_prepare(fc2d_plan_s* p) {
  fx::Modes* m;
  return wave_modes(p, &m);
}

#define FC2D_N2(ny, CALL) \
  switch ((ny) / 64) {    \
    case 8: CALL(8); break;   \
    case 16: CALL(16); break; \
    case 32: CALL(32); break; \
    case 64: CALL(64); break; \
  }

// Spectra [2 n_f][ny][nx/2+1] (F's, then G's) to integers for times up to 2^eT.
void wave_fx_spectra(const FftArgs& fa, int n_f, int eT, void* spec, int* exps, cudaStream_t s) {
  if (!wave_cols64(fa.ny)) return launch_spec_fix_mixed(fa, n_f, eT, spec, exps, s);
  const dim3 grid(fa.nx / 32 + 1, fa.ny / 64, n_f);
#define CALL(N2) \
  launch_pdl(fx::k_spec_fix<N2>, grid, dim3(fx::kColThreads), 0, s, fa.nx / 2 + 1, n_f, eT, (double2*)spec, exps)
  FC2D_N2(fa.ny, CALL)
#undef CALL
}

// Modal solutions at time t in FP64, in place of the spectra; their time derivatives to `deriv`
// (as large).  wave_fx_eval at time 0 then gives either.
void wave_modal_double(const FftArgs& fa, int n_f, double c, double t, double h, void* spec, void* deriv,
                       cudaStream_t s) {
  const int nxh = fa.nx / 2 + 1;
  launch_pdl(fx::k_modal_double, dim3((nxh + 127) / 128, fa.ny), dim3(128), 0, s, nxh, fa.ny, n_f, c, t,
             fa.nx * h, fa.ny * h, (double2*)spec, (double2*)deriv);
}

// u (or, deriv, u_t) at time t = (cells + cells_lo) h / c of the modal solutions, on the grid or, with
// off, at the listed points (out[point][n_f]).  spec, exps: from wave_fx_spectra (exps has wave_fx_exps ints); inter:
// 2 n_f ny pitch complex values of scratch.
fc2d_status wave_fx_eval(fc2d_plan_s* p, const FftArgs& fa, int n_f, bool deriv, double c, double t,
                         double cells, double cells_lo, int eT, const void* spec, int* exps,
                         void* inter, double* out, const int32_t* off, const int32_t* points,
                         cudaStream_t s) {
  fx::Modes* m;
  fc2d_status st = wave_modes(p, &m);
  if (st) return st;
  const int nxh = fa.nx / 2 + 1, groups = fa.nx / 32 + 1, N2 = fa.ny / 64;
  const unsigned pitch = (unsigned)fa.pitch;
  // a speed or time without finite factors: NaN everywhere
  const bool lost = !std::isfinite(8 * c / p->grid.h) || !std::isfinite(t);
  const fx::When w = lost ? fx::when(0.0, 0.0, 0.0, 1.0, p->grid.h, 0)
                           : fx::when(t, cells, cells_lo, c, p->grid.h, eT);
  const int eS = lost ? fx::kNaN : deriv ? w.eS : 0;
  const int chunk = wave_chunk(fa, n_f);
  const size_t slab = (size_t)fa.ny * fa.pitch;
  auto* mid = static_cast<fx::c64*>(inter);
  auto* res = reinterpret_cast<double2*>(mid + chunk * slab);
  int* mexps = exps + fx_exps(fa.nx, fa.ny, n_f);
  {
    ProfScope ps(p, "ff_factors", s);
    launch_pdl(fx::k_factors, dim3((nxh + 255) / 256, fa.ny / 2 + 1), dim3(256), 0, s, nxh, deriv, w,
               m->tab, m->turn, m->fac);
  }
  for (int f0 = 0; f0 < n_f; f0 += chunk) {
    const int nf = std::min(chunk, n_f - f0);
    {
      ProfScope ps(p, "ff_cols", s);
      if (!wave_cols64(fa.ny)) {
        launch_adv_mixed(fa, n_f, f0, nf, deriv, eS, m->fac, spec, exps, mid, mexps, res, s);
      } else {
#define CALL(N)                                                                                   \
  launch_pdl(deriv ? fx::k_adv_a<N, true> : fx::k_adv_a<N, false>, dim3(groups, N2, nf),           \
             dim3(fx::kColThreads), 0, s, nxh, pitch, n_f, f0, eS, m->fac,             \
             (const fx::c64*)spec, exps, fa.fxwy, mid, mexps);                                       \
  launch_pdl(fx::k_adv_b<N>, dim3(groups, N2, nf), dim3(fx::kColThreads), 0, s, nxh, pitch,          \
             (const fx::c64*)mid, (const int*)mexps, fa.fxwy, res)
        FC2D_N2(fa.ny, CALL)
#undef CALL
      }
    }
    ProfScope ps(p, "inverse_rows", s);
    double* dst = off ? out + f0 : out + (size_t)f0 * fa.nx * fa.ny;
    const fc2d_grid& gr = p->grid;
    if (!launch_inverse_rows_fx(fa, nf, res, nullptr, gr.a0, gr.b0, gr.h, dst, off, points, n_f, s))
      launch_inverse_rows_mixed(fa, nf, res, nullptr, gr.a0, gr.b0, gr.h, dst, off, points, n_f, s);
  }
  return FC2D_OK;
}

}  // namespace fc2d
