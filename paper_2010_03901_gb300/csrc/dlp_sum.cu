// Trapezoidal sums of the double-layer potential over the partition of dlp_tree.h.
//
// k_node_coef: the nodes' coefficients q_k and their largest magnitude.  k_dlp_expand: one
// warp per (box, up to 128 nodes): A_j = sum_k q_k w_k^(j+1), w_k = R0/(z_k - c), in 64-bit
// fixed point; the warps of a box add up by integer atomics (exact in any order).
// k_dlp_eval: one block per (leaf, up to 64 points): Horner's rule for each expansion of
// the leaf's chain, then the near nodes term by term in double-float arithmetic.
//
// The star r = 1 + 0.3 cos 5t at 1024^2 with 1024 nodes (8192 refined): far points 1765 us
// term by term (3.5e8 terms of 115 FP32 instructions, bound by their issue), 86 us so; the
// near band and the close points' sums 5300 and 250 us.  A complex product of 64-bit values
// is 12 integer multiply-adds (58 per clock and SM) and about 20 other instructions, where
// its four FP64 multiply-adds cost 256 issue slots.  The expansions are bound by the
// multiply-adds at 38% issue (168 registers for the 32 accumulators: 12 warps per SM), the
// evaluation at 44 to 51%.  Error against long double sums: 6e-16 to 1.2e-15 of the sum of the
// terms' moduli.
#include <cuda_runtime.h>

#include <cstdint>

#include "dfl.cuh"
#include "dlp_sum.h"
#include "fx.cuh"

namespace fc2d {

using namespace fx;

namespace {

constexpr int P = kDlpOrder;
static_assert(P == 32, "one coefficient per lane");
// From coefficient W on 32 bits do: |(z - c)/R0|^W <= 2^-34.7 scales their rounding (the errors
// measured against long double sums are the same as with 64 bits throughout).  At 1024^2 the
// near band takes 289 us for W = 20, 303 for 24, 327 for 32.
constexpr int W = 20;
constexpr int kUp = 8;    // q in units of 2^(E - 1075 - kUp): |Re|, |Im| < 2^61
constexpr int kFac = 61;  // factors w, t (at most 1) times 2^kFac

// factor limbs; the lowest bit is set so that no low limb is -2^31 (it is negated below)
__device__ __forceinline__ int4 limbs(c64 w) {
  w.x |= 1;
  w.y |= 1;
  return {hi32(w.x), lo32(w.x), hi32(w.y), lo32(w.y)};
}
// a w for |a| <= 2^61.5, |w| <= 1, w given as the limbs of w 2^kFac (products of the low
// limbs, at most 2 units, are left out)
__device__ __forceinline__ c64 mulf(c64 a, int4 w) {
  constexpr int D = 64 - kFac;
  const int xh = hi32(a.x), xl = lo32(a.x), yh = hi32(a.y), yl = lo32(a.y);
  const i64 half = i64(1) << (31 - D);
  const int nh = -w.z, nl = -w.w;
  const i64 mx = mad(xh, w.y, mad(xl, w.x, mad(yh, nl, mad(yl, nh, half))));
  const i64 my = mad(xh, w.w, mad(xl, w.z, mad(yh, w.y, mad(yl, w.x, half))));
  const i64 hx = mad(xh, w.x, mad(yh, nh, 0)), hy = mad(xh, w.z, mad(yh, w.x, 0));
  return {(i64)((unsigned long long)hx << D) + (mx >> (32 - D)),
          (i64)((unsigned long long)hy << D) + (my >> (32 - D))};
}

// v 2^-N as 32 bits, and the product of such a value with a factor w 2^30
template <int N> __device__ __forceinline__ int narrow(i64 v) {
  return (int)((v + (i64(1) << (N - 1))) >> N);
}
__device__ __forceinline__ void mul30(int& x, int& y, int wx, int wy) {
  const i64 px = mad(x, wx, mad(y, -wy, 1 << 29)), py = mad(x, wy, mad(y, wx, 1 << 29));
  x = (int)(px >> 30);
  y = (int)(py >> 30);
}

// v/m for a box's m: v times its reciprocal
__device__ __forceinline__ i64 over(i64 v, i64 inv) {
  return (i64)((unsigned long long)mulh(v, inv) << 2);
}

// R0/d 2^kFac for d = x 2^-shift: the float reciprocal (about 2^-20), two Newton steps
__device__ __forceinline__ c64 inverse(c64 x, const DlpBox& b, int shift) {
  const int lr = b.lr;
  const float dx = (float)(int)(x.x >> 32), dy = (float)(int)(x.y >> 32);
  // x 2^-32 = d 2^(shift - 32)
  const float s = __frcp_rn(fmaf(dx, dx, dy * dy)) * (float)b.one * exp2f((float)(kFac - 62));
  c64 w = {(i64)__float2int_rn(dx * s) << 30, -((i64)__float2int_rn(dy * s) << 30)};
  const int up = kFac - lr - shift;
#pragma unroll
  for (int it = 0; it < 2; ++it) {
    const int4 l = limbs(w);
    const c64 p = mulf(x, l);                           // R0 (1 - e)
    const c64 c = mulf(c64{b.one - p.x, -p.y}, l);      // e R0 w, in the unit of x
    w = {w.x + over(c.x << up, b.inv), w.y + over(c.y << up, b.inv)};
  }
  return w;
}

__global__ void __launch_bounds__(256) k_node_coef(int N, const double* x1, const double* y1,
                                                   const double* phi, double2* q, float4* ab,
                                                   unsigned* mag) {
  const int k = blockIdx.x * blockDim.x + threadIdx.x;
  unsigned m = 0;
  if (k < N) {
    const double a = y1[k] * phi[k] / N, b = x1[k] * phi[k] / N;
    q[k] = double2{b, a};
    float4 c;
    split_df(a, c.x, c.y);
    split_df(b, c.z, c.w);
    ab[k] = c;
    m = max(magnitude(a), magnitude(b));
  }
  block_max(m, mag);
}

// sums of a[0 .. 2 H) over the lanes, halving the number of values in each step: lane j of 32
// ends with the sums 2 j and 2 j + 1 in a[0], a[1]
template <int H> __device__ __forceinline__ void fold(i64* a, int lane) {
  const bool up = lane & (H / 2);
#pragma unroll
  for (int i = 0; i < H; ++i) {
    const i64 send = up ? a[i] : a[i + H], keep = up ? a[i + H] : a[i];
    a[i] = keep + __shfl_xor_sync(0xFFFFFFFFu, send, H / 2);
  }
  if constexpr (H > 2) fold<H / 2>(a, lane);
}

__global__ void __launch_bounds__(128, 3) k_dlp_expand(int n_spans, const DlpSpan* spans,
                                                    const DlpBox* boxes, const c64* pos, int shift,
                                                    const double2* q, const unsigned* mag,
                                                    unsigned long long* coef) {
  const int item = blockIdx.x * 4 + (threadIdx.x >> 5), lane = threadIdx.x & 31;
  if (item >= n_spans) return;  // a whole warp
  const DlpSpan sp = spans[item];
  const DlpBox b = boxes[sp.box];
  const int E = block_exp(*mag);
  const i64 half = b.hb ? i64(1) << (b.hb - 1) : 0;
  i64 a[2 * P];
  int n[2 * (P - W)];
#pragma unroll
  for (int j = 0; j < 2 * W; ++j) a[j] = 0;
#pragma unroll
  for (int j = 0; j < 2 * (P - W); ++j) n[j] = 0;
  for (int k = sp.k0 + lane; k < sp.k0 + sp.n; k += 32) {
    const c64 z = pos[k];
    const c64 wi = inverse(c64{z.x - b.cx, z.y - b.cy}, b, shift);
    const int4 w = limbs(wi);
    c64 g = mulf(from_double<kUp>(q[k], E), w);
    g = {(g.x + half) >> b.hb, (g.y + half) >> b.hb};
#pragma unroll
    for (int j = 0; j < W; ++j) {
      a[2 * j] += g.x;
      a[2 * j + 1] += g.y;
      if (j + 1 < P) g = mulf(g, w);
    }
    int gx = narrow<32>(g.x), gy = narrow<32>(g.y);
    const int wx = narrow<kFac - 30>(wi.x), wy = narrow<kFac - 30>(wi.y);
#pragma unroll
    for (int j = W; j < P; ++j) {
      n[2 * (j - W)] += gx;
      n[2 * (j - W) + 1] += gy;
      mul30(gx, gy, wx, wy);
    }
  }
#pragma unroll
  for (int j = 2 * W; j < 2 * P; ++j) a[j] = (i64)n[j - 2 * W] << 32;
  fold<P>(a, lane);  // lane j holds A_j
  unsigned long long* dst = coef + (size_t)sp.box * 2 * P + 2 * lane;
  atomicAdd(dst, (unsigned long long)a[0]);
  atomicAdd(dst + 1, (unsigned long long)a[1]);
}

// fixed-point coordinate -> integer part and fraction
__device__ __forceinline__ void cell(i64 X, int shift, float& n, float& fh, float& fl) {
  n = (float)(int)(X >> shift);
  split_df(scalbn((double)(X & ((i64(1) << shift) - 1)), -shift), fh, fl);
}

// GRID: the points are grid points lin[] and u[lin] += v/h; otherwise the points pts[] and
// out[p] = v/h
template <bool GRID>
__global__ void __launch_bounds__(kDlpPoints) k_dlp_eval(
    const DlpItem* items, const DlpLeaf* leaves, const int32_t* chain, const DlpSpan* near,
    const DlpBox* boxes, const c64* coef, int shift, const unsigned* mag, const int32_t* lin,
    int nx, const c64* pts, const int32_t* idx, double inv_h, const float4* pos, const float4* ab,
    double* out) {
  constexpr int T = kDlpPoints;
  __shared__ c64 A[P];
  __shared__ float4 s0[T], sc[T];
  __shared__ float2 s1[T];
  const DlpItem it = items[blockIdx.x];
  const DlpLeaf lf = leaves[it.leaf];
  const int t = threadIdx.x, p = it.p0 + min(t, it.n - 1);
  c64 X;
  int l;
  if (GRID) {
    l = lin[p];
    X = {(i64)(l % nx) << shift, (i64)(l / nx) << shift};
  } else {
    l = idx[p];
    X = pts[p];
  }
  const unsigned m = *mag;
  const int e0 = m >= 0x7FF00000u ? kNaN : block_exp(m) - 1075 - kUp;
  double v = 0.0;
  for (int c = 0; c < lf.nc; ++c) {
    const int box = chain[lf.c0 + c];
    if (c) __syncthreads();
    if (t < P) A[t] = coef[(size_t)box * P + t];
    const DlpBox b = boxes[box];
    __syncthreads();
    const int up = kFac - shift - b.lr;
    const c64 zi = {over((i64)((unsigned long long)(X.x - b.cx) << up), b.inv),
                    over((i64)((unsigned long long)(X.y - b.cy) << up), b.inv)};
    const int4 z = limbs(zi);
    c64 s;
    {
      const int zx = narrow<kFac - 30>(zi.x), zy = narrow<kFac - 30>(zi.y);
      int sx = (int)(A[P - 1].x >> 32), sy = (int)(A[P - 1].y >> 32);
#pragma unroll
      for (int j = P - 2; j >= W; --j) {
        mul30(sx, sy, zx, zy);
        sx += (int)(A[j].x >> 32);
        sy += (int)(A[j].y >> 32);
      }
      s = A[W - 1] + mulf(c64{(i64)sx << 32, (i64)sy << 32}, z);
    }
#pragma unroll 8
    for (int j = W - 2; j >= 0; --j) s = A[j] + mulf(s, z);
    const int e = e0 + b.hb - b.lr;
    v -= to_double(s.y, e, plain_exp(e)) * b.rm;
  }
  float px, pfh, pfl, py, qfh, qfl;
  if (GRID) {
    px = (float)(l % nx);
    py = (float)(l / nx);
  } else {
    cell(X.x, shift, px, pfh, pfl);
    cell(X.y, shift, py, qfh, qfl);
  }
  // three floats: a pair would round at 2^-48 of the sum so far with every term, and the close
  // points' Lagrange weights multiply that by several hundred
  float sh = 0.f, sl = 0.f, sr = 0.f;
  for (int d = 0; d < lf.nd; ++d) {
    const DlpSpan sp = near[lf.d0 + d];
    for (int k0 = sp.k0; k0 < sp.k0 + sp.n; k0 += T) {
      const int cnt = min(T, sp.k0 + sp.n - k0);
      __syncthreads();
      if (t < cnt) {
        s0[t] = pos[2 * (k0 + t)];
        const float4 y = pos[2 * (k0 + t) + 1];
        s1[t] = float2{y.x, y.y};
        sc[t] = ab[k0 + t];
      }
      __syncthreads();
      for (int k = 0; k < cnt; ++k) {
        const float4 a = s0[k], c = sc[k];
        const float2 b = s1[k];
        // (point - node) = (i_p - i_n) + (f_p - f_n)
        dfl dx = int_minus(px - a.x, a.z, a.w), dy = int_minus(py - a.y, b.x, b.y);
        if (!GRID) {
          dx = df_add(dx, {pfh, pfl});
          dy = df_add(dy, {qfh, qfl});
        }
        const dfl term = dl_term(dx, dy, c.x, c.y, c.z, c.w);
        const dfl s = two_sum(sh, term.hi), a1 = two_sum(sl, s.lo), a2 = two_sum(a1.hi, term.lo);
        sh = s.hi;
        sl = a2.hi;
        sr += a1.lo + a2.lo;
      }
    }
  }
  if (t >= it.n) return;
  v += (double)sh + ((double)sl + (double)sr);
  if (GRID) out[l] += v * inv_h;
  else out[l] = v * inv_h;
}

// Close points, a warp each: Re sum_k c_k z^k over the Hermitian half of the coefficients, lane l taking k = l, l + 32, .. by Horner's
// rule in z^32 and a last factor z^l; then the Lagrange combination along the normal.  In
// fixed point: 45 instructions per term and no sincos per lane, 35 us for the 7500 points of a
// star at 1024^2 (with an FP64 sincos per thread and the transform of the boundary values by a
// thread per frequency, 335 us).
__global__ void __launch_bounds__(128) k_close(int n_pts, const int32_t* lin, const double2* z,
                                               const double* w, int MP, const double* vals, int Nb,
                                               const double2* ghat, const unsigned* mag,
                                               double* u) {
  const int n = (blockIdx.x * blockDim.x + threadIdx.x) >> 5, lane = threadIdx.x & 31;
  if (n >= n_pts) return;
  const int half = Nb / 2, terms = half / 32 + 1;
  const unsigned m = *mag;
  // a lane's sum, of up to 2^(E' - E) terms below 2^60.5, stays below that
  const int E = block_exp(m) + (32 - __clz(terms - 1));
  const int e = m >= 0x7FF00000u ? kNaN : E - 1075 - kUp + 1;
  const double2 zd = z[n];
  const double one = scalbn(1.0, kFac);
  c64 p = {__double2ll_rn(zd.x * one), __double2ll_rn(zd.y * one)}, zl = {i64(1) << kFac, 0};
#pragma unroll
  for (int bit = 1; bit < 32; bit *= 2) {  // zl = z^lane, p = z^32
    const int4 l = limbs(p);
    const c64 t = mulf(zl, l);
    if (lane & bit) zl = t;
    p = mulf(p, l);
  }
  const int4 zp = limbs(p);
  c64 s = {0, 0};
  for (int i = terms - 1; i >= 0; --i) {
    const int k = lane + 32 * i;
    s = mulf(s, zp);
    if (k <= half) {
      const c64 c = from_double<kUp - 1>(ghat[k], E);
      s = s + c;
    }
  }
  s = mulf(s, limbs(zl));
  double v = to_double(s.x, e, plain_exp(e));
  for (int o = 16; o; o >>= 1) v += __shfl_xor_sync(0xFFFFFFFFu, v, o);
  v *= w[(size_t)n * MP];
  double q = 0.0;
  for (int j = 1 + lane; j < MP; j += 32)
    q = fma(w[(size_t)n * MP + j], vals[(size_t)n * (MP - 1) + j - 1], q);
  for (int o = 16; o; o >>= 1) q += __shfl_xor_sync(0xFFFFFFFFu, q, o);
  if (lane == 0) u[lin[n]] += v + q;
}

}  // namespace

void launch_close(int n, const int32_t* lin, const double2* z, const double* w, int MP,
                  const double* vals, int Nb, const double2* ghat, const unsigned* mag, double* u,
                  cudaStream_t s) {
  k_close<<<(unsigned)((n + 3) / 4), 128, 0, s>>>(n, lin, z, w, MP, vals, Nb, ghat, mag, u);
}

void launch_node_coef(int N, const double* x1, const double* y1, const double* phi, double2* q,
                      float4* ab, unsigned* mag, cudaStream_t s) {
  k_node_coef<<<(unsigned)((N + 255) / 256), 256, 0, s>>>(N, x1, y1, phi, q, ab, mag);
}

void launch_dlp_expand(const DlpDev& d, const double2* q, cudaStream_t s) {
  if (d.n_expand)
    k_dlp_expand<<<(unsigned)((d.n_expand + 3) / 4), 128, 0, s>>>(
        d.n_expand, d.expand, d.box, (const c64*)d.nodes, d.shift, q, d.mag, d.coef);
}

void launch_dlp_grid(const DlpDev& d, const int32_t* lin, int nx, double h, const float4* pos,
                     const float4* ab, double* u, cudaStream_t s) {
  if (d.n_grid)
    k_dlp_eval<true><<<(unsigned)d.n_grid, kDlpPoints, 0, s>>>(
        d.grid_items, d.leaf, d.chain, d.near, d.box, (const c64*)d.coef, d.shift, d.mag, lin, nx,
        nullptr, nullptr, 1.0 / h, pos, ab, u);
}

void launch_dlp_free(const DlpDev& d, double h, const float4* pos, const float4* ab, double* out,
                     cudaStream_t s) {
  if (d.n_free)
    k_dlp_eval<false><<<(unsigned)d.n_free, kDlpPoints, 0, s>>>(
        d.free_items, d.leaf, d.chain, d.near, d.box, (const c64*)d.coef, d.shift, d.mag, nullptr,
        0, (const c64*)d.points, d.points_idx, 1.0 / h, pos, ab, out);
}

}  // namespace fc2d
