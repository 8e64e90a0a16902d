// Strip values of double plans in fixed point (fx.cuh): the blend A_r c (eq. (2.6), Remark
// 2.2) and the interpolation onto the strip points (Section 3.4).
//
// Both are sums of products, 5 per fine point of every normal and 72 per strip point at
// M = 8, which FP64 issues at 2 per clock and SM.  Here the matching values and Gram
// coefficients stay FP64 (a few per normal); a normal's coefficients then share one exponent,
// its strip values are integers in that unit, and every product is three 32 x 32 -> 64 bit
// multiply-adds.  A_r is scaled column by column (its columns grow by orders of magnitude;
// the coefficients take the inverse powers of two), weights carry 56 bits or more.
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

// A running sum of products a b, exact but for the last 32 bits: (hi + mid 2^-32) 2^64.
struct Sum {
  i64 hi = 0, mid = 0;
  __device__ __forceinline__ void add(i64 a, int2 b) {
    const int h = hi32(a), l = lo32(a);
    hi = mad(h, b.x, hi);
    mid = mad(h, b.y, mad(l, b.x, add_high(mad(l, b.y, 0), mid)));
  }
  // the sum times 2^(k - 64), rounded, -8 <= k <= 31
  __device__ __forceinline__ i64 value(int k) const {
    if (k <= 0) return (add_high(mid, hi) + ((1ll << -k) >> 1)) >> -k;
    return (hi << k) + ((mid + (1ll << (31 - k))) >> (32 - k));
  }
};

// shift left by n (n < 0: right, rounded; -63 <= n)
__device__ __forceinline__ i64 shift(i64 v, int n) {
  return n >= 0 ? v << n : (v + (i64)((1ull << -n) >> 1)) >> -n;
}

// As k_gather_blend (extend.cu), a group of GS lanes per normal, up to the Gram coefficients;
// then the whole warp blends its 32/GS normals one after the other, every lane kBlendPoints
// fine points at once.  A normal's values are scaled to below 2^58 by their largest one.
// (With the group blending its own normal in two sweeps, the kernel took 51 us for 8192
// normals, a third of it waiting on A_r.)
constexpr int kBlendPoints = 6, kBlendThreads = 64;
template <int GS>
__global__ void __launch_bounds__(kBlendThreads) k_gather_blend_fx(GatherArgs a, StripFx x) {
  const int lane = threadIdx.x & 31;
  const int s = lane & (GS - 1), g0 = lane & ~(GS - 1);
  const int warp = (blockIdx.x * blockDim.x + threadIdx.x) >> 5;
  const int f = blockIdx.y;
  const int p = warp * (32 / GS) + lane / GS;
  const int pp = p < a.B ? p : 0;
  const int M = a.M, d = a.d, NS = M - 1, nq = a.nq;
  const double* fg = a.f_grid + (size_t)f * a.grid_stride;
  const double* fb = a.f_bdry ? a.f_bdry + (size_t)f * a.n_bdry : nullptr;
  pdl_wait();
  pdl_trigger();
  double star = 0.0;
  if (s < NS) {
    const int32_t* gi = a.gidx + ((size_t)pp * NS + s) * M;
    const double* gw = a.gw + ((size_t)pp * NS + s) * M;
    for (int e = 0; e < M; ++e) {
      const int32_t id = __ldg(gi + e);
      star = fma(__ldg(gw + e), id >= 0 ? __ldg(fg + id) : __ldg(fb + (-1 - id)), star);
    }
  }
  const double fbp = fb ? __ldg(fb + pp) : 0.0;
  const double* wn = a.wn + ((size_t)pp * nq + (s < nq ? s : 0)) * M;
  double acc = (s < nq) ? __ldg(wn) * fbp : 0.0;
  for (int e = 1; e < M; ++e) {
    const double v = __shfl_sync(0xffffffffu, star, g0 + e - 1);
    if (s < nq) acc = fma(__ldg(wn + e), v, acc);
  }
  const double fD = s < nq ? acc : (s == d - 1 ? fbp : 0.0);
  // the value at the foot: the boundary datum, or its extrapolation (interior data)
  const double f0 = __shfl_sync(0xffffffffu, fD, g0 + d - 1);
  double cs = 0.0;  // Gram coefficient c_s (lanes s < d)
  for (int i = 0; i < d; ++i) {
    const double v = __shfl_sync(0xffffffffu, fD, g0 + i);
    if (s < d) cs = fma(__ldg(a.Q + i * d + s), v, cs);
  }
  // the common exponent of c_j 2^Aexp_j and f0
  const int ae = s < d ? __ldg(x.Aexp + s) : 0;
  const int ec = (int)(magnitude(cs) >> 20), e0 = (int)(magnitude(f0) >> 20);
  int E = max(s < d ? max(ec, 1) + ae : 1, max(e0, 1));
  bool bad = (s < d && ec == 0x7FF) || e0 == 0x7FF;
#pragma unroll
  for (int o = GS / 2; o; o >>= 1) {
    E = max(E, __shfl_xor_sync(0xffffffffu, E, o));
    bad = __shfl_xor_sync(0xffffffffu, (int)bad, o) || bad;
  }
  // c_j 2^Aexp_j in units of 2^(E - 1081), below 2^59; the blend in units of 2^(E - 1077)
  const i64 ci = s < d ? from_double<6>(cs, E - ae) : 0;
  const i64 v0 = from_double<6>(f0, E);
  const int sweep = 32 * kBlendPoints, rounds = (a.Cr + sweep - 1) / sweep;
#pragma unroll 1
  for (int i = 0; i < 32 / GS; ++i) {
    const int pn = warp * (32 / GS) + i, src = i * GS;
    if (pn >= a.B) break;  // the same in every lane
    const i64 w0 = __shfl_sync(0xffffffffu, v0, src);
    const int En = __shfl_sync(0xffffffffu, E, src);
    const bool badn = __shfl_sync(0xffffffffu, (int)bad, src);
    Sum v[kBlendPoints];
    auto blend = [&](int r) {
#pragma unroll
      for (int u = 0; u < kBlendPoints; ++u) v[u] = Sum();
      for (int j = 0; j < d; ++j) {
        const i64 c = __shfl_sync(0xffffffffu, ci, src + j);
        const int2* col = x.Ar + j * a.Cr + r * sweep + lane;
#pragma unroll
        for (int u = 0; u < kBlendPoints; ++u)
          if (r * sweep + u * 32 + lane < a.Cr) v[u].add(c, __ldg(col + u * 32));
      }
    };
    unsigned h = spread(w0 >> kDrop);
    for (int r = 0; r < rounds; ++r) {
      blend(r);
#pragma unroll
      for (int u = 0; u < kBlendPoints; ++u) h |= spread(v[u].value(0));
    }
    h = __reduce_or_sync(0xffffffffu, h);
    const int k = min(headroom(h) - 4, 24);
    i64* F = x.F + ((size_t)f * a.B + pn) * (a.Cr + 1);
    if (lane == 0) {
      F[0] = shift(w0, k - kDrop);
      x.exps[(size_t)f * a.B + pn] = badn ? kNaN : En - 1077 - k;
    }
    for (int r = 0; r < rounds; ++r) {
      if (rounds > 1) blend(r);
#pragma unroll
      for (int u = 0; u < kBlendPoints; ++u) {
        const int q = r * sweep + u * 32 + lane;
        if (q < a.Cr) F[q + 1] = v[u].value(k);
      }
    }
  }
}

// As k_interp: one thread per (strip point, function).  |F| < 2^58, the weights along the
// normal are w 2^(60 - gain) and add up to less than 2^gain: their sums, times 2^(1 - gain),
// stay below 2^59; the weights across the normals (central: below 1, adding up to less than
// 4) are w 2^60.
template <int MM>
__global__ void __launch_bounds__(256) k_interp_fx(InterpArgs a, const int2* __restrict__ w,
                                                   const i64* __restrict__ F, const int* __restrict__ exps,
                                                   double* __restrict__ vals) {
  const int n = blockIdx.x * blockDim.x + threadIdx.x, f = blockIdx.y;
  const int M = MM > 0 ? MM : a.M, ns = a.n_strip, B = a.B, ld = a.ldF;
  if (n >= ns) return;
  int2 eta[MM > 0 ? MM : kMaxM], th[MM > 0 ? MM : kMaxM];
#pragma unroll
  for (int b = 0; b < (MM > 0 ? MM : kMaxM); ++b)
    if (b < M) {
      eta[b] = __ldg(w + (size_t)(M + b) * ns + n);
      th[b] = __ldg(w + (size_t)b * ns + n);
    }
  const int pb = __ldg(a.pb + n), s = __ldg(a.sb + n);
  pdl_wait();
  pdl_trigger();
  const i64* Ff = F + (size_t)f * B * ld + s;
  const int* ef = exps + (size_t)f * B;
  int er[MM > 0 ? MM : kMaxM], e = -(1 << 30);
#pragma unroll
  for (int i = 0; i < (MM > 0 ? MM : kMaxM); ++i)
    if (i < M) {
      int pr = pb + i;
      pr = pr < 0 ? pr + B : (pr >= B ? pr - B : pr);
      er[i] = ef[pr];
      e = max(e, er[i]);
    }
  Sum out;
#pragma unroll
  for (int i = 0; i < (MM > 0 ? MM : kMaxM); ++i) {
    if (i >= M) break;
    int pr = pb + i;
    pr = pr < 0 ? pr + B : (pr >= B ? pr - B : pr);
    const i64* row = Ff + (size_t)pr * ld;
    Sum v;
#pragma unroll
    for (int b = 0; b < (MM > 0 ? MM : kMaxM); ++b)
      if (b < M) v.add(row[b], eta[b]);
    out.add(shift(v.value(kDrop + 1), -min(e - er[i], 63)), th[i]);
  }
  const int eo = e + strip_gain(M) - 2;  // the last sum times 2
  vals[(size_t)f * ns + n] = to_double(out.value(kDrop + 1), eo, plain_exp(eo));
}

// the weights as limbs: across the normals (the first half) w 2^60, along them w 2^(60 - gain)
__global__ void k_weight_limbs(int64_t n, int gain, const double* __restrict__ w, int2* __restrict__ out) {
  const int64_t i = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
  if (i >= n) return;
  const i64 v = __double2ll_rn(ldexp(w[i], 2 * i < n ? 60 : 60 - gain));
  out[i] = {hi32(v), lo32(v)};
}

}  // namespace fx

void launch_gather_blend_fx(const GatherArgs& a, const StripFx& x, int n_f, cudaStream_t s) {
  const int GS = (a.M - 1 <= 8 && a.d <= 8) ? 8 : 16;
  const int per_warp = 32 / GS, warps = (a.B + per_warp - 1) / per_warp;
  const dim3 grid((warps * 32 + fx::kBlendThreads - 1) / fx::kBlendThreads, n_f);
  launch_pdl(GS == 8 ? fx::k_gather_blend_fx<8> : fx::k_gather_blend_fx<16>, grid, dim3(fx::kBlendThreads), 0, s, a, x);
}

void launch_interp_fx(const InterpArgs& a, const StripFx& x, int n_f, double* vals, cudaStream_t s) {
  if (a.n_strip == 0) return;
  const dim3 grid((a.n_strip + 255) / 256, n_f);
  auto k = a.M == 8 ? fx::k_interp_fx<8> : a.M == 7 ? fx::k_interp_fx<7> : fx::k_interp_fx<0>;
  launch_pdl(k, grid, dim3(256), 0, s, a, x.w, (const long long*)x.F, (const int*)x.exps, vals);
}

// A_r and the weights (already on the device as doubles) as limbs
fc2d_status strip_fx_plan(fc2d_plan_s* p) {
  const int d = p->prm.d, Cr = p->Cr, M = p->prm.M;
  const int64_t nw = (int64_t)p->strip_lin.size() * 2 * M;
  std::vector<int2> ar((size_t)d * Cr);
  std::vector<int> ae(d);
  for (int j = 0; j < d; ++j) {
    double top = 0.0;
    for (int q = 0; q < Cr; ++q) top = std::max(top, std::fabs(p->Ar[(size_t)q * d + j]));
    std::frexp(top, &ae[j]);
    for (int q = 0; q < Cr; ++q) {
      const int64_t v = (int64_t)std::nearbyint(std::ldexp(p->Ar[(size_t)q * d + j], 60 - ae[j]));
      const int32_t l = (int32_t)(uint32_t)(uint64_t)v;
      ar[(size_t)j * Cr + q] = {(int)((v - l) >> 32), l};
    }
  }
  if (cudaMalloc(&p->dev.fx_Ar, ar.size() * sizeof(int2)) != cudaSuccess ||
      cudaMalloc(&p->dev.fx_Aexp, d * sizeof(int)) != cudaSuccess ||
      cudaMalloc(&p->dev.fx_w, std::max<int64_t>(1, nw) * sizeof(int2)) != cudaSuccess)
    return set_error(FC2D_ERR_NOMEM, "cudaMalloc of a plan table failed");
  if (cudaMemcpy(p->dev.fx_Ar, ar.data(), ar.size() * sizeof(int2), cudaMemcpyHostToDevice) != cudaSuccess ||
      cudaMemcpy(p->dev.fx_Aexp, ae.data(), d * sizeof(int), cudaMemcpyHostToDevice) != cudaSuccess)
    return set_error(FC2D_ERR_CUDA, "cudaMemcpy of a plan table failed");
  if (nw == 0) return FC2D_OK;
  fx::k_weight_limbs<<<(unsigned)((nw + 255) / 256), 256>>>(nw, strip_gain(M), (const double*)p->dev.s_w,
                                                           p->dev.fx_w);
  return cuda_check(cudaDeviceSynchronize(), "interpolation weights");
}

}  // namespace fc2d
