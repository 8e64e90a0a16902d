// Fixed-point DFTs (fx.cuh) of lengths 2^a 3^b 5^c: Stockham stages of radix 2, 3, 4, 5, 6, 8,
// 9 and 10 chosen on the host, in two shared buffers.  Columns of any length run in the two
// passes of fx.cuh with N = n1 n2 (both near sqrt N) in place of 64 N/64; a row is one block.
#pragma once
#include "fx.cuh"

namespace fc2d {
namespace fx {

// v (base + m 2^-32 + r 2^-64), |m| <= 2^31
struct Const {
  int base, m, r;
};
__device__ __forceinline__ i64 mulk(i64 v, Const k) {
  const int h = hi32(v), l = lo32(v);
  const i64 t = mad(l, k.m, mad(h, k.r, i64(1) << 31));
  return add_high(t, mad(h, k.m, k.base > 0 ? v : k.base < 0 ? -v : 0));
}
__device__ __forceinline__ i64 half(i64 v) { return (v + (i64)((unsigned long long)v >> 63)) >> 1; }

__device__ __forceinline__ void dft3(c64& v0, c64& v1, c64& v2) {
  constexpr Const s3 = {1, -575416509, -1033546850};  // sin 2 pi/3
  const c64 a = v0, s = v1 + v2, d = v1 - v2;
  const c64 m = {a.x - half(s.x), a.y - half(s.y)};
  const c64 r = {mulk(d.y, s3), -mulk(d.x, s3)};  // -i sin (v1 - v2)
  v0 = a + s;
  v1 = m + r;
  v2 = m - r;
}

__device__ __forceinline__ void dft5(c64& v0, c64& v1, c64& v2, c64& v3, c64& v4) {
  constexpr Const c1 = {0, 1327217885, -1079689717}, s1 = {1, -210210662, 581434099};    // 2 pi/5
  constexpr Const c2 = {-1, 820265763, 1079689717}, s2 = {1, -1770448860, -1429016722};  // 4 pi/5
  const c64 a = v0, s14 = v1 + v4, d14 = v1 - v4, s23 = v2 + v3, d23 = v2 - v3;
  const c64 m1 = {a.x + mulk(s14.x, c1) + mulk(s23.x, c2), a.y + mulk(s14.y, c1) + mulk(s23.y, c2)};
  const c64 m2 = {a.x + mulk(s14.x, c2) + mulk(s23.x, c1), a.y + mulk(s14.y, c2) + mulk(s23.y, c1)};
  const c64 r1 = {mulk(d14.y, s1) + mulk(d23.y, s2), -(mulk(d14.x, s1) + mulk(d23.x, s2))};
  const c64 r2 = {mulk(d14.y, s2) - mulk(d23.y, s1), -(mulk(d14.x, s2) - mulk(d23.x, s1))};
  v0 = a + (s14 + s23);
  v1 = m1 + r1;
  v4 = m1 - r1;
  v2 = m2 + r2;
  v3 = m2 - r2;
}

// a (c - i s)
__device__ __forceinline__ c64 rotate(c64 a, Const c, Const s) {
  return {mulk(a.x, c) + mulk(a.y, s), mulk(a.y, c) - mulk(a.x, s)};
}

// Forward DFT of R values, |z| <= 2^58.5 (6 = 2 x 3 and 10 = 2 x 5 by the Chinese remainder
// theorem, without twiddles; 9 = 3 x 3)
template <int R> __device__ __forceinline__ void dft_any(c64* v) {
  if constexpr (R == 3) {
    dft3(v[0], v[1], v[2]);
  } else if constexpr (R == 5) {
    dft5(v[0], v[1], v[2], v[3], v[4]);
  } else if constexpr (R == 6) {  // n = 3 n1 + 2 n2, k = 3 k1 + 4 k2 (mod 6)
    c64 a[3], b[3];
#pragma unroll
    for (int n = 0; n < 3; ++n) {
      a[n] = v[2 * n] + v[(2 * n + 3) % 6];
      b[n] = v[2 * n] - v[(2 * n + 3) % 6];
    }
    dft3(a[0], a[1], a[2]);
    dft3(b[0], b[1], b[2]);
#pragma unroll
    for (int k = 0; k < 3; ++k) {
      v[4 * k % 6] = a[k];
      v[(3 + 4 * k) % 6] = b[k];
    }
  } else if constexpr (R == 10) {  // n = 5 n1 + 2 n2, k = 5 k1 + 6 k2 (mod 10)
    c64 a[5], b[5];
#pragma unroll
    for (int n = 0; n < 5; ++n) {
      a[n] = v[2 * n] + v[(2 * n + 5) % 10];
      b[n] = v[2 * n] - v[(2 * n + 5) % 10];
    }
    dft5(a[0], a[1], a[2], a[3], a[4]);
    dft5(b[0], b[1], b[2], b[3], b[4]);
#pragma unroll
    for (int k = 0; k < 5; ++k) {
      v[6 * k % 10] = a[k];
      v[(5 + 6 * k) % 10] = b[k];
    }
  } else if constexpr (R == 9) {  // n = 3 n1 + n2, k = k1 + 3 k2
    constexpr Const c1 = {1, -1004831466, 2055326097}, s1 = {1, -1534215534, -525277859};
    constexpr Const c2 = {0, 745813244, 384242502}, s2 = {1, -65250204, 148945616};
    constexpr Const c4 = {-1, 259018221, 1855398697}, s4 = {0, 1468965330, 674223475};
#pragma unroll
    for (int n = 0; n < 3; ++n) dft3(v[n], v[3 + n], v[6 + n]);  // v[3 k1 + n2]
    v[4] = rotate(v[4], c1, s1);
    v[5] = rotate(v[5], c2, s2);
    v[7] = rotate(v[7], c2, s2);
    v[8] = rotate(v[8], c4, s4);
#pragma unroll
    for (int k = 0; k < 3; ++k) dft3(v[3 * k], v[3 * k + 1], v[3 * k + 2]);  // v[3 k1 + k2]
    c64 t = v[1];
    v[1] = v[3];
    v[3] = t;
    t = v[2];
    v[2] = v[6];
    v[6] = t;
    t = v[5];
    v[5] = v[7];
    v[7] = t;
  } else {
    dft<R>(v);
  }
}

// One Stockham stage of radix R over N values (Ns: the product of the earlier radices): the
// butterflies first, first + every, ... of this thread.  src(i): input i; dst(i, v): output;
// tw[ts t] = w_N^t; L: the left shift of the block before a stage after the first.  Returns
// the outputs' spread.
template <int R, typename Src, typename Dst>
__device__ __forceinline__ unsigned mixed_stage(int N, int Ns, int first, int every, Src src, Dst dst,
                                                const int4* __restrict__ tw, int ts, int L) {
  const int NR = N / R, step = ts * (NR / Ns);
  // quotients by Ns as (j + 1/2) (1/Ns) truncated: exact for j < 2^22 and Ns = 2^a 3^b 5^c
  const float inv = 1.0f / (float)Ns;
  unsigned h = 0;
  for (int j = first; j < NR; j += every) {
    const int q = (int)(((float)j + 0.5f) * inv), k = j - q * Ns;
    c64 v[R];
#pragma unroll
    for (int r = 0; r < R; ++r) v[r] = src(j + r * NR);
    if (Ns > 1) {
      if (L) {
#pragma unroll
        for (int r = 0; r < R; ++r) v[r] = {v[r].x << L, v[r].y << L};
      }
      v[0] = drop(v[0]);
#pragma unroll
      for (int r = 1; r < R; ++r) v[r] = mulw(v[r], __ldg(tw + r * k * step));
    }
    dft_any<R>(v);
    const int base = q * Ns * R + k;
#pragma unroll
    for (int r = 0; r < R; ++r) {
      h |= spread(v[r]);
      dst(base + r * Ns, v[r]);
    }
  }
  return h;
}

// All stages.  in(i): the inputs (|z| <= 2^58.5, in units of 2^e); stage s writes to
// store(s & 1, i, v) and the next one reads load(s & 1, i).  The block is rescaled before
// every other stage, as shifts() says (st: kMixedSlots zeroed shared words).  Every thread of the block calls it;
// on return (after a barrier) the result is in buffer (n - 1) & 1, its spread in *out_spread
// if given.
constexpr int kMixedSlots = 20;
template <Order O, typename In, typename Load, typename Store>
__device__ __forceinline__ void mixed_dft(const FxRadices& rad, int N, int first, int every, In in,
                                          Load load, Store store, const int4* __restrict__ tw, int ts,
                                          unsigned* st, int& e) {
  int Ns = 1;
  for (int s = 0; s < rad.n; ++s) {
    const int R = rad.r[s];
    int L = 0;
    if (s > 0) {
      if (shifts(s, O)) L = headroom(st[s]);
      e += kDrop - L;
    }
    auto src = [&](int i) { return s ? load((s - 1) & 1, i) : in(i); };
    auto dst = [&](int i, c64 v) { store(s & 1, i, v); };
    unsigned h = 0;
    switch (R) {
      case 2: h = mixed_stage<2>(N, Ns, first, every, src, dst, tw, ts, L); break;
      case 3: h = mixed_stage<3>(N, Ns, first, every, src, dst, tw, ts, L); break;
      case 4: h = mixed_stage<4>(N, Ns, first, every, src, dst, tw, ts, L); break;
      case 5: h = mixed_stage<5>(N, Ns, first, every, src, dst, tw, ts, L); break;
      case 6: h = mixed_stage<6>(N, Ns, first, every, src, dst, tw, ts, L); break;
      case 8: h = mixed_stage<8>(N, Ns, first, every, src, dst, tw, ts, L); break;
      case 9: h = mixed_stage<9>(N, Ns, first, every, src, dst, tw, ts, L); break;
      default: h = mixed_stage<10>(N, Ns, first, every, src, dst, tw, ts, L); break;
    }
    Ns *= R;
    block_or(h, st + s + 1);
    __syncthreads();
  }
}

}  // namespace fx
}  // namespace fc2d
