// Block fixed-point arithmetic for the double-precision transforms.
//
// GB300 issues 2 FP64 multiply-adds per clock and SM, but 128 32-bit integer additions
// and 64 32 x 32 -> 64 bit integer multiply-adds (measured: 2.0, 122 and 58).  A DFT of
// doubles therefore runs here on 64-bit integers: the values of a transform share one
// exponent (a block exponent, chosen from their largest magnitude), additions are 64-bit
// integer additions, and a product with a twiddle factor is formed from 32-bit limbs.
// The doubles enter through their bit patterns and leave through them, rounded once; no
// FP64 instruction is issued.
//
// Error: a stage keeps its values within 2^62 of a unit and rounds to that unit after each
// twiddle product, whose result is at most 2^58.5: an error of 2^-58 of the block's
// largest value per stage, where FP64 rounds every operation to 2^-53 of its own result.
// Between stages the block is shifted left by the bits that its largest value leaves
// unused, so the unit follows the data.  Twiddles carry 60 bits.  A transform with an
// infinity or a NaN among its inputs returns NaN everywhere.
#pragma once
#include <cuda_runtime.h>

#include <cstdint>

#include "fc2d_kernels.cuh"

namespace fc2d {
namespace fx {

using i64 = long long;

// a complex value in units of 2^e (e: the block's exponent); 16 bytes, as double2
struct __align__(16) c64 {
  i64 x, y;
};

constexpr int kScale = 60;          // twiddles are w 2^60, in balanced 32-bit limbs
constexpr int kDrop = 64 - kScale;  // a product with a twiddle is scaled by 2^-kDrop
constexpr int kNaN = 1 << 20;       // block exponent of a transform with non-finite input

__device__ __forceinline__ c64 operator+(c64 a, c64 b) { return {a.x + b.x, a.y + b.y}; }
__device__ __forceinline__ c64 operator-(c64 a, c64 b) { return {a.x - b.x, a.y - b.y}; }
__device__ __forceinline__ c64 mul_mi(c64 a) { return {a.y, -a.x}; }  // -i a

// v = h 2^32 + l with l in [-2^31, 2^31)
__device__ __forceinline__ int lo32(i64 v) { return (int)v; }
__device__ __forceinline__ int hi32(i64 v) { return (int)((unsigned)(v >> 32) + ((unsigned)v >> 31)); }

__device__ __forceinline__ i64 mad(int a, int b, i64 c) {  // one instruction
  i64 d;
  asm("mad.wide.s32 %0, %1, %2, %3;" : "=l"(d) : "r"(a), "r"(b), "l"(c));
  return d;
}
// c + (v >> 32) as one multiply-add by a 1 that the compiler cannot see (a shift, a sign
// word and a 64-bit addition otherwise)
__constant__ int kOne = 1;
__device__ __forceinline__ i64 add_high(i64 v, i64 c) { return mad((int)(v >> 32), kOne, c); }

// a w 2^-kDrop for |a.x|, |a.y| <= 2^62.5: the products of the high limbs, plus the mixed
// products rounded at bit 32 (each sum of mixed products stays below 2^63); the products
// of the low limbs are below half a unit and are left out.  w = (re hi, re lo, im hi, im lo)
__device__ __forceinline__ c64 mulw(c64 a, int4 w) {
  const int xh = hi32(a.x), xl = lo32(a.x), yh = hi32(a.y), yl = lo32(a.y);
  const i64 half = i64(1) << 31;
  const int nh = -w.z, nl = -w.w;  // limbs are never -2^31
  const i64 mx = mad(xh, w.y, mad(xl, w.x, mad(yh, nl, mad(yl, nh, half))));
  const i64 my = mad(xh, w.w, mad(xl, w.z, mad(yh, w.y, mad(yl, w.x, half))));
  return {mad(xh, w.x, mad(yh, nh, add_high(mx, 0))), mad(xh, w.z, mad(yh, w.x, add_high(my, 0)))};
}

// a conj(w) 2^-kDrop
__device__ __forceinline__ c64 mulw_conj(c64 a, int4 w) { return mulw(a, int4{w.x, w.y, -w.z, -w.w}); }

// (a p + b q) 2^-kDrop for real factors p, q (limbs of p 2^60, q 2^60), |a|, |b| <= 2^62
__device__ __forceinline__ i64 dot(i64 a, i64 b, int4 pq) {
  const int ah = hi32(a), al = lo32(a), bh = hi32(b), bl = lo32(b);
  const i64 m = mad(ah, pq.y, mad(al, pq.x, mad(bh, pq.w, mad(bl, pq.z, i64(1) << 31))));
  return mad(ah, pq.x, mad(bh, pq.z, add_high(m, 0)));
}
// a p + b q = (hi + mid 2^-32) 2^64 up to 2^-32 (dot() rounds it to hi + (mid >> 32))
struct Wide {
  i64 hi, mid;
};
__device__ __forceinline__ Wide dot_wide(i64 a, i64 b, int4 pq) {
  const int ah = hi32(a), al = lo32(a), bh = hi32(b), bl = lo32(b);
  const i64 low = mad(al, pq.y, mad(bl, pq.w, 0));
  const i64 m = mad(ah, pq.y, mad(al, pq.x, mad(bh, pq.w, mad(bl, pq.z, low >> 32))));
  return {mad(ah, pq.x, mad(bh, pq.z, 0)), m};
}

// a b 2^-64, |a|, |b| <= 2^62
__device__ __forceinline__ i64 mulh(i64 a, i64 b) {
  const int ah = hi32(a), al = lo32(a), bh = hi32(b), bl = lo32(b);
  return mad(ah, bh, add_high(mad(ah, bl, mad(al, bh, i64(1) << 31)), 0));
}

// v c for a constant c in [1/2, 1) given as c - 1 = m 2^-32 + r 2^-64 (|v| < 2^62.5)
__device__ __forceinline__ i64 mulc(i64 v, int m, int r) {
  const int h = hi32(v), l = lo32(v);
  const i64 t = mad(l, m, mad(h, r, i64(1) << 31));
  return add_high(t, mad(h, m, v));
}
// sqrt(1/2) - 1 = kRtM 2^-32 + kRtR 2^-64
constexpr int kRtM = -1257966796;
constexpr int kRtR = -102865788;

// v 2^-kDrop, rounded to nearest, ties toward zero.  (Ties are frequent here; rounding them
// upward would shift a whole block by 1/32 of a unit, which the transform adds up in its
// zero frequency.  For the same reason the twiddle 1 is stored as 1 - 2^-60.)
__device__ __forceinline__ i64 drop(i64 v) {
  return (v + ((1 << (kDrop - 1)) - 1) + (i64)((unsigned long long)v >> 63)) >> kDrop;
}
__device__ __forceinline__ c64 drop(c64 v) { return {drop(v.x), drop(v.y)}; }

// X_k and X_{NH-k} (times 2^(1-kDrop), in the block's units) of a real row from its pairs'
// transform (|z| <= 2^61.5): with zk = Z_k and zl = Z_{NH-k}, e = (zk + conj zl)/2, o = (zk - conj zl)/2,
// X_k = e - i w^k o, X_{NH-k} = conj(e + i w^k o)
__device__ __forceinline__ void split_pair(c64 zk, c64 zl, int4 w, c64& xk, c64& xl) {
  const c64 e = drop(c64{zk.x + zl.x, zk.y - zl.y});
  const c64 wo = mulw(c64{zk.x - zl.x, zk.y + zl.y}, w);
  xk = {e.x + wo.y, e.y - wo.x};
  xl = {e.x - wo.y, -e.y - wo.x};
}

// bits that differ from their lower neighbour: the top one bounds |v| < 2^(32 + index)
__device__ __forceinline__ unsigned spread(i64 v) {
  const int h = (int)(v >> 32);
  return (unsigned)(h ^ (h + h));
}
__device__ __forceinline__ unsigned spread(c64 v) { return spread(v.x) | spread(v.y); }
// the left shift that brings a block with these spread bits to |v| <= 2^62
__device__ __forceinline__ int headroom(unsigned h) { return min(__clz((int)h) - 1, 30); }

// The magnitude bits of a double's high word (exponent in bits 20..30): the block maximum
// of these gives the block exponent.
__device__ __forceinline__ unsigned magnitude(double d) {
  return (unsigned)__double2hiint(d) & 0x7FFFFFFFu;
}
// x in units of 2^(E - 1075 - UP), E at least x's biased exponent: the 53-bit significand
// shifted to |v| < 2^(53 + UP) for exponent E, right by E - e bits for others
__device__ __forceinline__ i64 shift_right(i64 v, int n) {  // n >= 0; 0 from 64 on (v >= 0)
  i64 r;
  asm("shr.u64 %0, %1, %2;" : "=l"(r) : "l"(v), "r"(n));
  return r;
}
template <int UP = 5>
__device__ __forceinline__ i64 from_double(double d, int E) {
  const unsigned hi = (unsigned)__double2hiint(d);
  const int e = (int)(hi >> 20) & 0x7FF;
  unsigned mh = (hi & 0xFFFFFu) | 0x100000u;
  int sh = E - e;
  if (E <= 64 && e == 0) {  // for a larger block exponent a subnormal or zero shifts out
    mh = hi & 0xFFFFFu;
    sh = E - 1;
  }
  const i64 m = (i64)(((unsigned long long)mh << 32) | (unsigned)__double2loint(d)) << UP;
  const i64 v = shift_right(m, sh);
  const i64 s = (i64)((int)hi >> 31);
  return (v ^ s) - s;
}
template <int UP = 5>
__device__ __forceinline__ c64 from_double(double2 d, int E) {
  return {from_double<UP>(d.x, E), from_double<UP>(d.y, E)};
}
// block exponent of values converted with the block maximum mag of magnitude()
__device__ __forceinline__ int block_exp(unsigned mag) { return max((int)(mag >> 20), 1); }

// Whether every nonzero v with unit 2^e becomes a normal double (or overflows to infinity
// by its exponent field): the same for a whole block.
__device__ __forceinline__ bool plain_exp(int e) { return e + 1086 - 63 >= 1 && e + 1086 <= 2046; }
// v 2^e as a double, rounded to nearest: the conversion instruction (2 per clock and SM, on
// the FP64 pipe that is idle otherwise; the same in integer operations takes 24) and an
// addition to the exponent field
__device__ __forceinline__ double to_double(i64 v, int e, bool plain) {
  const double x = __ll2double_rn(v);
  if (plain) return __hiloint2double(__double2hiint(x) + (v ? e << 20 : 0), __double2loint(x));
  return e > kNaN / 2 ? __longlong_as_double(0x7FF8000000000000ll) : scalbn(x, e);
}
__device__ __forceinline__ double2 to_double(c64 v, int e, bool plain) {
  return {to_double(v.x, e, plain), to_double(v.y, e, plain)};
}

// ------------------------------------------------------------------------- //
// Small forward DFTs; inputs |z| <= 2^58.5 give outputs below 2^62
// ------------------------------------------------------------------------- //
__device__ __forceinline__ void dft4(c64& a0, c64& a1, c64& a2, c64& a3) {
  const c64 t0 = a0 + a2, t1 = a0 - a2, t2 = a1 + a3, t3 = mul_mi(a1 - a3);
  a0 = t0 + t2;
  a2 = t0 - t2;
  a1 = t1 + t3;
  a3 = t1 - t3;
}

template <int R> __device__ __forceinline__ void dft(c64* v) {
  if constexpr (R == 2) {
    const c64 a = v[0], b = v[1];
    v[0] = a + b;
    v[1] = a - b;
  } else if constexpr (R == 4) {
    dft4(v[0], v[1], v[2], v[3]);
  } else {
    static_assert(R == 8, "radix 2, 4 or 8");
    c64 e0 = v[0], e1 = v[2], e2 = v[4], e3 = v[6], o0 = v[1], o1 = v[3], o2 = v[5], o3 = v[7];
    dft4(e0, e1, e2, e3);
    dft4(o0, o1, o2, o3);
    const c64 w1 = {mulc(o1.x + o1.y, kRtM, kRtR), mulc(o1.y - o1.x, kRtM, kRtR)};
    const c64 w2 = mul_mi(o2);
    const c64 w3 = {mulc(o3.y - o3.x, kRtM, kRtR), mulc(-o3.x - o3.y, kRtM, kRtR)};
    v[0] = e0 + o0;
    v[4] = e0 - o0;
    v[1] = e1 + w1;
    v[5] = e1 - w1;
    v[2] = e2 + w2;
    v[6] = e2 - w2;
    v[3] = e3 + w3;
    v[7] = e3 - w3;
  }
}

// ------------------------------------------------------------------------- //
// A transform of N = 2^LOGN points by NT = N/8 threads, eight values each, on one padded
// shared buffer; Stockham stages of radix 8 (the last one N/NS).  Block statistics go
// through `st`, kSlots shared words that are zero when the transform starts: st[0] the
// largest magnitude of the inputs, st[k] the spread bits after stage k.  Every thread of
// the block takes part in the barriers and reductions.
// ------------------------------------------------------------------------- //
constexpr int kSlots = 8;
__device__ __forceinline__ int pad(int i) { return i + (i >> 3); }
__host__ __device__ constexpr int padded(int n) { return n + (n >> 3); }
// pad(i + r S) = pad(i) + r step(S) when S is a multiple of 8, or S = 1 and i of 8
template <int S> __host__ __device__ constexpr int step() { return S % 8 == 0 ? S + S / 8 : S; }

__device__ __forceinline__ void block_max(unsigned v, unsigned* slot) {
  v = __reduce_max_sync(0xFFFFFFFFu, v);
  if ((threadIdx.x & 31) == 0) atomicMax(slot, v);
}
__device__ __forceinline__ void block_or(unsigned v, unsigned* slot) {
  v = __reduce_or_sync(0xFFFFFFFFu, v);
  if ((threadIdx.x & 31) == 0) atomicOr(slot, v);
}

// Offset of the stage with sub-length NS in the per-stage twiddle table
__host__ __device__ constexpr int stage_off(int N, int NS) {
  int off = 0, ns = 1;
  while (ns < NS) {
    const int R = (N / ns >= 8) ? 8 : N / ns;
    if (ns > 1) off += R * ns;
    ns *= R;
  }
  return off;
}
template <int LOGN> __host__ __device__ constexpr int last_ns() {
  int ns = 1;
  while (true) {
    const int R = ((1 << LOGN) / ns >= 8) ? 8 : (1 << LOGN) / ns;
    if (ns * R == (1 << LOGN)) return ns;
    ns *= R;
  }
}

// Rescale and twiddle the eight inputs of a stage after the first: the first value of each
// butterfly by a shift, the others by their twiddles (tw[r NS + k]); radix-R DFTs.
template <int R, int NS, int NT, bool SHIFT>
__device__ __forceinline__ void butterflies(c64 (&v)[8], int t, const int4* __restrict__ tw, int L) {
#pragma unroll
  for (int m = 0; m < 8 / R; ++m) {
    const int k = (t + m * NT) & (NS - 1);
    c64* a = v + m * R;
    if constexpr (SHIFT) {
#pragma unroll
      for (int r = 0; r < R; ++r) a[r] = {a[r].x << L, a[r].y << L};
    }
    a[0] = drop(a[0]);
#pragma unroll
    for (int r = 1; r < R; ++r) a[r] = mulw(a[r], __ldg(tw + r * NS + k));
    dft<R>(a);
  }
}

// Whether the block is rescaled before stage k + 1 (k = 1, 2, ..): every other stage.  A
// stage that is not preceded by a shift works on values that lost at most the 3.5 bits of
// headroom of the stage before.  FORWARD: the inputs are about as large everywhere and grow in the
// first stage; shifts from the second on.  INVERSE: few modes of a spectrum are large, the first
// stage adds nothing to those, and unless the second one shifts, its products round at
// 2^-53 of the largest mode in every value at once.  Smooth fields, forward and inverse transforms: 2048^2
// 7.3e-16 -> 2.3e-16 of the 2-norm (FP64 4.4e-16), 1200 x 1728 5.8e-16 -> 1.8e-16, the same time.
enum Order { FORWARD = 0, INVERSE = 1 };
__host__ __device__ constexpr bool shifts(int k, Order o) { return k % 2 == o; }

// All stages but the first.  buf holds the outputs of the stage before (sub-length NS),
// st[SLOT] their spread.  On return v holds the thread's last-stage outputs (value r of
// butterfly m belongs at index out_index<LOGN>(t, m, r)) and e their exponent.
template <int LOGN, int NS, int SLOT, Order O>
__device__ __forceinline__ void rest(c64 (&v)[8], c64* buf, int t, bool active, unsigned* st,
                                     const int4* __restrict__ tw, int& e) {
  constexpr int N = 1 << LOGN, NT = N / 8;
  constexpr int R = N / NS >= 8 ? 8 : N / NS, NR = N / R, M = 8 / R;
  const int L = shifts(SLOT, O) ? headroom(st[SLOT]) : 0;
  e += kDrop - L;
  if (active) {
#pragma unroll
    for (int m = 0; m < M; ++m) {
      if constexpr (NR % 8 == 0) {
        const c64* src = buf + pad(t + m * NT);
#pragma unroll
        for (int r = 0; r < R; ++r) v[m * R + r] = src[r * step<NR>()];
      } else {
#pragma unroll
        for (int r = 0; r < R; ++r) v[m * R + r] = buf[pad(t + m * NT + r * NR)];
      }
    }
  }
  if constexpr (NS * R < N) __syncthreads();
  unsigned h = 0;
  if (active) {
    butterflies<R, NS, NT, shifts(SLOT, O)>(v, t, tw + stage_off(N, NS), L);
    if constexpr (NS * R < N) {  // R = 8
      const int k = t & (NS - 1);
      const int base = (t / NS) * NS * R + k;
      c64* dst = buf + pad(base);
#pragma unroll
      for (int r = 0; r < R; ++r) {
        dst[r * step<NS>()] = v[r];
        if (shifts(SLOT + 1, O)) h |= spread(v[r]);
      }
    }
  }
  if constexpr (NS * R < N) {
    if constexpr (shifts(SLOT + 1, O)) block_or(h, st + SLOT + 1);
    __syncthreads();
    rest<LOGN, NS * R, SLOT + 1, O>(v, buf, t, active, st, tw, e);
  }
}

// index of value r of the thread's last-stage butterfly m
template <int LOGN> __device__ __forceinline__ int out_index(int t, int m, int r) {
  constexpr int N = 1 << LOGN, NS = last_ns<LOGN>(), NT = N / 8;
  return t + m * NT + r * NS;  // j = t + m NT < NS: (j / NS) NS R + (j mod NS) + r NS
}
template <int LOGN> __host__ __device__ constexpr int last_radix() { return (1 << LOGN) / last_ns<LOGN>(); }

// The whole transform of the doubles u[r] = x[t + r N/8] (every thread's eight inputs are
// in registers; `buf` may have held them).  v, e: as rest().
template <int LOGN>
__device__ __forceinline__ void transform(const double2 (&u)[8], c64 (&v)[8], c64* buf, int t,
                                          bool active, unsigned* st, const int4* __restrict__ tw,
                                          int& e) {
  static_assert(LOGN >= 4, "at least two stages");
  unsigned mag = 0;
  if (active) {
#pragma unroll
    for (int r = 0; r < 8; ++r) mag = max(mag, max(magnitude(u[r].x), magnitude(u[r].y)));
  }
  block_max(mag, st);
  __syncthreads();
  const int E = block_exp(st[0]);
  e = E >= 0x7FF ? kNaN : E - 1080;
  if (active) {
#pragma unroll
    for (int r = 0; r < 8; ++r) v[r] = from_double(u[r], E);
    dft<8>(v);
    c64* dst = buf + pad(8 * t);
#pragma unroll
    for (int r = 0; r < 8; ++r) dst[r] = v[r];
  }
  static_assert(!shifts(1, FORWARD), "no statistics after the first stage");
  __syncthreads();
  rest<LOGN, 8, 1, FORWARD>(v, buf, t, active, st, tw, e);
  if (E >= 0x7FF) e = kNaN;
}

// The whole transform of the integers v[r] = x[t + r N/8], |z| <= 2^58.5 (read from `buf` by
// the caller), in units of 2^e; the order of an inverse.
template <int LOGN>
__device__ __forceinline__ void transform(c64 (&v)[8], c64* buf, int t, bool active, unsigned* st,
                                          const int4* __restrict__ tw, int& e) {
  static_assert(LOGN >= 4, "at least two stages");
  __syncthreads();
  unsigned h = 0;
  if (active) {
    dft<8>(v);
    c64* dst = buf + pad(8 * t);
#pragma unroll
    for (int r = 0; r < 8; ++r) {
      dst[r] = v[r];
      h |= spread(v[r]);
    }
  }
  block_or(h, st + 1);
  __syncthreads();
  rest<LOGN, 8, 1, INVERSE>(v, buf, t, active, st, tw, e);
}

// ------------------------------------------------------------------------- //
// Column transforms of N = 64 N2 points in two passes (the four-step form): with
// j = N2 j1 + j2 and m = m1 + 64 m2,
//   pass A: Y[m1][j2] = sum_j1 x[N2 j1 + j2] w_64^(j1 m1), in place of the rows N2 j1 + j2;
//   pass B: X[m1 + 64 m2] = sum_j2 (Y[m1][j2] w_N^(j2 m1)) w_N2^(j2 m2).
// A block serves kCols adjacent columns, so a row of a block is a contiguous 256 bytes and
// the lanes of a warp share their twiddles; eight values per thread.  Pass A leaves
// integers with one exponent per block (exps[f][j2][column group]); pass B brings its
// rows to a common exponent, fitted to its own largest value, as it reads them.
// ------------------------------------------------------------------------- //
constexpr int kCols = 16;
constexpr int kColThreads = 128;

// 8 R2-point DFT of v[i] = x[l + R2 i] held by the threads l < R2 of a column; on return
// v[mm R2 + q] = X[m + 8 q] with m = l (8/R2) + mm.  ex: the group's [8][R2][kCols] exchange
// buffer; w: w[ws t] = w_{8 R2}^t.  One barrier (none for R2 = 1); adds kDrop to the
// exponent unless R2 = 1.  FIT (an inverse's spectra, see shifts()): the block is rescaled between the
// two halves, another barrier; st: a zeroed shared word; returns the left shift.
template <int R2, bool FIT = false>
__device__ __forceinline__ int dft_group(c64 (&v)[8], int c, int l, c64* ex,
                                         const int4* __restrict__ w, int ws, unsigned* st = nullptr) {
  int L = 0;
  dft<8>(v);
  if constexpr (FIT) {
    unsigned h = 0;
#pragma unroll
    for (int m = 0; m < 8; ++m) h |= spread(v[m]);
    block_or(h, st);
    __syncthreads();
    L = headroom(*st);
#pragma unroll
    for (int m = 0; m < 8; ++m) v[m] = {v[m].x << L, v[m].y << L};
  }
  if constexpr (R2 > 1) {
    v[0] = drop(v[0]);
#pragma unroll
    for (int m = 1; m < 8; ++m) v[m] = mulw(v[m], __ldg(w + ws * (l * m)));
#pragma unroll
    for (int m = 0; m < 8; ++m) ex[(m * R2 + l) * kCols + c] = v[m];
    __syncthreads();
#pragma unroll
    for (int k = 0; k < 8; ++k) v[k] = ex[(l * 8 + k) * kCols + c];
#pragma unroll
    for (int mm = 0; mm < 8 / R2; ++mm) dft<R2>(v + mm * R2);
  }
  return L;
}

// Pass A for rows N2 j1 + j2 of the columns from kx0 on.  load(row, kx): the doubles;
// live: whether this thread's column exists.  st: two zeroed shared words.
template <int N2, typename Load>
__device__ __forceinline__ void cols_pass_a(Load load, c64* __restrict__ mid, unsigned pitch, int j2,
                                            int kx, bool live, c64* ex, unsigned* st,
                                            const int4* __restrict__ w, int* exp_out) {
  const int c = threadIdx.x & (kCols - 1), l = threadIdx.x / kCols;
  double2 u[8];
  c64 v[8];
  unsigned mag = 0;
#pragma unroll
  for (int i = 0; i < 8; ++i) {
    u[i] = live ? load(N2 * (l + 8 * i) + j2, kx) : double2{0.0, 0.0};
    mag = max(mag, max(magnitude(u[i].x), magnitude(u[i].y)));
  }
  block_max(mag, st);
  __syncthreads();
  const int E = block_exp(st[0]);
#pragma unroll
  for (int i = 0; i < 8; ++i) v[i] = from_double(u[i], E);
  dft_group<8>(v, c, l, ex, w, N2);
  if (live) {
#pragma unroll
    for (int q = 0; q < 8; ++q) mid[(unsigned)(N2 * (l + 8 * q) + j2) * pitch + kx] = v[q];
  }
  if (threadIdx.x == 0) *exp_out = E >= 0x7FF ? kNaN : E - 1080 + kDrop;
}

// Pass B for m1: v[mm R2 + q] = X[m1 + 64 (m + 8 q)], m = l (8/R2) + mm, and their exponent.
// exps: exponents of the rows j2, at stride estride.
template <int N2>
__device__ __forceinline__ int cols_pass_b(c64 (&v)[8], const c64* __restrict__ mid, unsigned pitch,
                                           int m1, int l, int kx, bool live, c64* ex, unsigned* st,
                                           const int4* __restrict__ w, const int* __restrict__ exps,
                                           int estride) {
  constexpr int R2 = N2 / 8;
  const int c = threadIdx.x & (kCols - 1);
  int er[8], top = -2048;
#pragma unroll
  for (int i = 0; i < 8; ++i) {
    er[i] = exps[(l + R2 * i) * estride];
    v[i] = live ? mid[(unsigned)(N2 * m1 + l + R2 * i) * pitch + kx] : c64{0, 0};
    top = max(top, er[i] + 63 - __clz((int)(spread(v[i]) | 1u)));
  }
  block_max((unsigned)(top + 4096), st);
  __syncthreads();
  const int e0 = (int)st[0] - 4096 - 62;
#pragma unroll
  for (int i = 0; i < 8; ++i) {
    const int s = er[i] - e0, up = max(s, 0), dn = min(max(-s, 0), 63);
    const i64 rnd = (i64)((1ull << dn) >> 1);
    const c64 a = {((v[i].x << up) + rnd) >> dn, ((v[i].y << up) + rnd) >> dn};
    v[i] = mulw(a, __ldg(w + (l + R2 * i) * m1));
  }
  dft_group<R2>(v, c, l, ex, w, 64);
  return e0 + kDrop + (R2 > 1 ? kDrop : 0);
}

// v times an FxFactor, its power of two left to the exponent
__device__ __forceinline__ c64 scaled(c64 v, const FxFactor& f) {
  return f.m ? c64{mulc(v.x, f.m, f.r), mulc(v.y, f.m, f.r)} : v;
}

}  // namespace fx
}  // namespace fc2d
