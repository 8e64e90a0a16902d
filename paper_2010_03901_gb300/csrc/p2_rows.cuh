// Shared pieces of the power-of-two DFT kernels (FP32: fft_pow2.cu; double, in fixed
// point: fft_fx.cu): complex types, L2 hints, rounding of doubles to float on the integer
// pipe, the padding of shared buffers, and the assembly of an extended row.
#pragma once
#include <cuda_runtime.h>

#include <cstdint>

#include "fc2d_kernels.cuh"

namespace fc2d {
namespace p2 {

template <typename T> struct Cx;
template <> struct Cx<double> { using type = double2; };
template <> struct Cx<float> { using type = float2; };

// L2 residency hints (PTX eviction priorities; no value changes).  The grid values f
// are read once per call: they bypass L1 and go first when L2 evicts, so that the row
// transforms' output (the intermediate, read again by both column passes) stays in L2.
// The intermediate's stores ask L2 to keep their lines; the spectrum, written once,
// asks it to evict its lines first.  Bits: 1 f loads, 2 intermediate stores, 4 spectrum
// stores.
#ifndef FC2D_L2_HINTS
#define FC2D_L2_HINTS 1
#endif
__device__ __forceinline__ uint64_t l2_keep() {
  uint64_t pol;
  asm("createpolicy.fractional.L2::evict_last.b64 %0, 1.0;" : "=l"(pol));
  return pol;
}
__device__ __forceinline__ uint64_t l2_drop() {
  uint64_t pol;
  asm("createpolicy.fractional.L2::evict_first.b64 %0, 1.0;" : "=l"(pol));
  return pol;
}
__device__ __forceinline__ double2 ld_stream(const double2* p, uint64_t pol) {
#if FC2D_L2_HINTS & 1
  double2 v;
  asm("ld.global.nc.L1::no_allocate.L2::cache_hint.v2.f64 {%0, %1}, [%2], %3;"
      : "=d"(v.x), "=d"(v.y) : "l"(p), "l"(pol));
  return v;
#else
  return __ldg(p);
#endif
}
// store with an L2 policy (FP32 complex); other types store plainly
template <int BIT, typename C> __device__ __forceinline__ void st_hint(C* p, C v, uint64_t pol) {
  if constexpr (sizeof(C) == 8 && (FC2D_L2_HINTS & BIT)) {
    asm volatile("st.global.L2::cache_hint.v2.f32 [%0], {%1, %2}, %3;"
                 ::"l"(p), "f"(v.x), "f"(v.y), "l"(pol) : "memory");
  } else {
    *p = v;
  }
}

// Round-to-nearest-even double -> float on the integer pipe (the FP64 pipe that the
// conversion instruction uses is narrow on this part), for doubles whose exponent e lies
// in [897, 1148] (float exponents 1..252, so no overflow even after rounding up): add
// 2^28 - 1 plus bit 29 to the 64-bit pattern (round half to even at bit 29; a mantissa
// carry moves into the exponent), keep bits 29..60 (e's low 9 bits over the top 23
// mantissa bits), rebase the exponent by 896 (mod 2^32) and put the sign back.  Other
// values (zero, subnormal, huge, inf, NaN) take the hardware conversion.
__device__ __forceinline__ bool d2f_in_range(unsigned hi) {
  return (hi & 0x7FF00000u) - (897u << 20) <= (251u << 20);
}
__device__ __forceinline__ float d2f_in(double x) {
  const unsigned long long b = (unsigned long long)__double_as_longlong(x);
  const unsigned long long u = b + 0x0FFFFFFFull + ((b >> 29) & 1ull);
  const unsigned r = (unsigned)(u >> 29) - (896u << 23);
  return __uint_as_float(r | ((unsigned)(b >> 32) & 0x80000000u));
}
__device__ __forceinline__ float d2f_rn(double x) {
  return d2f_in_range((unsigned)__double2hiint(x)) ? d2f_in(x) : __double2float_rn(x);
}
// both values of a pair, one range test
__device__ __forceinline__ float2 d2f2_rn(double2 v) {
  if (d2f_in_range((unsigned)__double2hiint(v.x)) && d2f_in_range((unsigned)__double2hiint(v.y)))
    return float2{d2f_in(v.x), d2f_in(v.y)};
  return float2{__double2float_rn(v.x), __double2float_rn(v.y)};
}
template <typename T> __device__ __forceinline__ T from_double(double x) { return (T)x; }
template <> __device__ __forceinline__ float from_double<float>(double x) { return d2f_rn(x); }

// One pad element per E = elems<T>() elements: the first stage writes at stride E
// (index E j + r), which the pad spreads over all banks; the other stages access
// contiguous runs of the thread index, which the pad leaves contiguous.
template <typename T> __host__ __device__ constexpr int pad_shift() { return sizeof(T) == 4 ? 4 : 3; }
template <typename T> __device__ __forceinline__ int pad(int i) { return i + (i >> pad_shift<T>()); }
template <typename T> __host__ __device__ constexpr int padded(int n) { return n + (n >> pad_shift<T>()); }
// pad(i + r S) for r = 0..R-1 as pad(i) plus a compile-time offset, which the shared
// memory instructions take as an immediate: exact when S is a multiple of the pad unit
// U (then pad(i + r S) = pad(i) + r (S + S / U)), or when S = 1, R divides U and i is a
// multiple of R (then i and i + R - 1 lie in one unit).
template <typename T, int S, int R> __host__ __device__ constexpr bool pad_affine() {
  return S % (1 << pad_shift<T>()) == 0 || (S == 1 && (1 << pad_shift<T>()) % R == 0);
}
template <typename T, int S> __host__ __device__ constexpr int pad_step() {
  return S % (1 << pad_shift<T>()) == 0 ? S + S / (1 << pad_shift<T>()) : S;
}

// The extended row j of function f as NH complex pairs z_n = x_{2n} + i x_{2n+1} in the
// padded shared buffer: mode 0 from an extended grid; mode 1 assembled (zeros, the
// inside reals of f, the strip values).  Ends with a barrier.  It makes the kernel's
// dependent-launch wait: in mode 0 before anything else; in the assembled modes only
// before the strip values, which the previous kernel (the blend + interpolation) writes.
// f itself was written before that kernel's own wait returned, and this kernel was
// launched after that kernel triggered, so f may be read before the wait.
// NTHR: the block size (blockDim.x) when known at compile time, else 0
template <typename T, typename TV, int NTHR = 0>
__device__ __forceinline__ void assemble_row(const RowArgs& ra, int mode, int NH, int j, int f,
                                             const T* __restrict__ ext,
                                             const double* __restrict__ f_grid,
                                             const TV* __restrict__ vals,
                                             typename Cx<T>::type* buf) {
  using C = typename Cx<T>::type;
  const int nx = 2 * NH;
  const int nthr = NTHR ? NTHR : (int)blockDim.x;
  auto put = [&](int i, T v) { reinterpret_cast<T*>(&buf[pad<T>(i >> 1)])[i & 1] = v; };
  if (mode == 0) {
    pdl_wait();
    pdl_trigger();
    const T* src = ext + (size_t)f * ra.grid_stride + (size_t)j * nx;
    for (int n = threadIdx.x; n < NH; n += nthr) {
      const C v = reinterpret_cast<const C*>(src)[n];
      buf[pad<T>(n)] = v;
    }
  } else {
    // mode 1: element i of the row at fg[i]; mode 2 (compact): at fin[coff_k + i - lo_k]
    const double* fg = mode == 1 ? f_grid + (size_t)f * ra.grid_stride + (size_t)j * nx
                                 : f_grid + (size_t)f * ra.grid_stride;
    const int iv0 = __ldg(ra.row_iv_off + j), iv1 = __ldg(ra.row_iv_off + j + 1);
    if (NTHR > 0 && NTHR % (1 << pad_shift<T>()) == 0 && NH % NTHR == 0) {
      C* z = buf + pad<T>(threadIdx.x);  // n = t + i NTHR: pad(n) = pad(t) + i pad_step
      for (int i = 0; i < NH / (NTHR > 0 ? NTHR : 1); ++i)
        z[i * pad_step<T, (NTHR > 0 ? NTHR : 1)>()] = C{(T)0, (T)0};
    } else {
      for (int n = threadIdx.x; n < NH; n += nthr) buf[pad<T>(n)] = C{(T)0, (T)0};
    }
    __syncthreads();
    // inside intervals [lo, hi]: the pairs n with lo <= 2n and 2n + 1 <= hi as one
    // 16-byte load each when the source is 16-byte aligned at even i (eight loads in
    // flight per thread), the odd ends element by element
    for (int k = iv0; k < iv1; ++k) {
      const int lo = __ldg(ra.row_iv + 2 * k), hi = __ldg(ra.row_iv + 2 * k + 1);
      const double* src = mode == 1 ? fg : fg + ((int64_t)__ldg(ra.row_iv_coff + k) - lo);
      const bool vec = (reinterpret_cast<uintptr_t>(src) & 15) == 0;
      if (vec) {
        const int p0 = (lo + 1) >> 1, p1 = (hi + 1) >> 1;  // pairs p0 .. p1 - 1
        const double2* fg2 = reinterpret_cast<const double2*>(src);
        const uint64_t pol = l2_drop();
        for (int n0 = p0 + threadIdx.x; n0 < p1; n0 += 8 * nthr) {
          // pairs n0 + u nthr from two base pointers (with a compile-time block size that
          // is a multiple of the pad unit, pad(n0 + u nthr) = pad(n0) + u pad_step)
          constexpr bool affine = NTHR > 0 && NTHR % (1 << pad_shift<T>()) == 0;
          const double2* s2 = fg2 + n0;
          C* d2 = buf + pad<T>(n0);
          double2 d[8];
#pragma unroll
          for (int u = 0; u < 8; ++u) {
            const int n = n0 + u * nthr;
            d[u] = n < p1 ? ld_stream(s2 + u * nthr, pol) : make_double2(0.0, 0.0);
          }
#pragma unroll
          for (int u = 0; u < 8; ++u) {
            const int n = n0 + u * nthr;
            if (n < p1) {
              C* dst = affine ? d2 + u * pad_step<T, (NTHR > 0 ? NTHR : 1)>() : buf + pad<T>(n);
              if constexpr (sizeof(T) == 4) *dst = d2f2_rn(d[u]);
              else *dst = C{d[u].x, d[u].y};
            }
          }
        }
        if (threadIdx.x == 0 && (lo & 1)) put(lo, from_double<T>(__ldg(src + lo)));
        if (threadIdx.x == 0 && !(hi & 1)) put(hi, from_double<T>(__ldg(src + hi)));
      } else {
        for (int i = lo + threadIdx.x; i <= hi; i += nthr) put(i, from_double<T>(__ldg(src + i)));
      }
    }
    const int s0 = __ldg(ra.row_strip_off + j), s1 = __ldg(ra.row_strip_off + j + 1);
    const int base = j * nx;
    const TV* v = vals + (size_t)f * ra.n_strip;
    pdl_wait();
    pdl_trigger();
    for (int k = s0 + threadIdx.x; k < s1; k += nthr) put(__ldg(ra.s_lin + k) - base, (T)__ldg(v + k));
  }
  __syncthreads();
}

}  // namespace p2
}  // namespace fc2d
