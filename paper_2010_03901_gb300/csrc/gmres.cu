// GMRES without restart for a dense real matrix: Arnoldi with classical Gram-Schmidt twice,
// Givens rotations on the device.
//
// At the sizes of a boundary integral equation (n about 1000) an iteration is a few
// microseconds of work with three points at which every block needs every other one's
// result.  The whole solve is one cooperative launch of one block per SM (fewer where
// they do not fit at once): the blocks keep
// their rows of A in shared memory (from L2 where they do not fit) and their rows of the
// basis in L1, and meet three times per iteration.  Each phase ends with the blocks' partial
// sums (projections or squares), which every block adds up in the same order.  w is kept
// unscaled: A v_j is (A w) / |w|.
//   1  v_j = w / |w|; w' = A v_j; partial h1 = V^T w'.  Block 0, which has no rows, takes
//      iteration j - 1's column through the rotations meanwhile.
//   2  w' -= V h1; partial h2 = V^T w'         3  w' -= V h2; partial |w'|^2
// What bounds it: 2 n^2 FP64 operations per iteration, 1.9 us for n = 1024, and the latency
// of the three meetings.  A kernel per dot product, norm and rotation (eight per iteration)
// took 722 us for the star at 1024^2 (15 iterations), three kernels per iteration 561 us,
// this form 283.
#include <cuda_runtime.h>

#include <algorithm>
#include <cmath>

#include "gmres.h"

namespace fc2d {

namespace {

constexpr int kT = 256;             // threads: 32 groups of 8 lanes
constexpr int kLd = kGmresMax + 1;  // row length of the partial projections

__device__ __forceinline__ double warp_sum(double v) {
  for (int o = 16; o; o >>= 1) v += __shfl_xor_sync(0xFFFFFFFFu, v, o);
  return v;
}

// sum of x[k stride], k = k0, k0 + step, .. < n, with N loads in flight at a time (the
// blocks' partial sums come from L2, 0.7 us away)
template <int N>
__device__ __forceinline__ double gather(const double* x, size_t stride, int k0, int step, int n) {
  double v = 0.0;
  for (int k = k0; k < n; k += N * step) {
    double r[N];
#pragma unroll
    for (int q = 0; q < N; ++q) r[q] = k + q * step < n ? __ldcg(x + (k + q * step) * stride) : 0.0;
#pragma unroll
    for (int q = 0; q < N; ++q) v += r[q];
  }
  return v;
}

// sum of x[0 .. n) by a warp.  (An FP64 instruction occupies the SM's pipe for 16 clocks
// whatever the number of active lanes: what one warp can do for the block, one warp does.)
__device__ __forceinline__ double total(const double* x, int n) {
  return warp_sum(gather<5>(x, 1, threadIdx.x & 31, 32, n));
}

// partial projections part[i] = sum over the block's rows of V_i w, i < m
__device__ __forceinline__ void partials(int n, int rows, int m, const double* V, const double* ws,
                                         double* part) {
  const int r = threadIdx.x & 7;
  for (int i = threadIdx.x >> 3; i < (m + 31) / 32 * 32; i += 32) {  // whole warps
    double v = 0.0;
    if (i < m)
      for (int k = r; k < rows; k += 8) v = fma(V[(size_t)i * n + k], ws[k], v);
    for (int o = 4; o; o >>= 1) v += __shfl_xor_sync(0xFFFFFFFFu, v, o);
    if (i < m && r == 0) part[i] = v;
  }
}

// Iteration j after both projections and |w|^2 = nn: column j of H, the earlier rotations
// applied to it, its own rotation, the residual estimate.
__device__ void rotate(GmresDev* G, int j, double nn, double tol, double* col, double* cs,
                       double* sn) {
  const int t = threadIdx.x;
  for (int i = t; i <= j; i += kT) {
    col[i] = __ldcg(G->h1 + i) + __ldcg(G->h2 + i);
    cs[i] = G->cs[i];
    sn[i] = G->sn[i];
  }
  __syncthreads();
  if (t == 0) {
    const double hn = sqrt(nn);
    double a = col[0];
    for (int i = 0; i < j; ++i) {
      const double b = col[i + 1];
      col[i] = cs[i] * a + sn[i] * b;
      a = -sn[i] * a + cs[i] * b;
    }
    const double r = hypot(a, hn), c = r == 0 ? 1.0 : a / r, s = r == 0 ? 0.0 : hn / r;
    G->cs[j] = c;
    G->sn[j] = s;
    col[j] = r;
    const double e = G->e[j], e1 = -s * e;
    G->e[j + 1] = e1;
    G->e[j] = c * e;
    G->m = j + 1;
    G->resid = fabs(e1) / G->beta;
    if (fabs(e1) <= tol * G->beta || hn == 0.0 || j + 1 == kGmresMax) {
      G->done = 1;
      G->stop = 1;
    }
  }
  __syncthreads();
  for (int i = t; i <= j; i += kT) G->H[i * kGmresMax + j] = col[i];
}

// Waits until all blocks of the launch have come here `gen` times; false when a block does
// not come within a second or so (every block then leaves).
constexpr unsigned kMeetPolls = 1u << 21;
__device__ bool meet(unsigned* count, unsigned gen, unsigned limit = kMeetPolls) {
  __syncthreads();
  bool ok = true;
  if (threadIdx.x == 0) {
    __threadfence();
    atomicAdd(count, 1u);
    const unsigned all = gen * gridDim.x;
    unsigned polls = 0;
    while (*(volatile unsigned*)count < all && ok) ok = ++polls < limit;
    __threadfence();
  }
  return !__syncthreads_or(!ok);
}

// ws -= V h for the block's rows, h the sum of the blocks' partial projections
__device__ __forceinline__ void project(int n, int nr, int n_blk, int m, const double* V, double* ws,
                                        const double* part, double* hs, double (*red)[32],
                                        double* h_out) {
  const int t = threadIdx.x, lane = t & 31, wp = t >> 5;
  for (int i0 = 0; i0 < m; i0 += 32) {
    // width lanes per partial vector, 32 / width of those per warp
    const int width = m - i0 > 16 ? 32 : m - i0 > 8 ? 16 : 8;
    const int i = i0 + (lane & (width - 1)), per = 32 / width;
    double v = 0.0;
    if (i < m) v = gather<10>(part + i, kLd, wp * per + lane / width, kT / width, n_blk);
    if (width < 32) v += __shfl_xor_sync(0xFFFFFFFFu, v, 16);
    if (width < 16) v += __shfl_xor_sync(0xFFFFFFFFu, v, 8);
    red[wp][lane] = v;
    __syncthreads();
    if (wp == 0 && lane < width && i < m) {
      for (int k = 1; k < kT / 32; ++k) v += red[k][lane];
      hs[i] = v;
      if (h_out) h_out[i] = v;
    }
    __syncthreads();
  }
  // 8 rows at a time; 32 groups share the vectors
  const int r = t & 7;
  for (int k = 0; k < nr; k += 8) {
    double v = 0.0;
    if (k + r < nr)
      for (int i = t >> 3; i < m; i += 32) v = fma(hs[i], V[(size_t)i * n + k + r], v);
    v += __shfl_xor_sync(0xFFFFFFFFu, v, 8);
    v += __shfl_xor_sync(0xFFFFFFFFu, v, 16);
    if (lane < 8) red[wp][lane] = v;
    __syncthreads();
    if (t < 8 && k + t < nr) {
      for (int q = 1; q < kT / 32; ++q) v += red[q][t];
      ws[k + t] -= v;
    }
    __syncthreads();
  }
}

// partial square of the block's rows
__device__ __forceinline__ void square(int nr, const double* ws, double* out) {
  if (threadIdx.x >= 32) return;
  double v = 0.0;
  for (int k = threadIdx.x; k < nr; k += 32) v = fma(ws[k], ws[k], v);
  v = warp_sum(v);
  if (threadIdx.x == 0) *out = v;
}

// y from the triangular system R y = e over the first m columns, column by column
__device__ void triangle(GmresDev* G, int m, double* yi) {
  const int k = threadIdx.x;
  double e = k < m ? G->e[k] : 0.0;
  double h = k < m ? G->H[k * kGmresMax + m - 1] : 0.0;  // rows k <= column only
  for (int i = m - 1; i >= 0; --i) {
    const double next = i > 0 && k < i ? G->H[k * kGmresMax + i - 1] : 0.0;
    if (k == i) *yi = e / h;
    __syncthreads();
    if (k == i) G->y[i] = *yi;
    if (k < i) e = fma(-h, *yi, e);
    h = next;
    __syncthreads();
  }
}

// out = the block's rows of A times w, both from L2 or HBM: four rows per warp share the
// vector and keep 32 loads per lane in flight (64 KB per SM, about the latency times the
// bandwidth)
__device__ __forceinline__ void rows_times(int n, int nr, const double* __restrict__ A,
                                           const double* w, double* out) {
  constexpr int R = 4, U = 8;
  const int lane = threadIdx.x & 31;
  for (int k0 = (threadIdx.x >> 5) * R; k0 < nr; k0 += kT / 32 * R) {
    const double* a[R];
    double v[R];
#pragma unroll
    for (int r = 0; r < R; ++r) {
      a[r] = A + (size_t)min(k0 + r, nr - 1) * n;
      v[r] = 0.0;
    }
    int i = lane;
    for (; i + 32 * (U - 1) < n; i += 32 * U) {
      double x[U], y[R][U];
#pragma unroll
      for (int u = 0; u < U; ++u) {
        x[u] = __ldcg(w + i + 32 * u);
#pragma unroll
        for (int r = 0; r < R; ++r) y[r][u] = __ldcg(a[r] + i + 32 * u);
      }
#pragma unroll
      for (int u = 0; u < U; ++u)
#pragma unroll
        for (int r = 0; r < R; ++r) v[r] = fma(y[r][u], x[u], v[r]);
    }
    for (; i < n; i += 32) {
      const double x = __ldcg(w + i);
#pragma unroll
      for (int r = 0; r < R; ++r) v[r] = fma(__ldcg(a[r] + i), x, v[r]);
    }
#pragma unroll
    for (int r = 0; r < R; ++r) {
      v[r] = warp_sum(v[r]);
      if (lane == 0 && k0 + r < nr) out[k0 + r] = v[r];
    }
  }
}

// SMEM: the block's rows of A and the vector in shared memory
template <bool SMEM>
__global__ void __launch_bounds__(kT, 1) k_gmres(int n, int rows, const double* __restrict__ A,
                                              const double* __restrict__ g, double* V, double* w,
                                              double* part0, double* part1, double* norm,
                                              GmresDev* G, double* x, double tol) {
  extern __shared__ double sm[];
  __shared__ double hs[kGmresMax], red[kT / 32][32];
  const int t = threadIdx.x, lane = t & 31, wp = t >> 5;
  const int n_blk = gridDim.x - 1, blk = (int)blockIdx.x - 1;
  const int r0 = blk * rows, nr = blk < 0 ? 0 : min(rows, n - r0);
  double* As = sm;
  double* wv = sm + (SMEM ? (size_t)rows * n : 0);
  double* ws = wv + (SMEM ? n : 0);  // the block's rows of w; block 0: the rotations
  double* wn = ws + rows;
  double* Vb = V + r0;
  unsigned gen = 0;
  for (int k = t; k < nr; k += kT) {
    const double v = g[r0 + k];
    ws[k] = v;
    w[r0 + k] = v;
  }
  __syncthreads();
  if (blk >= 0) square(nr, ws, norm + blk);
  if (SMEM)
    for (size_t k = t; k < (size_t)nr * n; k += kT) As[k] = A[(size_t)r0 * n + k];
  bool ok = meet(&G->count, ++gen);
  for (int j = 0; ok; ++j) {
    if (wp == kT / 32 - 1) {
      const double nn = total(norm, n_blk);
      if (lane == 0) {
        red[0][0] = nn;
        red[0][1] = 1.0 / sqrt(nn);
      }
    }
    if (blk < 0) {
      __syncthreads();
      const double nn = red[0][0];
      if (j > 0) {
        rotate(G, j - 1, nn, tol, ws, ws + kLd, ws + 2 * kLd);
      } else if (t == 0) {
        const double beta = sqrt(nn);
        G->beta = beta;
        G->e[0] = beta;
        G->m = 0;
        G->resid = 0.0;
        G->done = G->stop = beta == 0.0 ? 1 : 0;
      }
    } else if (j < kGmresMax) {
      if (SMEM) {
#pragma unroll 4
        for (int k = t; k < n; k += kT) wv[k] = __ldcg(w + k);
        __syncthreads();
      }
      if (SMEM) {
        for (int k = wp; k < nr; k += kT / 32) {  // a warp per row
          const double* a = As + (size_t)k * n;
          double v0 = 0.0, v1 = 0.0;
          int i = lane;
#pragma unroll 4
          for (; i + 32 < n; i += 64) {
            v0 = fma(a[i], wv[i], v0);
            v1 = fma(a[i + 32], wv[i + 32], v1);
          }
          if (i < n) v0 = fma(a[i], wv[i], v0);
          const double v = warp_sum(v0 + v1);
          if (lane == 0) wn[k] = v;
        }
      } else {
        rows_times(n, nr, A + (size_t)r0 * n, w, wn);
      }
      __syncthreads();
      const double scale = red[0][1];
      for (int k = t; k < nr; k += kT) {
        Vb[(size_t)j * n + k] = ws[k] * scale;
        ws[k] = wn[k] * scale;
      }
      __syncthreads();
      partials(n, nr, j + 1, Vb, ws, part0 + (size_t)blk * kLd);
    }
    ok = meet(&G->count, ++gen);
    if (!ok || *(volatile int*)&G->stop) break;
    if (blk >= 0) {
      project(n, nr, n_blk, j + 1, Vb, ws, part0, hs, red, blk == 0 ? G->h1 : nullptr);
      partials(n, nr, j + 1, Vb, ws, part1 + (size_t)blk * kLd);
    }
    if (!(ok = meet(&G->count, ++gen))) break;
    if (blk >= 0) {
      project(n, nr, n_blk, j + 1, Vb, ws, part1, hs, red, blk == 0 ? G->h2 : nullptr);
      square(nr, ws, norm + blk);
      for (int k = t; k < nr; k += kT) w[r0 + k] = ws[k];
    }
    ok = meet(&G->count, ++gen);
  }
  if (!ok) {
    if (t == 0) G->done = -1;
    return;
  }
  const int m = *(volatile int*)&G->m;
  if (blk < 0) triangle(G, m, hs);
  ok = meet(&G->count, ++gen);
  if (!ok) {
    if (t == 0) G->done = -1;
    return;
  }
  if (blk >= 0) {
    for (int i = t; i < m; i += kT) hs[i] = __ldcg(G->y + i);
    __syncthreads();
    for (int k = t; k < nr; k += kT) {
      double v = 0.0;
#pragma unroll 8
      for (int i = 0; i < m; ++i) v = fma(hs[i], Vb[(size_t)i * n + k], v);
      x[r0 + k] = v;
    }
  }
}

// A meeting whose other block never comes: meet(), as k_gmres calls it, with a given number
// of polls, so that the way out can be taken on purpose.  One warp.
__global__ void __launch_bounds__(32) k_meet_probe(int* status, unsigned limit) {
  __shared__ unsigned count;
  if (threadIdx.x == 0) count = 0;
  if (!meet(&count, 2, limit) && threadIdx.x == 0) atomicExch(status, (int)FC2D_ERR_TIMEOUT);
}

constexpr size_t kSmemMax = 220 * 1024;
size_t smem_bytes(int n, int rows, bool in_smem) {
  return ((in_smem ? (size_t)rows * n + n : 0) + std::max<size_t>(2 * rows, 3 * kLd)) * sizeof(double);
}

}  // namespace

fc2d_status launch_meet_probe(int* status, unsigned limit, cudaStream_t s) {
  k_meet_probe<<<1, 32, 0, s>>>(status, limit);
  return cuda_check(cudaGetLastError(), "meeting probe launch");
}

// One block per SM, one of them for the rotations
int gmres_rows(int n, int n_sm) {
  const int most = std::max(1, n_sm - 1);
  return (n + most - 1) / most;
}

fc2d_status gmres_solve(Gmres& q, const double* g, double* x, double tol, int* iters,
                        double* resid, cudaStream_t s) {
  static_assert(kT >= kGmresMax, "triangle: a thread per column");
  int n = q.n, rows = q.rows;
  void* args[] = {&n, &rows, &q.A, &g, &q.V, &q.w, &q.part[0], &q.part[1], &q.norm, &q.dev, &x, &tol};
  for (int n_blk = q.n_blk;; n_blk = (n_blk + 1) / 2) {
    rows = (n + n_blk - 1) / n_blk;
    const bool in_smem = smem_bytes(n, rows, true) <= kSmemMax;
    const size_t sm = smem_bytes(n, rows, in_smem);
    auto kernel = in_smem ? k_gmres<true> : k_gmres<false>;
    cudaFuncSetAttribute(kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)sm);
    cudaMemsetAsync(&q.dev->count, 0, sizeof(unsigned), s);
    const unsigned blocks = (unsigned)((n + rows - 1) / rows) + 1;
    const cudaError_t e =
        cudaLaunchCooperativeKernel((const void*)kernel, dim3(blocks), dim3(kT), args, sm, s);
    if (e == cudaSuccess) break;
    cudaGetLastError();
    // a stream whose context has a part of the SMs only: fewer blocks, of more rows each
    if (e != cudaErrorCooperativeLaunchTooLarge || n_blk == 1) return cuda_check(e, "GMRES");
  }
  GmresDev::State st;
  cudaMemcpyAsync(&st, static_cast<GmresDev::State*>(q.dev), sizeof(st), cudaMemcpyDeviceToHost, s);
  if (cudaStreamSynchronize(s) != cudaSuccess) return cuda_check(cudaGetLastError(), "GMRES");
  if (st.done < 0) return set_error(FC2D_ERR_CUDA, "GMRES: the blocks of the launch did not meet");
  *iters = st.m;
  *resid = st.resid;
  if (st.resid > 1e3 * tol)
    return set_error(FC2D_ERR_NOT_CONVERGED, "GMRES did not reach its tolerance");
  return FC2D_OK;
}

}  // namespace fc2d
