// The small squares of Fourier Forwarding in fixed point (fx_squares.cu).
#pragma once
#include <cuda_runtime.h>

#include <cstddef>
#include <cstdint>

namespace fc2d {

// Device tables of a set of n squares
struct SquareArgs {
  int n;
  const int32_t* origin;        // [n][2] (row, column) of the first grid point
  const double *A, *Q;          // 1D-FC: continuation [C][d], Gram [d][d]
  const int4* tw;               // exp(-2 pi i t/64) 2^60 in limbs
  const int32_t *served_off, *served_at, *served_local;  // served_at: interface point
  const int32_t* rows;          // [n][2]: first and last box row holding served points
};

size_t squares_spectrum_bytes(int n_sq, int n_f);
size_t squares_factor_bytes(int S);
// the time factors of the small steps s < S at s dt, for u_t scaled by 2^eT (2^eT >= S dt)
void squares_factors(int S, double c, double h, double dt, int eT, void* fac, cudaStream_t s);
// the spectra of u and u_t on every square (exps: n n_f ints)
void squares_expand(const SquareArgs& q, int n_side, int C, int d, int nx, int64_t grid_stride,
                    int n_f, int eT, const double* u, const double* ut, void* spec, int* exps,
                    cudaStream_t s);
// the modal solution of small step `step` at the served interface points, out [point][n_f]
void squares_solve(const SquareArgs& q, int max_rows, int n_f, const void* spec, const int* exps,
                   const void* fac, int step, double* out, cudaStream_t s);

}  // namespace fc2d
