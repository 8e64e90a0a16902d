// GMRES for a dense real system on the device (gmres.cu).
#pragma once
#include <cuda_runtime.h>

#include "plan_internal.h"

namespace fc2d {

constexpr int kGmresMax = 200;

// Small dense part: the Hessenberg matrix H, the Givens rotations (cs, sn), the rotated
// right-hand side e, and the state that the host reads.
struct GmresState {
  double beta, resid;  // ||g||, |e_m| / beta
  int stop, done, m;   // done < 0: the launch failed
  unsigned count;      // arrivals of blocks
};
struct GmresDev : GmresState {
  using State = GmresState;
  double H[(kGmresMax + 1) * kGmresMax];  // H[i][j] at i kGmresMax + j
  double cs[kGmresMax], sn[kGmresMax], e[kGmresMax + 1], y[kGmresMax];
  double h1[kGmresMax + 1], h2[kGmresMax + 1];  // the two Gram-Schmidt passes' projections
};

struct Gmres {
  int n = 0, n_blk = 0, rows = 0;  // unknowns; blocks of `rows` consecutive rows
  const double* A = nullptr;       // [n][n]
  double* V = nullptr;             // [kGmresMax + 1][n]
  double* w = nullptr;             // [n]
  double* part[2] = {nullptr, nullptr};  // [n_blk][kGmresMax + 1] partial projections
  double* norm = nullptr;                // [n_blk] partial squares
  GmresDev* dev = nullptr;
};

// rows per block for n unknowns on n_sm SMs
int gmres_rows(int n, int n_sm);
// A x = g to |residual| <= tol |g|; iterations and the relative residual estimate
fc2d_status gmres_solve(Gmres& q, const double* g, double* x, double tol, int* iters,
                        double* resid, cudaStream_t s);
// the blocks' bounded meeting with a block missing: FC2D_ERR_TIMEOUT in *status after `limit` polls
fc2d_status launch_meet_probe(int* status, unsigned limit, cudaStream_t s);

}  // namespace fc2d
