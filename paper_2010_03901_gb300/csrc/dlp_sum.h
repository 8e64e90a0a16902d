// Launches of the double-layer sums over a partition on the device (dlp_sum.cu).
#pragma once
#include <cuda_runtime.h>

#include "dlp_tree.h"

namespace fc2d {

struct DlpDev {
  int shift = 0, n_expand = 0, n_grid = 0, n_free = 0;
  const long long* nodes = nullptr;    // [N][2]
  const DlpBox* box = nullptr;
  const DlpSpan *expand = nullptr, *near = nullptr;
  const int32_t* chain = nullptr;
  const DlpLeaf* leaf = nullptr;
  const DlpItem *grid_items = nullptr, *free_items = nullptr;
  const long long* points = nullptr;   // [n][2] free points in leaf order
  const int32_t* points_idx = nullptr; // their places in the output
  unsigned long long* coef = nullptr;  // [n_box][kDlpOrder][2], zero before an expansion
  unsigned* mag = nullptr;             // largest magnitude of the node coefficients, zeroed likewise
};

// q = (x' + i y') phi / N per node, its double-float parts ab = (y' phi/N, x' phi/N)
void launch_node_coef(int N, const double* x1, const double* y1, const double* phi, double2* q,
                      float4* ab, unsigned* mag, cudaStream_t s);
void launch_dlp_expand(const DlpDev& d, const double2* q, cudaStream_t s);
// pos, ab: the nodes of the near terms
void launch_dlp_grid(const DlpDev& d, const int32_t* lin, int nx, double h, const float4* pos,
                     const float4* ab, double* u, cudaStream_t s);
void launch_dlp_free(const DlpDev& d, double h, const float4* pos, const float4* ab, double* out,
                     cudaStream_t s);

// u[lin] += Lagrange combination (weights w[n][MP]) of the trigonometric interpolant with
// coefficients ghat[0 .. Nb/2] (largest magnitude *mag) at the angles with e^{i theta} = z and
// vals[n][MP - 1]
void launch_close(int n, const int32_t* lin, const double2* z, const double* w, int MP,
                  const double* vals, int Nb, const double2* ghat, const unsigned* mag, double* u,
                  cudaStream_t s);

}  // namespace fc2d
