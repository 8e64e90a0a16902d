// Plain types of the fixed-point DFT (fx.cuh) that the plan and its kernels share.
#pragma once

namespace fc2d {

// 1/(nx ny) for the fixed-point DFT: 2^exp (1 + m 2^-32 + r 2^-64), m = r = 0 for a power
// of two
struct FxFactor {
  int exp, m, r;
};

// Stages of a fixed-point DFT of length 2^a 3^b 5^c, and of columns of n1 n2 (fx_mixed.cuh)
constexpr int kFxMaxRadices = 16;
struct FxRadices {
  int n;
  signed char r[kFxMaxRadices];
};
struct FxMixed {
  FxRadices row, a, b;  // nx/2, n1, n2: at least one stage each (nx, ny >= 8)
  int n1, n2;           // ny = n1 n2, n2 the largest divisor up to sqrt(ny)
  int ta, tb;           // threads per column of both passes
};
FxMixed fx_mixed(int nx, int ny);

}  // namespace fc2d
