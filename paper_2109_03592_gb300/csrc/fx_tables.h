// Host tables of the fixed-point FP64 operator (ax_fx_impl.cuh).
#pragma once

#include <vector>

namespace sem {

// D of order N in long double, M = W^-1 D^T W (W: the GLL weights w) and the scales of their fixed-point tables D d and
// M dt, with 1 / (d dt) = kappa 2^-j, kappa in [1, 2], and scale = 192 - j.
struct FxScale {
  std::vector<long double> D, M;  // [n][n]
  std::vector<long double> w;     // [n]
  long double d, dt, kappa;
  int scale;
};
const FxScale& fx_scale(int N);  // N = 1 .. 11; built once per order

// w_i w_j w_k kappa of the points (FxOp::W64), [n^3].
std::vector<double> fx_weights(int N);

// GLL points of order N in long double.
void gll_points_ld(int N, std::vector<long double>& x);

}  // namespace sem
