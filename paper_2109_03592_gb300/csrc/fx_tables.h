// Host tables of the fixed-point FP64 operator (ax_fx_impl.cuh).
#pragma once

#include <vector>

namespace sem {

// D of order N in long double and the scales of its fixed-point tables: the tables are D d and D^T dt, the stored
// factors G kappa 2^sG with kappa = K / 2^63 = 2^j / (d dt) in [1, 2], and scale = 192 - j.
struct FxScale {
  std::vector<long double> D;  // [n][n]
  long double d, dt;
  unsigned long long K;
  int scale;
};
const FxScale& fx_scale(int N);  // N = 1 .. 11; built once per order

// GLL points of order N in long double.
void gll_points_ld(int N, std::vector<long double>& x);

}  // namespace sem
