#include "fx_tables.h"

#include <algorithm>
#include <cmath>
#include <mutex>

#include "sem_internal.h"

namespace sem {

void gll_points_ld(int N, std::vector<long double>& x) {
  std::vector<double> xd, w, D;
  gll(N, xd, w, D);
  x.assign(xd.begin(), xd.end());
  for (int i = 1; i < N; ++i)  // roots of P_{N-1} - x P_N, whose derivative is -(N + 1) P_N
    for (int it = 0; it < 4; ++it) {
      long double q = 1, p = x[i];  // P_{j-1}, P_j
      for (int j = 1; j < N; ++j) {
        const long double t = ((2 * j + 1) * x[i] * p - j * q) / (j + 1);
        q = p;
        p = t;
      }
      x[i] += (q - x[i] * p) / ((N + 1) * p);
    }
  for (int i = 0; i <= N - i; ++i) {
    const long double a = (x[N - i] - x[i]) / 2;
    x[i] = -a;
    x[N - i] = a;
  }
}

namespace {

// d = g 2^64 / (largest row sum of magnitudes): a contraction takes values below B to values below g B.  g = 0.8 keeps
// the sums of fx::dot below 2^63 for values of 60 bits (at worst 2^62.68, N = 9, for these tables; a caller that scales
// them checks the sums again); an odd n has a middle point whose
// entry stands for itself, and g = 0.5 keeps the entries below 2^63.
FxScale build(int N) {
  const int n = N + 1;
  FxScale f;
  std::vector<long double> x;
  gll_points_ld(N, x);
  f.D.assign((size_t)n * n, 0);
  for (int i = 0; i < n; ++i) {
    for (int l = 0; l < n; ++l) {
      if (l == i) continue;
      long double v = 1 / (x[l] - x[i]);
      for (int k = 0; k < n; ++k)
        if (k != i && k != l) v *= (x[i] - x[k]) / (x[l] - x[k]);
      f.D[i * n + l] = v;
    }
    long double s = 0;
    for (int l = 0; l < n; ++l) s += f.D[i * n + l];
    f.D[i * n + i] = -s;
  }
  f.w.resize(n);
  for (int i = 0; i < n; ++i) {  // w_i = 2 / (N (N + 1) P_N(x_i)^2)
    long double q = 1, p = x[i];
    for (int j = 1; j < N; ++j) {
      const long double t = ((2 * j + 1) * x[i] * p - j * q) / (j + 1);
      q = p;
      p = t;
    }
    f.w[i] = 2 / (N * (N + 1) * p * p);
  }
  f.M.assign((size_t)n * n, 0);
  long double rows = 0, rows_m = 0;
  for (int i = 0; i < n; ++i) {
    long double a = 0, b = 0;
    for (int l = 0; l < n; ++l) {
      f.M[i * n + l] = f.D[l * n + i] * f.w[l] / f.w[i];
      a += std::fabs(f.D[i * n + l]);
      b += std::fabs(f.M[i * n + l]);
    }
    rows = std::max(rows, a);
    rows_m = std::max(rows_m, b);
  }
  const long double g = std::ldexp(n % 2 ? 0.5L : 0.8L, 64);
  f.d = g / rows;
  f.dt = g / rows_m;
  int j = 0;
  const long double m = std::frexp(f.d * f.dt, &j);  // m in [1/2, 1)
  f.kappa = 1 / m;
  f.scale = 192 - j;
  return f;
}

}  // namespace

const FxScale& fx_scale(int N) {
  static std::once_flag once[kMaxN + 1];
  static FxScale table[kMaxN + 1];
  std::call_once(once[N], [N] { table[N] = build(N); });
  return table[N];
}

std::vector<double> fx_weights(int N) {
  const FxScale& f = fx_scale(N);
  const int n = N + 1;
  std::vector<double> W((size_t)n * n * n);
  for (int q = 0; q < n * n * n; ++q) W[q] = (double)(f.w[q % n] * f.w[q / n % n] * f.w[q / (n * n)] * f.kappa);
  return W;
}

}  // namespace sem
