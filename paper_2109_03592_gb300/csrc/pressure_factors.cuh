// A factor of the pressure operators in FP64, from the form that the mesh keeps them in (PressureFactors).
#pragma once

#include "fixed.cuh"
#include "kernels.h"

namespace sem {

// F[b][a] at the GL point q = (K m + J) m + I of element e
__device__ __forceinline__ double pressure_factor(const PressureFactors& f, int m, int64_t e, int b, int a, int q) {
  const int m2 = m * m, m3 = m2 * m;
  if (f.direct) return static_cast<const double*>(f.data)[(e * 9 + 3 * b + a) * m3 + q];
  const int I = q % m, KJ = q / m;
  const int2 x = static_cast<const int2*>(f.data)[(((e * 3 + a) * m + I) * 3 + b) * m2 + KJ];
  const double w = f.rho[I] * f.rho[KJ % m] * f.rho[KJ / m];
  return w * ldexp(__ll2double_rn(fx::shl(x.y, 32) + x.x), -f.sF[e * 3 + a]);
}

}  // namespace sem
