// Launchers of the weak gradient and divergence (pressure_eo.cuh), included by the two translation units that
// instantiate them (pressure_op64.cu in fixed point, pressure_op32.cu in FP32).
#pragma once

#include <type_traits>
#include <vector>

#include "fx_tables.h"
#include "kernels.h"
#include "pressure_eo.cuh"
#include "sem_internal.h"

namespace sem {
namespace {
template <typename T>
using Arith = std::conditional_t<std::is_same<T, double>::value, peo::Fixed, peo::F32>;

struct OrderTables {
  peo::Matrix Ig, Dg, rho, igt, dgt;  // igt, dgt: the transposes
  peo::Scale scale;
  explicit OrderTables(int N) {
    gl_matrices_ld(N, Ig, Dg, rho);
    scale = peo::table_scale(N, Ig, Dg, rho, fx_scale(N).w);
    const int n = N + 1, m = N - 1;
    igt.resize(n * m);
    dgt.resize(n * m);
    for (int q = 0; q < n * m; ++q) {
      igt[q] = Ig[q % m * n + q / m];
      dgt[q] = Dg[q % m * n + q / m];
    }
  }
};
template <int N>
const OrderTables& order_tables() {
  static const OrderTables t(N);
  return t;
}

// The parameters that depend on the order and the mesh alone.
template <typename T, int N>
peo::Params<Arith<T>, N> pressure_params(bool grad, const PressureOp& op, int64_t E, int64_t n_local) {
  using A = Arith<T>;
  const OrderTables& o = order_tables<N>();
  const peo::Scale& c = o.scale;
  static const auto ig = peo::make_table<A, N>(o.Ig, c.s_ig, A::fixed ? c.gi : o.igt, c.s_gi),
                    dg = peo::make_table<A, N>(o.Dg, c.s_dg, A::fixed ? c.gd : o.dgt, c.s_gd);
  peo::Params<A, N> p{};
  if constexpr (A::fixed) {
    p.F = static_cast<const int2*>(op.f.data);
    p.sF = op.f.sF;
    p.f = op.f;
    p.Ig = op.Ig;
    p.Dg = op.DIg;
    p.scale = grad ? c.scale_grad : c.scale_div;
    p.W = grad ? op.Wgrad : op.Wdiv;
    p.direct = op.f.direct;
  } else {
    p.F = op.F32;
  }
  p.E = E;
  p.n_local = n_local;
  p.ig = ig;
  p.dg = dg;
  return p;
}

template <typename T, int N>
cudaError_t launch_pressure(bool grad, const peo::Params<Arith<T>, N>& p, cudaStream_t s) {
  using A = Arith<T>;
  using S = peo::Shape<A, N>;
  static DeviceOnce once;
  cudaError_t err = once.get([&](int, int*) {
    cudaError_t e = cudaFuncSetAttribute(peo::k_pgrad<A, N>, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)S::smem);
    if (e != cudaSuccess) return e;
    return cudaFuncSetAttribute(peo::k_pdiv<A, N>, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)S::smem);
  });
  if (err != cudaSuccess) return err;
  if (p.E == 0) return cudaSuccess;
  const unsigned grid = (unsigned)((p.E + S::EPB - 1) / S::EPB);
  if (grad)
    peo::k_pgrad<A, N><<<grid, S::threads, S::smem, s>>>(p);
  else
    peo::k_pdiv<A, N><<<grid, S::threads, S::smem, s>>>(p);
  return cudaGetLastError();
}
}  // namespace

#define SEM_PRESSURE_ORDERS(X) X(2) X(3) X(4) X(5) X(6) X(7) X(8) X(9) X(10) X(11)

template <typename T>
cudaError_t launch_pgrad(int N, const PressureOp& op, const T* p, int64_t E, T* u, int64_t n_local, cudaStream_t s) {
  switch (N) {
#define SEM_CASE(N)                                           \
  case N: {                                                   \
    auto a = pressure_params<T, N>(true, op, E, n_local);           \
    a.in = p;                                                 \
    a.out = u;                                                \
    return launch_pressure<T, N>(true, a, s);                 \
  }
    SEM_PRESSURE_ORDERS(SEM_CASE)
#undef SEM_CASE
    default: return cudaErrorNotSupported;
  }
}

template <typename T>
cudaError_t launch_pdiv(int N, const PressureOp& op, const T* u, bool scaled, int64_t E, T* out, int64_t n_local,
                        cudaStream_t s) {
  const T* invB = nullptr;
  if (scaled) {
    if constexpr (std::is_same<T, double>::value)
      invB = op.invB;
    else
      invB = op.invB32;
  }
  switch (N) {
#define SEM_CASE(N)                                           \
  case N: {                                                   \
    auto a = pressure_params<T, N>(false, op, E, n_local);           \
    a.in = u;                                                 \
    a.out = out;                                              \
    a.invB = invB;                                            \
    return launch_pressure<T, N>(false, a, s);                \
  }
    SEM_PRESSURE_ORDERS(SEM_CASE)
#undef SEM_CASE
    default: return cudaErrorNotSupported;
  }
}

}  // namespace sem
