// Weak gradient and divergence of the pressure space, FP64 by fixed point.
#include "pressure_op.cuh"

namespace sem {

template cudaError_t launch_pgrad<double>(int, const PressureOp&, const double*, int64_t, double*, int64_t, cudaStream_t);
template cudaError_t launch_pdiv<double>(int, const PressureOp&, const double*, bool, int64_t, double*, int64_t,
                                         cudaStream_t);

cudaError_t launch_pressure_pack(void* F, int N, int64_t E, int* sF, int* bad, cudaStream_t s) {
  const int m = N - 1;
  const size_t smem = sizeof(double) * 9 * m * m * m;
  cudaError_t err = cudaFuncSetAttribute(peo::k_pack_fx, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem);
  if (err != cudaSuccess) return err;
  if (E > 0) peo::k_pack_fx<<<(unsigned)E, 256, smem, s>>>(static_cast<double*>(F), m, E, sF, bad);
  return cudaGetLastError();
}

bool pressure_weights(int N, std::vector<double>& grad, std::vector<double>& div) {
  const OrderTables* o = nullptr;
  switch (N) {
#define SEM_CASE(N) \
  case N: o = &order_tables<N>(); break;
    SEM_PRESSURE_ORDERS(SEM_CASE)
#undef SEM_CASE
    default: return false;
  }
  auto cube = [](const peo::Matrix& w, long double kappa, std::vector<double>& out) {
    const int n = (int)w.size();
    out.resize((size_t)n * n * n);
    for (int q = 0; q < n * n * n; ++q) out[q] = (double)(w[q % n] * w[q / n % n] * w[q / (n * n)] * kappa);
  };
  cube(fx_scale(N).w, o->scale.kappa_grad, grad);
  cube(o->rho, o->scale.kappa_div, div);
  return true;
}

}  // namespace sem
