// Weak gradient and divergence of the pressure space, FP64 by fixed point.
#include "pressure_op.cuh"

namespace sem {

template cudaError_t launch_pgrad<double>(int, const PressureOp&, const double*, int64_t, double*, int64_t, cudaStream_t);
template cudaError_t launch_pdiv<double>(int, const PressureOp&, const double*, bool, int64_t, double*, int64_t,
                                         cudaStream_t);

cudaError_t launch_pressure_pack(const double* F, int N, int64_t E, int2* Ffx, int* sF, int* bad, cudaStream_t s) {
  unsigned long long K = 0;
  switch (N) {
#define SEM_CASE(N) \
  case N: K = order_tables<N>().scale.K; break;
    SEM_PRESSURE_ORDERS(SEM_CASE)
#undef SEM_CASE
    default: return cudaErrorNotSupported;
  }
  if (E > 0) peo::k_pack_fx<<<(unsigned)E, 256, 0, s>>>(F, N - 1, E, K, Ffx, sF, bad);
  return cudaGetLastError();
}

}  // namespace sem
