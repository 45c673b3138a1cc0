// Weak gradient and divergence of the pressure space in FP32.
#include "pressure_op.cuh"

namespace sem {

template cudaError_t launch_pgrad<float>(int, const PressureOp&, const float*, int64_t, float*, int64_t, cudaStream_t);
template cudaError_t launch_pdiv<float>(int, const PressureOp&, const float*, bool, int64_t, float*, int64_t, cudaStream_t);

cudaError_t launch_pressure_pack32(const PressureFactors& F, int N, int64_t E, float* F32, cudaStream_t s) {
  if (E > 0) peo::k_pack_f32<<<(unsigned)E, 256, 0, s>>>(F, N - 1, E, F32);
  return cudaGetLastError();
}

}  // namespace sem
