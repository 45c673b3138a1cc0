// Parts of the fixed-point FP64 operators (ax_fx_impl.cuh, pressure_eo.cuh).
#pragma once

#include "fixed.cuh"
#include "kernels.h"

namespace sem {
namespace fxk {

using namespace fx;

constexpr int kExpMin = 1023 - 500, kExpMax = 1023 + 500;  // biased exponents of u on the integer path

// Maximum of v over an element's threads.  put() by every thread of the CTA, which is whole warps (so all 32 lanes meet
// in its warp operations, also behind a branch that some of them took), a barrier, then get(); `s` is one of the CTA's
// arrays, used once.  Where an element is whole warps each warp has a word of its own;
// otherwise the elements' words are cleared beforehand (clear(), and a barrier).
template <int T, int EPB>
struct ElemMax {
  static constexpr int kWarps = (EPB * T + 31) / 32;
  static constexpr bool whole = EPB == 1 || T % 32 == 0;
  static constexpr int size = whole ? kWarps : EPB;
  __device__ static __forceinline__ void clear(int* s) {
    if constexpr (!whole)
      for (int q = threadIdx.x; q < EPB; q += blockDim.x) s[q] = 0;
  }
  __device__ static __forceinline__ void put(int* s, int le, int v) {  // v >= 0
    if constexpr (whole) {
      v = __reduce_max_sync(0xffffffffu, v);
      if ((threadIdx.x & 31) == 0) s[threadIdx.x >> 5] = v;
    } else if constexpr (T < 32 && 32 % T == 0) {
#pragma unroll
      for (int o = T / 2; o > 0; o >>= 1) v = max(v, __shfl_xor_sync(0xffffffffu, v, o));
      if (threadIdx.x % T == 0) atomicMax(s + le, v);
    } else {
      atomicMax(s + le, v);
    }
  }
  __device__ static __forceinline__ int get(const int* s, int le) {
    if constexpr (!whole) return s[le];
    constexpr int w = EPB == 1 ? kWarps : T / 32;
    int v = s[EPB == 1 ? 0 : le * w];
#pragma unroll
    for (int q = 1; q < w; ++q) v = max(v, s[(EPB == 1 ? 0 : le * w) + q]);
    return v;
  }
};

// w at one point of an element in FP64, straight from memory (Alg. 1, with the factors taken back from their
// fixed-point form): for the rare element that the integer path does not cover.
template <int N>
__device__ __forceinline__ double slow_point(const AxParams<double>& P, const double* v, int64_t e, int i, int j, int k) {
  constexpr int n = N + 1, n2 = n * n, n3 = n2 * n;
  const double* ue = v + e * n3;
  const int sG = P.fx.sG[e];
  auto G = [&](int f, int a, int b, int c) {
    const int4 x = P.fx.G[(e * 3 + (f >> 1)) * n3 + a + n * b + n2 * c];
    const int2 y = (f & 1) ? make_int2(x.z, x.w) : make_int2(x.x, x.y);
    return ldexp(__ll2double_rn(shl(y.y, 32) + y.x), -sG) * (P.fx.wq[a] * P.fx.wq[b] * P.fx.wq[c]);
  };
  double out = 0.0;
#pragma unroll 1
  for (int d = 0; d < 3; ++d) {
#pragma unroll 1
    for (int l = 0; l < n; ++l) {
      const int a = d == 0 ? l : i, b = d == 1 ? l : j, c = d == 2 ? l : k;
      double ur = 0.0, us = 0.0, ut = 0.0;
#pragma unroll 1
      for (int q = 0; q < n; ++q) {
        ur += P.D[a * n + q] * ue[q + n * b + n2 * c];
        us += P.D[b * n + q] * ue[a + n * q + n2 * c];
        ut += P.D[c * n + q] * ue[a + n * b + n2 * q];
      }
      const int f0 = d == 0 ? 0 : d == 1 ? 3 : 4, f1 = d == 0 ? 3 : d == 1 ? 1 : 5, f2 = d == 0 ? 4 : d == 1 ? 5 : 2;
      const double w = G(f0, a, b, c) * ur + G(f1, a, b, c) * us + G(f2, a, b, c) * ut;
      out += P.D[l * n + (d == 0 ? i : d == 1 ? j : k)] * w;
    }
  }
  out *= P.h1;
  const int p = i + n * j + n2 * k;
  if (P.helm) out += P.h2 * P.B[e * n3 + p] * ue[p];
  return out;
}

// h2 B u of a point onto the stiffness part, both without the quadrature weights, in the coarser of the two terms' units.
// B has 62 bits below the element's largest, h2's mantissa (over kappa) 62, u 60; their product is taken to 59 bits.
struct MassTerm {
  int2 h2;
  int down;  // the mass term's unit over the stiffness part's is 2^-down
  // o (the stiffness part) + the mass term of B (fixed) and u
  __device__ __forceinline__ ll add(ll o, int2 B, int2 u) const {
    const int2 b[1] = {B}, hh[1] = {h2};
    const int2 hb = split(dot<1>(b, hh));  // at most 2^60
    const ll m = mad(mad(1ll << 28, hb.x, u.y), hb.y, u.x);
    const ll v = (((ll)hb.y * u.y) << 3) + (m >> 29);  // hb u / 2^61
    return down >= 0 ? o + (v >> min(down, 63)) : (o >> min(-down, 63)) + v;
  }
};

}  // namespace fxk
}  // namespace sem
