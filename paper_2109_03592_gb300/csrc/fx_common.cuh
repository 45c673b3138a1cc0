// Parts of the fixed-point FP64 operators (ax_fx_impl.cuh, pressure_eo.cuh).
#pragma once

#include "fixed.cuh"
#include "kernels.h"

namespace sem {
namespace fxk {

using namespace fx;

constexpr int kExpMin = 1023 - 500, kExpMax = 1023 + 500;  // biased exponents of u on the integer path

// The values of an element share one exponent, FP64's do not: an element whose small values stand alone is evaluated in
// FP64.  w at a point is a sum over the three lines through it, so a small value does no harm where one of its lines has
// a larger one; a line is
//   good   its largest value lies at most kLineBits below the element's (less the factors' own range, FxOp::sG),
//   zero   all its values are zero or more than kNoiseBits below (the rounding of zeros such as sin(pi)),
//   small  otherwise,
// and the element is taken in FP64 if a point has small lines and no good one.  The integer path's error is then at most
// 2^(kLineBits - 7) of FP64's bound, which is reached at such points alone.  Emulated: no element of CG directions of
// smooth right-hand sides is, at any order; a Gaussian of 0.5 element widths has a quarter of its elements taken.
constexpr int kLineBits = 12, kNoiseBits = 44;
enum { kZeroLine, kSmallLine, kGoodLine };
__device__ __forceinline__ int line_state(int below, int range) {  // below: bits below the element's largest
  return below + range <= kLineBits ? kGoodLine : below > kNoiseBits ? kZeroLine : kSmallLine;
}

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
