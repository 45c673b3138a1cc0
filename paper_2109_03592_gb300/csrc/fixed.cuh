// 64-bit fixed-point arithmetic on the integer pipe, for the operators whose
// results must be as accurate as FP64.
//
// GB300 issues 1.7 FP64 FMAs per clock and SM (measured), but 63 IMAD.WIDE
// (32 x 32 + 64 -> 64 bits).  A contraction of fixed-point numbers v = vh 2^32 +
// vl, c = ch 2^32 + cl (low halves signed) keeps the upper 64 bits of the
// 128-bit products:
//   sum_l c_l v_l / 2^64 = sum ch vh + (sum (ch vl + cl vh)) / 2^32 + O(1/4) per term,
// three IMAD.WIDE per multiply-add (6 issue slots; an FP32 pair needs 12
// instructions for 48 bits, a native FMA 60+ slots).  Values of one element share
// one exponent and are kept left-aligned at 60 bits, so the rounding of each
// stage is 2^-57 or less of the element's largest value.
#pragma once

#include <cuda_runtime.h>

#include <cstdint>

namespace sem {
namespace fx {

typedef long long ll;

constexpr int kBits = 60;   // magnitudes of fields: at most 2^60
constexpr int kOpExp = 200;  // exponents of G and B on the integer path lie within 2^+-200

// A 64-bit value split with a signed low half: v = y 2^32 + x (the register order of v itself).
__host__ __device__ __forceinline__ int2 split(ll v) {
  const int l = (int)v;
  return make_int2(l, (int)(v >> 32) + (int)((unsigned)l >> 31));
}

#ifdef __CUDACC__
// acc + a b.  As PTX: from the plain expression the compiler made two multiplies and a sign extension where an
// operand comes from constant memory (twice the instructions in the pressure kernels).
__device__ __forceinline__ ll mad(ll acc, int a, int b) {
  ll r;
  asm("mad.wide.s32 %0, %1, %2, %3;" : "=l"(r) : "r"(a), "r"(b), "l"(acc));
  return r;
}

// sum of c_l v_l / 2^64, rounded; the caller bounds 2^31 + sum (|cl vh| + |ch vl|) < 2^63.  fma_pipe: the upper products
// accumulate in the multiply-adds themselves (half their rate, no additions on the busier integer pipe); as mad() does
// it, the compiler adds them up apart.  Faster by 4 to 7% in kernels of even n, slower by 4% at n = 9.
template <int n, bool fma_pipe = true>
__device__ __forceinline__ ll dot(const int2 (&c)[n], const int2 (&v)[n]) {
  ll m = 0x80000000ll;
#pragma unroll
  for (int l = 0; l < n; ++l) {
    m = mad(m, c[l].x, v[l].y);
    m = mad(m, c[l].y, v[l].x);
  }
  ll r = m >> 32;
#pragma unroll
  for (int l = 0; l < n; ++l) r = fma_pipe ? r + (ll)c[l].y * v[l].y : mad(r, c[l].y, v[l].y);
  return r;
}

// Biased exponent (11 bits) of a double's high word.
__device__ __forceinline__ int expo(int hi) { return (hi >> 20) & 0x7ff; }

// x 2^(bits + 1022 - emax), truncated, for a finite x with biased exponent <= emax;
// entries below 2^-bits of 2^(emax - 1022) and denormals give 0 (emax > 64).
template <int bits = kBits>
__device__ __forceinline__ ll from_double(double x, int emax) {
  const int hi = __double2hiint(x);
  const unsigned lo = (unsigned)__double2loint(x);
  const unsigned long long m = ((unsigned long long)((hi & 0xfffff) | 0x100000) << 32) | lo;
  const int d = min(emax - expo(hi), 63);
  const ll v = (ll)((m << (bits - 53)) >> d);
  return hi < 0 ? -v : v;
}

// v 2^e, rounded to nearest; |e| small enough that the result is a normal number or 0.
__device__ __forceinline__ double to_double(ll v, int e) {
  const double d = __ll2double_rn(v);
  const double s = __hiloint2double(__double2hiint(d) + (e << 20), __double2loint(d));
  return v == 0 ? 0.0 : s;
}

__device__ __forceinline__ ll shl(ll v, int s) { return (ll)((unsigned long long)v << s); }
// bits that hold |hi word| of the largest value seen by `m` (m collects hi ^ (hi >> 31))
__device__ __forceinline__ int mag(ll v) {
  const int h = (int)(v >> 32);
  return h ^ (h >> 31);
}
__device__ __forceinline__ int bits_of(int m) { return 64 - __clz(m); }
#endif

}  // namespace fx
}  // namespace sem
