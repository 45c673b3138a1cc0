// Weak gradient and divergence of the pressure space (included by pressure.cu;
// the operators are described there), as 1D contractions of whole lines in
// even-odd form, in FP32 or, for the FP64 operators, in 64-bit fixed point on the
// integer pipe (fixed.cuh).
//
// The GLL and GL points are symmetric about 0, so Ig[m-1-I][n-1-l] = Ig[I][l] and
// Dg (values of the derivative) changes sign: with P = v[l] + v[l'], M = v[l] - v[l']
//   A = sum_l E[I][l] P[l], B = sum_l O[I][l] M[l],  E, O = (X[I][l] +- X[I][l']) / 2,
//   (Ig v)[I], (Ig v)[I'] = A +- B;   (Dg v)[I], (Dg v)[I'] = B +- A
// (a middle point, where n or m is odd, has a P of its own and no M), and the
// transposes alike: half the multiply-adds of the plain form.  FP32 uses the plain form
// where the folds' roundings would put the error above its own: in the gradient's j- and
// k-stages (not what bounds it; E's error is then 8 to 18% below the plain form's on random
// elements) and everywhere for N <= 4 and N = 6 (E's error with folds 13 to 33% above at N = 3,
// 3 to 27% at N = 4, up to 4% at N = 6).  E and O are kernel
// parameters and every loop over them is unrolled, so they come from constant
// memory as operands of the multiply-adds; shared memory only carries the lines
// from one direction to the next.
//
// One thread per line and stage, EPB elements per CTA, n^2 threads each:
//   divergence  along k (from global memory, coalesced): XD = Dg v, XI = Ig v;
//               along j: Y0 = Ig XD, Y1 = Dg XI, Y2 = Ig XI;
//               along i: g_2 = Ig Y0, g_1 = Ig Y1, g_0 = Dg Y2, then the factors
//   gradient    the transposes in reverse order, with the terms that meet the same
//               next contraction added up; along k last, coalesced to global memory.
// Two barriers per velocity component.  The factors are stored as the threads of
// the i-stage read them: [e][a][I][b][K][J].
//
// Fixed point: v and p are brought to 60 bits below the element's (and component's)
// largest exponent, and so are lines that go from one stage to the next, for the orders
// where the stages' bounds, which no smooth or random field comes near, would cost more
// bits than FP64 loses (Shape).  Each table is scaled, not by a power of two, so that its largest
// row sum of magnitudes takes a value of 60 bits to less than 60 bits.  The factors are
// kept without the GL weights rho, with 62 bits below the largest of their element and
// component; the gradient's tables are W^-1 Ig^T rho and W^-1 Dg^T rho (W: the GLL weights),
// whose rows are alike in size, and its results are multiplied by the weights at the end,
// the divergence's by rho (as in ax_fx_impl.cuh, for the same reason); these carry the
// inverse of the scales.  The tables come from long-double GLL and GL points.  Error of E
// against 64 bits by emulation, random and smooth pressures on affine elements: 0.2 to 0.9
// times FP64's; of the gradient at its interior, face, edge and corner points 0.1 to 1.3 times
// (without the two measures 0.7 to 8 and up to 410 times, N = 5 to 11).
//
// What bounds them: fixed point, issue slots (9 in 10 instructions are multiply-adds, 64-bit additions and the
// splits between them) and the barriers between stages of different width; FP32, shared memory and DRAM (70% and
// 50% busy).  E = 32,768, N = 7: E in FP64 1.38 ms (0.28 TB/s of p, u and factors; 1.32 before the weights and the
// lines' lifts) against 8.76 ms on the FP64 pipe; E in FP32 350 us against 604 us for plain contractions with the
// matrices in shared memory.
//
// An element whose input is not finite, or whose exponents lie outside 2^+-500, is
// evaluated in FP64 (slow_div, slow_grad).
#pragma once

#include <algorithm>
#include <cmath>
#include <type_traits>
#include <vector>

#include "fixed.cuh"
#include "fx_common.cuh"
#include "pressure_factors.cuh"

namespace sem {
namespace peo {

using fx::ll;

__host__ __device__ constexpr int imax(int a, int b) { return a > b ? a : b; }

// Even-odd tables of one m x n matrix and its transpose, rows of the first half only.
template <class C, int N>
struct Table {
  static constexpr int n = N + 1, m = N - 1;
  C e[(m + 1) / 2][(n + 1) / 2], o[(m + 1) / 2][imax(n / 2, 1)];
  C te[(n + 1) / 2][(m + 1) / 2], to[(n + 1) / 2][imax(m / 2, 1)];
  C x[std::is_same<C, float>::value ? m : 1][n];  // FP32: the matrix itself
};

// ---- arithmetic ------------------------------------------------------------------

struct F32 {
  using In = float;   // fields in global memory
  using V = float;    // line values in registers and shared memory
  using C = float;    // multiply-add operands: table entries, factors, P and M
  static constexpr bool fixed = false;
  __device__ static __forceinline__ float operand(float v) { return v; }
  __device__ static __forceinline__ float factor(float c, float v) { return c * v; }
};

struct Fixed {
  using In = double;
  using V = ll;
  using C = int2;
  static constexpr bool fixed = true;
  // rounding of the terms of weight 2^-32 (fx::dot)
  __device__ static __forceinline__ ll half() { return 0x80000000ll; }
  __device__ static __forceinline__ int2 operand(ll v) { return fx::split(v); }
  // c v / 2^62
  __device__ static __forceinline__ ll factor(int2 c, int2 v) {
    const ll m = fx::mad(fx::mad(1ll << 29, c.x, v.y), c.y, v.x);
    return (((ll)c.y * v.y) << 2) + (m >> 30);
  }
};

constexpr int kFieldBits = fx::kBits;

template <class A, int N>
struct Shape {
  static constexpr int n = N + 1, m = N - 1, n2 = n * n, n3 = n2 * n, m2 = m * m, m3 = m2 * m;
  static constexpr int np = (n + 1) / 2, nm = n / 2, mp = (m + 1) / 2, mm = m / 2;  // P and M values of a line
  static constexpr bool plain = !A::fixed && (N <= 4 || N == 6);
  // Fixed point: where lines between stages are brought to 60 bits (gradient: after its first and second stage;
  // divergence: after its first).  Errors over FP64's by emulation, with and without: gradient's 0.4 to 1.3 and (N = 4)
  // 1.6 to (N = 10) 17; with one of the two 1.1 at N = 6 and 7, 2 to 3 above.  Divergence's 0.4 (N = 7) without, 1.1 at N = 6,
  // 1.9 at 8, 3.7 at 10, 1.3 at 11; 0.3 to 0.9 with.
  static constexpr bool grad_lift1 = A::fixed && N >= 4, grad_lift2 = A::fixed && N >= 6;
  static constexpr bool div_lift = A::fixed && (N == 6 || N >= 8);
  static constexpr int banks = 128 / (int)sizeof(typename A::V);
  // [K][j][i]: planes padded so that the threads (K, i) of the j-stage meet distinct banks
  static constexpr int sX = n2 + ((n - n2) % banks + banks) % banks;
  // [K][J][i]: odd rows, so that the threads (K, J) of the i-stage do
  static constexpr int rY = n | 1, sY = m * rY;
  static constexpr int elem = 2 * m * sX + 3 * m * sY;
  // Elements per CTA: the fewest warps per element over the three stages (a stage's last warp may be mostly
  // empty), where CTAs above 128 threads count 8% more (warps of small CTAs wait less at the barriers: E = 32,768,
  // N = 7, two elements: 1.38 ms FP64, 353 us FP32; four: 1.43 ms, 363 us; eight: 1.50 ms, 385 us).
  static constexpr int warps(int k) { return (k * n2 + 31) / 32 + (k * n * m + 31) / 32 + (k * m2 + 31) / 32; }
  static constexpr int best_epb() {
    int best = 1;
    long cost = 0;
    for (int k = 1; k * n2 <= 256 || k == 1; ++k) {
      const long c = 100000L * warps(k) * (k * n2 <= 128 ? 100 : 108) / k;
      if (k == 1 || c < cost) {
        cost = c;
        best = k;
      }
    }
    return best;
  }
  static constexpr int EPB = best_epb();
  static constexpr int threads = (EPB * n2 + 31) / 32 * 32;
  static constexpr size_t smem = sizeof(typename A::V) * (size_t)EPB * elem;
  // Resident threads per SM.  Fixed point, N = 7: the gradient 530 us with 512, 515 with 640; the divergence 622
  // and 654 (its spills).  The gradient of N = 2 and 3 fits 1152 (E at N = 2, 155,392 elements: 240 us, 264 with what the
  // compiler takes).
  static constexpr int grad_blocks = imax((A::fixed ? (N <= 3 ? 1152 : 640) : 1024) / threads, 1);
  static constexpr int div_blocks = imax((A::fixed ? 512 : 1024) / threads, 1);
};

template <class A, int N>
struct Params {
  const typename A::In* in;    // divergence: velocity, gradient: pressure
  typename A::In* out;
  const typename A::In* invB;  // reciprocal assembled mass (divergence), or null
  const typename A::C* F;
  const int* sF;               // fixed point: [E][3], the factors are F 2^sF
  PressureFactors f;           // for slow_div and slow_grad, with the matrices
  const double *Ig, *Dg;
  int64_t E, n_local;
  int scale;                   // fixed point: F C v = 2^scale W x the integers' product along the path, over 2^254
  const double* W;             // [n^3] (gradient) or [m^3]: the weights and the inverse of the scales
  int direct;                  // fixed point: every element in FP64 (factors out of range)
  Table<typename A::C, N> ig, dg;
};

// P and M of a line
template <class A, int L>
__device__ __forceinline__ void fold(const typename A::V (&v)[L], typename A::C (&p)[(L + 1) / 2],
                                     typename A::C (&q)[imax(L / 2, 1)]) {
#pragma unroll
  for (int l = 0; l < L / 2; ++l) {
    p[l] = A::operand(v[l] + v[L - 1 - l]);
    q[l] = A::operand(v[l] - v[L - 1 - l]);
  }
  if constexpr (L & 1) p[L / 2] = A::operand(v[L / 2]);
}

// sum_l c[l] v[l] over the first `count`
template <class A, int K>
__device__ __forceinline__ typename A::V dot(const typename A::C (&c)[K], const typename A::C (&v)[K], int count) {
  if constexpr (A::fixed) {
    ll m = A::half();
#pragma unroll
    for (int l = 0; l < K; ++l)
      if (l < count) m = fx::mad(fx::mad(m, c[l].x, v[l].y), c[l].y, v[l].x);
    ll r = m >> 32;  // the upper products: see fx::dot
#pragma unroll
    for (int l = 0; l < K; ++l)
      if (l < count) r = r + (ll)c[l].y * v[l].y;
    return r;
  } else {
    float s = 0.f;
#pragma unroll
    for (int l = 0; l < K; ++l)
      if (l < count) s = fmaf(c[l], v[l], s);
    return s;
  }
}

// sum_l c[l] v[l] + sum_l d[l] w[l] in fixed point; fx::dot's bound holds for each sum, not for both together
template <int K, int L>
__device__ __forceinline__ ll dot2(const int2 (&c)[K], const int2 (&v)[K], int nc, const int2 (&d)[L], const int2 (&w)[L],
                                   int nd) {
  ll m = Fixed::half(), k = Fixed::half();
#pragma unroll
  for (int l = 0; l < K; ++l)
    if (l < nc) m = fx::mad(fx::mad(m, c[l].x, v[l].y), c[l].y, v[l].x);
#pragma unroll
  for (int l = 0; l < L; ++l)
    if (l < nd) k = fx::mad(fx::mad(k, d[l].x, w[l].y), d[l].y, w[l].x);
  ll r = (m >> 32) + (k >> 32);
#pragma unroll
  for (int l = 0; l < K; ++l)
    if (l < nc) r = r + (ll)c[l].y * v[l].y;
#pragma unroll
  for (int l = 0; l < L; ++l)
    if (l < nd) r = r + (ll)d[l].y * w[l].y;
  return r;
}

// A row of the matrix times a line, and a column of it: the plain form (FP32).
template <int L>
__device__ __forceinline__ float row(const float (&x)[L], const float (&v)[L]) {
  float s = 0.f;
#pragma unroll
  for (int l = 0; l < L; ++l) s = fmaf(x[l], v[l], s);
  return s;
}
template <int M, int L>
__device__ __forceinline__ float column(const float (&x)[M][L], int l, const float (&v)[M]) {
  float s = 0.f;
#pragma unroll
  for (int r = 0; r < M; ++r) s = fmaf(x[r][l], v[r], s);
  return s;
}

// The most bits of an element's values, for the T threads of each of EPB elements: put by every thread of the CTA (those
// beyond the elements with le >= EPB or v = 0) onto a cleared word, a barrier, then lift().
template <int T, int EPB>
__device__ __forceinline__ void put_bits(int* s, int le, int v) {
  if constexpr (T >= 32) {  // a warp meets two elements at most
    const int first = __shfl_sync(0xffffffffu, le, 0), last = __shfl_sync(0xffffffffu, le, 31);
    const int a = __reduce_max_sync(0xffffffffu, le == first ? v : 0);
    const int b = __reduce_max_sync(0xffffffffu, le == first ? 0 : v);
    if ((threadIdx.x & 31) == 0) {
      if (first < EPB) atomicMax(s + first, a);
      if (last != first && last < EPB) atomicMax(s + last, b);
    }
  } else if (le < EPB) {
    atomicMax(s + le, v);
  }
}
// The shift that brings them to 60 bits.
__device__ __forceinline__ int lift(int bits) { return max(kFieldBits - bits, 0); }
template <int L>
__device__ __forceinline__ void lift_line(ll (&v)[L], int s) {
#pragma unroll
  for (int l = 0; l < L; ++l) v[l] = fx::shl(v[l], s);
}

template <class A, int L>
__device__ __forceinline__ void load_line(const typename A::V* s, int stride, typename A::V (&v)[L]) {
#pragma unroll
  for (int l = 0; l < L; ++l) v[l] = s[l * stride];
}

__device__ __forceinline__ void prefetch_l2(const void* p, size_t bytes) {  // a hint; 16-byte aligned ranges only
  if (((uintptr_t)p & 15u) || (bytes & 15u) || bytes == 0 || bytes >= (1ull << 31)) return;
  asm volatile("cp.async.bulk.prefetch.L2.global [%0], %1;" ::"l"(p), "r"((uint32_t)bytes) : "memory");
}

// One element's divergence in FP64, by the whole CTA; `sm` holds an element's lines.
template <int N>
__device__ __noinline__ void slow_div(const Params<Fixed, N>& P, int64_t e, double* sm) {
  constexpr int n = N + 1, m = N - 1, n2 = n * n, n3 = n2 * n, m2 = m * m, m3 = m2 * m;
  double *XI = sm, *XD = XI + m * n2, *Y0 = XD + m * n2, *Y1 = Y0 + m2 * n, *Y2 = Y1 + m2 * n;
#pragma unroll 1
  for (int a = 0; a < 3; ++a) {
    __syncthreads();
    for (int q = threadIdx.x; q < m * n2; q += blockDim.x) {
      const int K = q / n2, ji = q % n2;
      double xi = 0.0, xd = 0.0;
#pragma unroll 1
      for (int k = 0; k < n; ++k) {
        const int64_t g = e * n3 + k * n2 + ji;
        const double u = P.in[a * P.n_local + g], v = P.invB ? u * P.invB[g] : u;
        xi += P.Ig[K * n + k] * v;
        xd += P.Dg[K * n + k] * v;
      }
      XI[q] = xi;
      XD[q] = xd;
    }
    __syncthreads();
    for (int q = threadIdx.x; q < m2 * n; q += blockDim.x) {
      const int K = q / (m * n), J = q / n % m, i = q % n;
      double y0 = 0.0, y1 = 0.0, y2 = 0.0;
#pragma unroll 1
      for (int j = 0; j < n; ++j) {
        const double xi = XI[(K * n + j) * n + i], xd = XD[(K * n + j) * n + i];
        y0 += P.Ig[J * n + j] * xd;
        y1 += P.Dg[J * n + j] * xi;
        y2 += P.Ig[J * n + j] * xi;
      }
      Y0[q] = y0;
      Y1[q] = y1;
      Y2[q] = y2;
    }
    __syncthreads();
    for (int q = threadIdx.x; q < m3; q += blockDim.x) {
      const int KJ = q / m, I = q % m;
      double g0 = 0.0, g1 = 0.0, g2 = 0.0;
#pragma unroll 1
      for (int i = 0; i < n; ++i) {
        g0 += P.Dg[I * n + i] * Y2[KJ * n + i];
        g1 += P.Ig[I * n + i] * Y1[KJ * n + i];
        g2 += P.Ig[I * n + i] * Y0[KJ * n + i];
      }
      const double v = pressure_factor(P.f, m, e, 0, a, q) * g0 + pressure_factor(P.f, m, e, 1, a, q) * g1 +
                       pressure_factor(P.f, m, e, 2, a, q) * g2;
      double* o = P.out + e * m3 + q;
      *o = a == 0 ? v : *o + v;
    }
  }
}

// The hi words' magnitudes of a stage's results, for put_bits; nothing in FP32.
template <class... V>
__device__ __forceinline__ void note(int& mg, V... v) {
  if constexpr ((std::is_same<V, ll>::value && ...)) ((mg |= fx::mag(v)), ...);
}

template <int N>
__device__ __noinline__ void slow_grad(const Params<Fixed, N>& P, int64_t e, double* sm) {
  constexpr int n = N + 1, m = N - 1, n2 = n * n, n3 = n2 * n, m2 = m * m, m3 = m2 * m;
  double *S0 = sm, *S1 = S0 + m2 * n, *S2 = S1 + m2 * n, *AI = S2 + m2 * n, *AD = AI + m * n2;
#pragma unroll 1
  for (int a = 0; a < 3; ++a) {
    __syncthreads();
    for (int q = threadIdx.x; q < m2 * n; q += blockDim.x) {
      const int KJ = q / n, i = q % n;
      double s0 = 0.0, s1 = 0.0, s2 = 0.0;
#pragma unroll 1
      for (int I = 0; I < m; ++I) {
        const double p = P.in[e * m3 + KJ * m + I];
        s0 += P.Dg[I * n + i] * (pressure_factor(P.f, m, e, 0, a, KJ * m + I) * p);
        s1 += P.Ig[I * n + i] * (pressure_factor(P.f, m, e, 1, a, KJ * m + I) * p);
        s2 += P.Ig[I * n + i] * (pressure_factor(P.f, m, e, 2, a, KJ * m + I) * p);
      }
      S0[q] = s0;
      S1[q] = s1;
      S2[q] = s2;
    }
    __syncthreads();
    for (int q = threadIdx.x; q < m * n2; q += blockDim.x) {
      const int K = q / n2, j = q / n % n, i = q % n;
      double ai = 0.0, ad = 0.0;
#pragma unroll 1
      for (int J = 0; J < m; ++J) {
        const int s = (K * m + J) * n + i;
        ai += P.Dg[J * n + j] * S1[s] + P.Ig[J * n + j] * S0[s];
        ad += P.Ig[J * n + j] * S2[s];
      }
      AI[q] = ai;
      AD[q] = ad;
    }
    __syncthreads();
    for (int q = threadIdx.x; q < n3; q += blockDim.x) {
      const int k = q / n2, ji = q % n2;
      double u = 0.0;
#pragma unroll 1
      for (int K = 0; K < m; ++K) u += P.Ig[K * n + k] * AI[K * n2 + ji] + P.Dg[K * n + k] * AD[K * n2 + ji];
      P.out[a * P.n_local + e * n3 + q] = u;
    }
  }
}

// The element's exponent: of its largest value; an element of zeros takes the smallest one of the integer path.
__device__ __forceinline__ int element_expo(int ehi) { return ehi ? fx::expo(ehi) : fxk::kExpMin; }
__device__ __forceinline__ bool out_of_range(int ex) { return ex < fxk::kExpMin || ex > fxk::kExpMax; }

// q = sum_a sum_b F[b][a] C_b v_a, v_a = u_a invB or u_a.
template <class A, int N>
__global__ void __launch_bounds__(Shape<A, N>::threads, Shape<A, N>::div_blocks)
    k_pdiv(const __grid_constant__ Params<A, N> P) {
  using S = Shape<A, N>;
  using V = typename A::V;
  using C = typename A::C;
  using In = typename A::In;
  constexpr int n = S::n, m = S::m, n2 = S::n2, n3 = S::n3, m2 = S::m2, m3 = S::m3, EPB = S::EPB;
  extern __shared__ __align__(16) unsigned char sm_raw[];
  V* sm = reinterpret_cast<V*>(sm_raw);
  using Max = fxk::ElemMax<n2, EPB>;
  __shared__ int smax[3][A::fixed ? Max::size : 1];
  __shared__ int sbits[S::div_lift ? 3 * EPB : 1];  // of the lines between the stages, per component and element

  const int tid = threadIdx.x;
  const int64_t e0 = (int64_t)blockIdx.x * EPB;
  const int ne = (int)min((int64_t)EPB, P.E - e0);
  if (tid == 0) prefetch_l2(P.F + e0 * 9 * m3, sizeof(C) * (size_t)ne * 9 * m3);
  // this thread's line in the three stages
  const int le1 = min(tid / n2, EPB - 1), ji = tid % n2;
  const bool a1 = tid < ne * n2;
  const int le2 = tid / (n * m), K2 = tid % (n * m) / n, i2 = tid % n;
  const bool a2 = le2 < ne;
  const int le3 = tid / m2, KJ = tid % m2;
  const bool a3 = le3 < ne;
  auto XD = [&](int le) { return sm + le * S::elem; };
  auto Y0 = [&](int le) { return sm + le * S::elem + 2 * m * S::sX; };

  In raw[n];
  auto load = [&](int a) {
#pragma unroll
    for (int k = 0; k < n; ++k) raw[k] = In(0);
    if (a1) {
      const In* u = P.in + a * P.n_local + e0 * n3 + le1 * n3 + ji;
#pragma unroll
      for (int k = 0; k < n; ++k) raw[k] = u[k * n2];
      if (P.invB) {
        const In* b = P.invB + e0 * n3 + le1 * n3 + ji;
#pragma unroll
        for (int k = 0; k < n; ++k) raw[k] *= b[k * n2];
      }
    }
  };
  auto put_max = [&](int a) {
    if constexpr (A::fixed) {
      int ehi = 0;
#pragma unroll
      for (int k = 0; k < n; ++k) ehi = max(ehi, __double2hiint(raw[k]) & 0x7fffffff);
      Max::put(smax[a], le1, ehi);
    }
  };
  load(0);
  if constexpr (A::fixed) {
    for (int a = 0; a < 3; ++a) Max::clear(smax[a]);
    if constexpr (S::div_lift)
      for (int q = tid; q < 3 * EPB; q += blockDim.x) sbits[q] = 0;
    if (!Max::whole) __syncthreads();
    put_max(0);
    __syncthreads();
  }

  V o[m];
  int eo[S::mp];
  bool slow = A::fixed && P.direct;
#pragma unroll
  for (int I = 0; I < m; ++I) {
    o[I] = V(0);
    eo[I < m / 2 ? I : m - 1 - I] = 0;
  }
#pragma unroll 1
  for (int a = 0; a < 3; ++a) {
    int mg = 0;
    if (a1) {
      V v[n];
      if constexpr (A::fixed) {
        const int ex = element_expo(Max::get(smax[a], le1));
#pragma unroll
        for (int k = 0; k < n; ++k) v[k] = fx::from_double(raw[k], ex);
      } else {
#pragma unroll
        for (int k = 0; k < n; ++k) v[k] = raw[k];
      }
      V* x = XD(le1) + ji;
      if constexpr (S::plain) {
#pragma unroll
        for (int I = 0; I < m; ++I) {
          x[I * S::sX] = row(P.dg.x[I], v);
          x[(m + I) * S::sX] = row(P.ig.x[I], v);
        }
      } else {
      C p[S::np], q[imax(S::nm, 1)];
      fold<A, n>(v, p, q);
#pragma unroll
      for (int I = 0; I < S::mp; ++I) {
        const V dA = dot<A>(P.dg.e[I], p, S::np), dB = dot<A>(P.dg.o[I], q, S::nm), iA = dot<A>(P.ig.e[I], p, S::np), iB = dot<A>(P.ig.o[I], q, S::nm);
        x[I * S::sX] = dB + dA;
        x[(m + I) * S::sX] = iA + iB;
        if constexpr (S::div_lift) note(mg, dB + dA, iA + iB);
        if (2 * I + 1 != m) {
          x[(m - 1 - I) * S::sX] = dB - dA;
          x[(2 * m - 1 - I) * S::sX] = iA - iB;
          if constexpr (S::div_lift) note(mg, dB - dA, iA - iB);
        }
      }
      }
    }
    if constexpr (S::div_lift) put_bits<n2, EPB>(sbits + a * EPB, le1, a1 ? fx::bits_of(mg) : 0);
    if (a < 2) load(a + 1);
    __syncthreads();
    if (a2) {
      const V* x = XD(le2) + K2 * S::sX + i2;
      V* y = Y0(le2) + K2 * S::sY + i2;
      if constexpr (S::plain) {
        V d[n], v[n];
        load_line<A, n>(x, n, d);
        load_line<A, n>(x + m * S::sX, n, v);
#pragma unroll
        for (int J = 0; J < m; ++J) {
          y[J * S::rY] = row(P.ig.x[J], d);
          y[m * S::sY + J * S::rY] = row(P.dg.x[J], v);
          y[2 * m * S::sY + J * S::rY] = row(P.ig.x[J], v);
        }
      } else {
      C pd[S::np], qd[imax(S::nm, 1)], pi[S::np], qi[imax(S::nm, 1)];
      {
        V v[n];
        load_line<A, n>(x, n, v);
        if constexpr (S::div_lift) lift_line(v, lift(sbits[a * EPB + le2]));
        fold<A, n>(v, pd, qd);
        load_line<A, n>(x + m * S::sX, n, v);
        if constexpr (S::div_lift) lift_line(v, lift(sbits[a * EPB + le2]));
        fold<A, n>(v, pi, qi);
      }
#pragma unroll
      for (int J = 0; J < S::mp; ++J) {
        const V A0 = dot<A>(P.ig.e[J], pd, S::np), B0 = dot<A>(P.ig.o[J], qd, S::nm);
        const V A1 = dot<A>(P.dg.e[J], pi, S::np), B1 = dot<A>(P.dg.o[J], qi, S::nm);
        const V A2 = dot<A>(P.ig.e[J], pi, S::np), B2 = dot<A>(P.ig.o[J], qi, S::nm);
        y[J * S::rY] = A0 + B0;
        y[m * S::sY + J * S::rY] = B1 + A1;
        y[2 * m * S::sY + J * S::rY] = A2 + B2;
        if (2 * J + 1 != m) {
          y[(m - 1 - J) * S::rY] = A0 - B0;
          y[m * S::sY + (m - 1 - J) * S::rY] = B1 - A1;
          y[2 * m * S::sY + (m - 1 - J) * S::rY] = A2 - B2;
        }
      }
      }
    }
    if (a < 2) put_max(a + 1);
    __syncthreads();
    if (a3) {
      const V* y = Y0(le3) + KJ * S::rY;
      const C* F = P.F + ((e0 + le3) * 3 + a) * 3 * m3 + KJ;
      if constexpr (S::plain) {
        V v[3][n];  // along r, s, t
#pragma unroll
        for (int b = 0; b < 3; ++b) load_line<A, n>(y + (2 - b) * m * S::sY, 1, v[b]);
#pragma unroll
        for (int I = 0; I < m; ++I)
          o[I] = fmaf(__ldg(F + 3 * I * m2), row(P.dg.x[I], v[0]),
                      fmaf(__ldg(F + (3 * I + 1) * m2), row(P.ig.x[I], v[1]),
                           fmaf(__ldg(F + (3 * I + 2) * m2), row(P.ig.x[I], v[2]), o[I])));
      } else {
      C p[3][S::np], q[3][imax(S::nm, 1)];
#pragma unroll
      for (int b = 0; b < 3; ++b) {  // Y2, Y1, Y0: along r, s, t
        V v[n];
        load_line<A, n>(y + (2 - b) * m * S::sY, 1, v);
        fold<A, n>(v, p[b], q[b]);
      }
      int ex = 0;
      if constexpr (A::fixed) {
        const int ev = element_expo(Max::get(smax[a], le3));
        slow = slow || out_of_range(ev);
        ex = ev - 1022 - kFieldBits + P.scale + 1 - P.sF[(e0 + le3) * 3 + a];
        if constexpr (S::div_lift) ex -= lift(sbits[a * EPB + le3]);
      }
#pragma unroll
      for (int I = 0; I < S::mp; ++I) {
        const V A0 = dot<A>(P.dg.e[I], p[0], S::np), B0 = dot<A>(P.dg.o[I], q[0], S::nm);
        const V A1 = dot<A>(P.ig.e[I], p[1], S::np), B1 = dot<A>(P.ig.o[I], q[1], S::nm);
        const V A2 = dot<A>(P.ig.e[I], p[2], S::np), B2 = dot<A>(P.ig.o[I], q[2], S::nm);
        V g[2][3] = {{B0 + A0, A1 + B1, A2 + B2}, {B0 - A0, A1 - B1, A2 - B2}};
        constexpr bool odd = m & 1;
        const bool one = odd && I == m / 2;  // the middle point
        int up = 0, down = 0;
        if constexpr (A::fixed) {
          // the pair's values up to 60 bits (gradients are small against the terms that cancel in them), then
          // the products onto the coarser of the sum's and this component's units
          int mg = 0;
#pragma unroll
          for (int s = 0; s < 2; ++s)
#pragma unroll
            for (int b = 0; b < 3; ++b) mg |= fx::mag(g[s][b]);
          const int s = max(kFieldBits - fx::bits_of(mg), 0);
#pragma unroll
          for (int b = 0; b < 3; ++b) {
            g[0][b] = fx::shl(g[0][b], s);
            g[1][b] = fx::shl(g[1][b], s);
          }
          const int ep = ex - s;
          if (a == 0) eo[I] = ep;
          up = min(max(ep - eo[I], 0), 63);
          down = min(max(eo[I] - ep, 0), 63);
          eo[I] = max(eo[I], ep);
        }
#pragma unroll
        for (int s = 0; s < 2; ++s) {
          if (s == 1 && one) continue;
          const int q_ = s ? m - 1 - I : I;
          const C g0 = A::operand(g[s][0]), g1 = A::operand(g[s][1]), g2 = A::operand(g[s][2]);
          const C f0 = __ldg(F + (3 * q_) * m2), f1 = __ldg(F + (3 * q_ + 1) * m2), f2 = __ldg(F + (3 * q_ + 2) * m2);
          if constexpr (A::fixed) {  // sum of the three products / 2^63
            const ll lo = fx::mad(fx::mad(fx::mad(fx::mad(fx::mad(fx::mad(1ll << 30, f0.x, g0.y), f0.y, g0.x), f1.x, g1.y),
                                                  f1.y, g1.x), f2.x, g2.y), f2.y, g2.x);
            const ll hi = fx::mad(fx::mad((ll)f0.y * g0.y, f1.y, g1.y), f2.y, g2.y);
            o[q_] = (o[q_] >> up) + ((fx::shl(hi, 1) + (lo >> 31)) >> down);
          } else {
            o[q_] = fmaf(f0, g0, fmaf(f1, g1, fmaf(f2, g2, o[q_])));
          }
        }
      }
      }
    }
  }
  if (a3 && !slow) {
    In* out = P.out + (e0 + le3) * m3 + KJ * m;
#pragma unroll
    for (int I = 0; I < m; ++I) {
      if constexpr (A::fixed)
        out[I] = fx::to_double(o[I], eo[I < m / 2 ? I : m - 1 - I]) * __ldg(P.W + KJ * m + I);
      else
        out[I] = o[I];
    }
  }
  if constexpr (A::fixed) {
    if (__syncthreads_or(a3 && slow)) {
#pragma unroll 1
      for (int le = 0; le < ne; ++le) {
        bool s = P.direct;
        for (int a = 0; a < 3; ++a) s = s || out_of_range(element_expo(Max::get(smax[a], le)));
        if (s) slow_div<N>(P, e0 + le, reinterpret_cast<double*>(sm));
      }
    }
  }
}

// u_a = sum_b C_b^T (F[b][a] p) for a = 0, 1, 2 (local, unassembled).
template <class A, int N>
__global__ void __launch_bounds__(Shape<A, N>::threads, Shape<A, N>::grad_blocks)
    k_pgrad(const __grid_constant__ Params<A, N> P) {
  using S = Shape<A, N>;
  using V = typename A::V;
  using C = typename A::C;
  using In = typename A::In;
  constexpr int n = S::n, m = S::m, n2 = S::n2, n3 = S::n3, m2 = S::m2, m3 = S::m3, EPB = S::EPB;
  extern __shared__ __align__(16) unsigned char sm_raw[];
  V* sm = reinterpret_cast<V*>(sm_raw);
  __shared__ int smax[A::fixed ? EPB : 1];
  __shared__ int sbits[S::grad_lift1 ? 6 * EPB : 1];  // of the lines between the stages, two words per component and element

  const int tid = threadIdx.x;
  const int64_t e0 = (int64_t)blockIdx.x * EPB;
  const int ne = (int)min((int64_t)EPB, P.E - e0);
  if (tid == 0) prefetch_l2(P.F + e0 * 9 * m3, sizeof(C) * (size_t)ne * 9 * m3);
  const int le1 = tid / m2, KJ = tid % m2;
  const bool a1 = le1 < ne;
  const int le2 = tid / (n * m), K2 = tid % (n * m) / n, i2 = tid % n;
  const bool a2 = le2 < ne;
  const int le3 = tid / n2, ji = tid % n2;
  const bool a3 = le3 < ne;
  auto S0 = [&](int le) { return sm + le * S::elem; };
  auto AI = [&](int le) { return sm + le * S::elem + 3 * m * S::sY; };

  C pc[m];  // the thread's line of p, as operands
  {
    In p[m];
#pragma unroll
    for (int I = 0; I < m; ++I) p[I] = a1 ? P.in[(e0 + le1) * m3 + KJ * m + I] : In(0);
    if constexpr (A::fixed) {
      if (tid < EPB) smax[tid] = 0;
      if constexpr (S::grad_lift1)
        for (int q = tid; q < 6 * EPB; q += blockDim.x) sbits[q] = 0;
      __syncthreads();
      int ehi = 0;
#pragma unroll
      for (int I = 0; I < m; ++I) ehi = max(ehi, __double2hiint(p[I]) & 0x7fffffff);
      if (a1) atomicMax(smax + le1, ehi);
      __syncthreads();
      const int ex = a1 ? element_expo(smax[le1]) : 1023;
#pragma unroll
      for (int I = 0; I < m; ++I) pc[I] = fx::split(fx::from_double(p[I], ex));
    } else {
#pragma unroll
      for (int I = 0; I < m; ++I) pc[I] = p[I];
    }
  }
  int ex = 0;
  bool slow = A::fixed && P.direct;
  if constexpr (A::fixed) {
    if (a3) {
      ex = element_expo(smax[le3]);
      slow = slow || out_of_range(ex);
      ex += -1022 - kFieldBits + P.scale;
    }
  }

#pragma unroll 1
  for (int a = 0; a < 3; ++a) {
    int mg = 0;
    if (a1) {  // along I -> i: S0 = Dg^T t0, S1 = Ig^T t1, S2 = Ig^T t2, t_b = F[b][a] p
      const C* F = P.F + ((e0 + le1) * 3 + a) * 3 * m3 + KJ;
      V* s = S0(le1) + KJ * S::rY;
      if constexpr (S::plain) {
        V t[3][m];
#pragma unroll
        for (int b = 0; b < 3; ++b)
#pragma unroll
          for (int I = 0; I < m; ++I) t[b][I] = A::factor(__ldg(F + (3 * I + b) * m2), pc[I]);
#pragma unroll
        for (int i = 0; i < n; ++i) {
          s[i] = column(P.dg.x, i, t[0]);
          s[m * S::sY + i] = column(P.ig.x, i, t[1]);
          s[2 * m * S::sY + i] = column(P.ig.x, i, t[2]);
        }
      } else {
      C p[3][S::mp], q[3][imax(S::mm, 1)];
#pragma unroll
      for (int b = 0; b < 3; ++b) {
        V t[m];
#pragma unroll
        for (int I = 0; I < m; ++I) t[I] = A::factor(__ldg(F + (3 * I + b) * m2), pc[I]);
        fold<A, m>(t, p[b], q[b]);
      }
#pragma unroll
      for (int i = 0; i < S::np; ++i) {
        const V A0 = dot<A>(P.dg.te[i], p[0], S::mp), B0 = dot<A>(P.dg.to[i], q[0], S::mm);
        const V A1 = dot<A>(P.ig.te[i], p[1], S::mp), B1 = dot<A>(P.ig.to[i], q[1], S::mm);
        const V A2 = dot<A>(P.ig.te[i], p[2], S::mp), B2 = dot<A>(P.ig.to[i], q[2], S::mm);
        s[i] = B0 + A0;
        s[m * S::sY + i] = A1 + B1;
        s[2 * m * S::sY + i] = A2 + B2;
        if constexpr (S::grad_lift1) note(mg, B0 + A0, A1 + B1, A2 + B2);
        if (2 * i + 1 != n) {
          s[n - 1 - i] = B0 - A0;
          s[m * S::sY + n - 1 - i] = A1 - B1;
          s[2 * m * S::sY + n - 1 - i] = A2 - B2;
          if constexpr (S::grad_lift1) note(mg, B0 - A0, A1 - B1, A2 - B2);
        }
      }
      }
    }
    if constexpr (S::grad_lift1) put_bits<m2, EPB>(sbits + 2 * a * EPB, le1, a1 ? fx::bits_of(mg) : 0);
    mg = 0;
    __syncthreads();
    if (a2) {  // along J -> j: AI = Ig^T S0 + Dg^T S1, AD = Ig^T S2
      const V* s = S0(le2) + K2 * S::sY + i2;
      V* x = AI(le2) + K2 * S::sX + i2;
      if constexpr (!A::fixed) {
        V v[3][m];
#pragma unroll
        for (int b = 0; b < 3; ++b) load_line<A, m>(s + b * m * S::sY, S::rY, v[b]);
#pragma unroll
        for (int j = 0; j < n; ++j) {
          V ai = 0.f, ad = 0.f;
#pragma unroll
          for (int J = 0; J < m; ++J) {
            ai = fmaf(P.dg.x[J][j], v[1][J], ai);
            ai = fmaf(P.ig.x[J][j], v[0][J], ai);
            ad = fmaf(P.ig.x[J][j], v[2][J], ad);
          }
          x[j * n] = ai;
          x[m * S::sX + j * n] = ad;
        }
      } else {
      C p[3][S::mp], q[3][imax(S::mm, 1)];
#pragma unroll
      for (int b = 0; b < 3; ++b) {
        V v[m];
        load_line<A, m>(s + b * m * S::sY, S::rY, v);
        if constexpr (S::grad_lift1) lift_line(v, lift(sbits[2 * a * EPB + le2]));
        fold<A, m>(v, p[b], q[b]);
      }
#pragma unroll
      for (int j = 0; j < S::np; ++j) {
        const ll Ev = dot2(P.ig.te[j], p[0], S::mp, P.dg.to[j], q[1], S::mm);
        const ll Od = dot2(P.dg.te[j], p[1], S::mp, P.ig.to[j], q[0], S::mm);
        const ll A2 = dot<A>(P.ig.te[j], p[2], S::mp), B2 = dot<A>(P.ig.to[j], q[2], S::mm);
        x[j * n] = Ev + Od;
        x[m * S::sX + j * n] = A2 + B2;
        if constexpr (S::grad_lift2) note(mg, Ev + Od, A2 + B2);
        if (2 * j + 1 != n) {
          x[(n - 1 - j) * n] = Ev - Od;
          x[m * S::sX + (n - 1 - j) * n] = A2 - B2;
          if constexpr (S::grad_lift2) note(mg, Ev - Od, A2 - B2);
        }
      }
      }
    }
    if constexpr (S::grad_lift2) put_bits<n * m, EPB>(sbits + (2 * a + 1) * EPB, le2, a2 ? fx::bits_of(mg) : 0);
    __syncthreads();
    if (a3) {  // along K -> k: u = Ig^T AI + Dg^T AD
      const V* x = AI(le3) + ji;
      In* u = P.out + a * P.n_local + (e0 + le3) * n3 + ji;
      if constexpr (!A::fixed) {
        V v[2][m];
#pragma unroll
        for (int b = 0; b < 2; ++b) load_line<A, m>(x + b * m * S::sX, S::sX, v[b]);
#pragma unroll
        for (int k = 0; k < n; ++k) {
          V w = 0.f;
#pragma unroll
          for (int K = 0; K < m; ++K) {
            w = fmaf(P.dg.x[K][k], v[1][K], w);
            w = fmaf(P.ig.x[K][k], v[0][K], w);
          }
          u[k * n2] = w;
        }
      } else {
      C p[2][S::mp], q[2][imax(S::mm, 1)];
#pragma unroll
      for (int b = 0; b < 2; ++b) {
        V v[m];
        load_line<A, m>(x + b * m * S::sX, S::sX, v);
        if constexpr (S::grad_lift2) lift_line(v, lift(sbits[(2 * a + 1) * EPB + le3]));
        fold<A, m>(v, p[b], q[b]);
      }
      int eu = ex - P.sF[(e0 + le3) * 3 + a];
      if constexpr (S::grad_lift1) eu -= lift(sbits[2 * a * EPB + le3]);
      if constexpr (S::grad_lift2) eu -= lift(sbits[(2 * a + 1) * EPB + le3]);
#pragma unroll
      for (int k = 0; k < S::np; ++k) {
        const ll Ev = dot2(P.ig.te[k], p[0], S::mp, P.dg.to[k], q[1], S::mm);
        const ll Od = dot2(P.dg.te[k], p[1], S::mp, P.ig.to[k], q[0], S::mm);
        if (!slow) {
          u[k * n2] = fx::to_double(Ev + Od, eu) * __ldg(P.W + ji + k * n2);
          if (2 * k + 1 != n) u[(n - 1 - k) * n2] = fx::to_double(Ev - Od, eu) * __ldg(P.W + ji + (n - 1 - k) * n2);
        }
      }
      }
    }
  }
  if constexpr (A::fixed) {
    if (__syncthreads_or(a3 && slow)) {
#pragma unroll 1
      for (int le = 0; le < ne; ++le)
        if (P.direct || out_of_range(element_expo(smax[le]))) slow_grad<N>(P, e0 + le, reinterpret_cast<double*>(sm));
    }
  }
}

// The factors F[b][a](q) in FP32, as the kernels read them.
static __global__ void __launch_bounds__(256) k_pack_f32(const PressureFactors F, int m, int64_t E, float* __restrict__ out) {
  const int m2 = m * m, m3 = m2 * m;
  const int64_t e = blockIdx.x;
  for (int r = threadIdx.x; r < 9 * m3; r += blockDim.x) {
    const int KJ = r % m2, b = r / m2 % 3, I = r / (3 * m2) % m, a = r / (3 * m3);
    out[e * 9 * m3 + r] = (float)pressure_factor(F, m, e, b, a, KJ * m + I);
  }
}

// F [3 (b)][3 (a)][m^3] of an element, without the GL weights, into its fixed-point form in place: 62 bits below the
// largest of the element and component; *bad where an exponent lies outside 2^+-kOpExp.
static __global__ void __launch_bounds__(256) k_pack_fx(double* F, int m, int64_t E, int* __restrict__ sF, int* bad) {
  extern __shared__ double f[];  // [9 m^3]
  __shared__ int top[3];
  const int m2 = m * m, m3 = m2 * m;
  const int64_t e = blockIdx.x;
  if (threadIdx.x < 3) top[threadIdx.x] = 0;
  __syncthreads();
  for (int r = threadIdx.x; r < 9 * m3; r += blockDim.x) {
    f[r] = F[e * 9 * m3 + r];
    atomicMax(top + r / m3 % 3, __double2hiint(f[r]) & 0x7fffffff);
  }
  __syncthreads();
  if (threadIdx.x < 3) {
    const int x = fx::expo(top[threadIdx.x]);
    if (abs(x - 1023) > fx::kOpExp) atomicExch(bad, 1);
    sF[e * 3 + threadIdx.x] = 62 + 1022 - x;
  }
  for (int r = threadIdx.x; r < 9 * m3; r += blockDim.x) {
    const int KJ = r % m2, b = r / m2 % 3, I = r / (3 * m2) % m, a = r / (3 * m3);
    reinterpret_cast<int2*>(F)[e * 9 * m3 + r] = fx::split(fx::from_double<62>(f[(3 * b + a) * m3 + KJ * m + I], fx::expo(top[a])));
  }
}

// ---- host: the tables, from Ig and Dg [m][n] and the GL and GLL weights ---------------

typedef std::vector<long double> Matrix;

// Of one order: the gradient's matrices W^-1 Ig^T rho and W^-1 Dg^T rho [n][m], the scales of all four tables, and
// Params::scale and the inverse of the scales that W carries, for both operators.
struct Scale {
  Matrix gi, gd;
  long double s_ig, s_dg, s_gi, s_gd;
  int scale_div, scale_grad;
  long double kappa_div, kappa_grad;
};

// sigma = g 2^64 / (largest row sum of magnitudes): a contraction takes values below B to values below g B.  With g = 0.8
// (divergence) and 0.62 (gradient, where two results are added: 1.24 B) and B = 2^60 every sum of fx::dot stays
// below 2^63 (at worst 2^62.69, N = 11), also for the folds of the last contraction's 1.24 B.  Odd n has a middle
// point whose entry stands for itself: g = 0.5 there keeps the entries below 2^63.
inline Scale table_scale(int N, const Matrix& Ig, const Matrix& Dg, const Matrix& rho, const Matrix& w) {
  const int n = N + 1, m = N - 1;
  auto sigma = [&](const Matrix& X, int rows, int len, long double g) {
    long double top = 0;
    for (int r = 0; r < rows; ++r) {
      long double s = 0;
      for (int l = 0; l < len; ++l) s += std::fabs(X[r * len + l]);
      top = std::max(top, s);
    }
    return std::ldexp(n % 2 ? 0.5L * (1 - 0x1p-20L) : g, 64) / top;
  };
  Scale s;
  s.gi.resize(n * m);
  s.gd.resize(n * m);
  for (int i = 0; i < n; ++i)
    for (int I = 0; I < m; ++I) {
      s.gi[i * m + I] = Ig[I * n + i] * rho[I] / w[i];
      s.gd[i * m + I] = Dg[I * n + i] * rho[I] / w[i];
    }
  s.s_ig = sigma(Ig, m, n, 0.8L);
  s.s_dg = sigma(Dg, m, n, 0.8L);
  s.s_gi = sigma(s.gi, n, m, 0.62L);
  s.s_gd = sigma(s.gd, n, m, 0.62L);
  auto inverse = [](long double i, long double d, int& scale) {
    int j = 0;
    const long double f = std::frexp(i * i * d, &j);  // f 2^j, f in [1/2, 1)
    scale = 3 * 64 + 62 - j;
    return 1 / f;
  };
  s.kappa_div = inverse(s.s_ig, s.s_dg, s.scale_div);
  s.kappa_grad = inverse(s.s_gi, s.s_gd, s.scale_grad);
  return s;
}

// The tables of X [m][n] and, for the transposes, of Y [n][m].
template <class A, int N>
Table<typename A::C, N> make_table(const Matrix& X, long double sx, const Matrix& Y, long double sy) {
  constexpr int n = N + 1, m = N - 1;
  Table<typename A::C, N> t{};
  auto fill = [&](const Matrix& M, long double s, int rows, int len, auto& e, auto& o) {
    auto conv = [&](long double v) {
      if constexpr (A::fixed)
        return fx::split(std::llround(v * s));
      else
        return (float)v;
    };
    auto at = [&](int r, int l) { return M[r * len + l]; };
    for (int r = 0; r < (rows + 1) / 2; ++r) {
      for (int l = 0; l < len / 2; ++l) {
        e[r][l] = conv((at(r, l) + at(r, len - 1 - l)) / 2);
        o[r][l] = conv((at(r, l) - at(r, len - 1 - l)) / 2);
      }
      if (len & 1) e[r][len / 2] = conv(at(r, len / 2));
    }
  };
  if constexpr (!A::fixed)
    for (int r = 0; r < m; ++r)
      for (int l = 0; l < n; ++l) t.x[r][l] = (float)X[r * n + l];
  fill(X, sx, m, n, t.e, t.o);
  fill(Y, sy, n, m, t.te, t.to);
  return t;
}

}  // namespace peo
}  // namespace sem
