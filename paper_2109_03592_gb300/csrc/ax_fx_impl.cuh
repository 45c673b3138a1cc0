// FP64 local operator (Alg. 1 + h2 mass term) in 64-bit fixed point on the
// integer pipe (fixed.cuh), any n = N + 1.
//
// One thread per line: n^2 threads per element, each of which contracts the
// t-line (i, j), the r-line (j, k) and the s-line (i, k) of its two indices, every
// line in even-odd form (D and D^T are centro-antisymmetric): with P = v[l] + v[l'],
// M = v[l] - v[l'], l' = n-1-l,
//   A = sum_l E[i][l] P[l], B = sum_l O[i][l] M[l];  (D v)[i], (D v)[i'] = B +- A
// (the middle point of an odd n stands for itself).  A line's n loads and 2 (n/2)
// folds serve n outputs, and the tables are kernel parameters under unrolled loops, so
// they are constant operands of the multiply-adds (fx::mad); t-lines stay in registers.
//
// Quadrature weights: A = D^T W G D = W M G D with M = W^-1 D^T W, whose entries are as large as D's (off the diagonal
// they are -D's).  So the factors are kept without the weights, which multiply the result of a point at the end: they
// fall by up to 7000 (N = 11) from an element's middle to its corners, and all values that share an exponent would carry
// that.  Error against 64 bits over FP64's own, by emulation, at the corners: 0.4 (N = 11, random u; 340 with D^T W G D);
// inside elements 0.1 to 1.3 (0.2 to 1.8).  The weights take 2% more time at N = 7, E = 262,144, none or less elsewhere.
//
// Scaling: u is brought to 60 bits below the element's largest exponent, the
// gradients once more (those of smooth fields are small against the terms of D that
// cancel), and so is G grad u; each table is scaled, not by a power of two, so that its
// largest row sum of magnitudes keeps 60 bits within 60 bits, and the weights
// carry the inverse of the scales, with 62 bits.  The tables come from long-double GLL
// points (fx_tables.cpp).
//
// An element whose values are not finite, whose exponents lie outside the range
// that the shifts are written for (2^-500 .. 2^500), or whose small values stand
// alone beside large ones (line_state) is evaluated in FP64 (element_fp64).
//
// What bounds it: issue, of multiply-adds and of the additions between them (integer pipe 50% busy, multiply pipe
// 35%, FP64 19%, DRAM 49%).  One thread per 2x2x2 octant instead of per line needed twice the shared-memory reads and splits
// (N = 7, E = 32,768: 361 us; this kernel 274 with the weights in the factors and without the checks of small values, 285
// with both as they are, 3.8 TB/s of u, G and w; even-odd FP32 pairs 407, the FP64 pipe 1900; odd n, column threads
// without the fold, N = 8, E = 22,528: 660; this kernel 312 and 327).  The Helmholtz term, from B in fixed point loaded ahead of the
// stores of w, adds 12% (308 us; converted from FP64 at each use, 25%).  Not kept: the r- and s-lines
// through one copy of the code in a loop (no faster at N = 7, 4 to 11% slower above).
#pragma once

#include <algorithm>
#include <cmath>
#include <cstdlib>
#include <iterator>

#include "ax_eo_impl.cuh"
#include "ax_impl.cuh"
#include "fixed.cuh"
#include "fx_common.cuh"
#include "fx_tables.h"

namespace sem {
namespace fxk {

// Even-odd tables of D and of M = W^-1 D^T W (rows of the first half).
template <int N>
struct LineTable {
  static constexpr int n = N + 1, np = (n + 1) / 2, nm = n / 2;
  int2 e[np][np], o[np][nm], te[np][np], to[np][nm];
};

template <int N>
struct LineParams {
  AxParams<double> a;
  int scale;  // FxScale::scale and the exponent of h1
  int2 h2;    // the mantissa of h2 / kappa, 62 bits, and its exponent
  int e2;
  int mass_limit;  // sG - sB beyond which the mass term outweighs the stiffness and is added in FP64
  LineTable<N> d;
};

// One element's values in shared memory.  A half-warp's 8-byte accesses are free of bank conflicts where the 16
// threads meet distinct banks.  n = 8: rows swapped in pairs and XOR-swizzled, so that all three line directions do;
// other n: rows padded to odd length (t- and r-lines; s-lines nearly).
template <int n>
struct LineLayout {
  static constexpr bool swz = n == 8;
  static constexpr int row = swz ? 8 : n | 1, plane = n * row, size = n * plane;
  __device__ static __forceinline__ int idx(int i, int j, int k) {
    if constexpr (swz) return k * 64 + (j ^ (k & 1)) * 8 + (i ^ ((j >> 1) + 4 * (k & 1)));
    return k * plane + j * row + i;
  }
};

template <int n>
__device__ __forceinline__ void fold(const ll (&v)[n], int2 (&p)[(n + 1) / 2], int2 (&m)[n / 2]) {
#pragma unroll
  for (int l = 0; l < n / 2; ++l) {
    p[l] = split(v[l] + v[n - 1 - l]);
    m[l] = split(v[l] - v[n - 1 - l]);
  }
  if constexpr (n & 1) p[n / 2] = split(v[n / 2]);
}

// out = (table) v
template <int n>
__device__ __forceinline__ void contract(const int2 (&e)[(n + 1) / 2][(n + 1) / 2], const int2 (&o)[(n + 1) / 2][n / 2],
                                         const ll (&v)[n], ll (&out)[n]) {
  constexpr int np = (n + 1) / 2;
  int2 p[np], m[n / 2];
  fold<n>(v, p, m);
#pragma unroll
  for (int r = 0; r < np; ++r) {
    const ll B = dot<n / 2, n % 2 == 0>(o[r], m);
    if ((n & 1) && r == n / 2) {  // antisymmetric: the middle row has no even part
      out[r] = B;
    } else {
      const ll A = dot<np, n % 2 == 0>(e[r], p);
      out[r] = B + A;
      out[n - 1 - r] = B - A;
    }
  }
}

// Whether a point of the t-line (x, y) of u has small lines and no good one (line_state); *alone tells whether any of the
// element has.  By all threads of the CTA, one to a t-line.  rows (4 n words): the r-lines (j, k) that are not good in bit
// k of row j, the small ones of these; the s-lines (i, k) in bit k of row i alike.
template <int n>
__device__ __noinline__ bool find_alone(const ll* U, int range, bool act, unsigned (&rows)[4][n], int* alone, int x, int y) {
  using L = LineLayout<n>;
  if (act) {
    *alone = 0;
    if (y == 0)
      for (int q = 0; q < 4; ++q) rows[q][x] = 0;
  }
  __syncthreads();
  int t = kGoodLine;
  if (act) {
    ll m[3] = {0, 0, 0};
#pragma unroll 1
    for (int l = 0; l < n; ++l) {
      const ll a[3] = {U[L::idx(l, x, y)], U[L::idx(x, l, y)], U[L::idx(x, y, l)]};
      for (int d = 0; d < 3; ++d) m[d] |= a[d] ^ (a[d] >> 63);
    }
    int st[3];
    for (int d = 0; d < 3; ++d) st[d] = line_state(kBits - 64 + __clzll(m[d]), range);
    for (int d = 0; d < 2; ++d) {
      if (st[d] != kGoodLine) atomicOr(&rows[2 * d][x], 1u << y);
      if (st[d] == kSmallLine) atomicOr(&rows[2 * d + 1][x], 1u << y);
    }
    t = st[2];
  }
  __syncthreads();
  const bool a = t != kGoodLine && (rows[0][y] & rows[2][x] & (t == kSmallLine ? ~0u : rows[1][y] | rows[3][x])) != 0;
  if (a) *alone = 1;
  return a;
}

// The elements that the integer path does not cover, in FP64 (Alg. 1), by all threads of the CTA: those with `on`
// evaluate the t-line (x, y) of element e from v into P.w and return its part of <v, A_L v>.  U: the element's shared
// memory (three arrays).  FP64 multiply-adds bound it (1.7 per clock and SM), so the loops are left rolled.
template <int N>
__device__ __noinline__ double element_fp64(const AxParams<double>& P, const double* v, int64_t e, int x, int y, bool on,
                                            double* U) {
  constexpr int n = N + 1, n2 = n * n, n3 = n2 * n;
  using L = LineLayout<n>;
  double *R = U + L::size, *S = R + L::size;
  const int line = x + n * y;
  const int64_t base = e * n3 + line;
  double pw = 0.0;
  __syncthreads();
  if (on)
#pragma unroll 1
    for (int k = 0; k < n; ++k) U[L::idx(x, y, k)] = v[base + k * n2];
  __syncthreads();
  if (on) {
    const int s = P.fx.sG[e].x;
#pragma unroll 1
    for (int k = 0; k < n; ++k) {
      double ur = 0.0, us = 0.0, ut = 0.0;
#pragma unroll 1
      for (int l = 0; l < n; ++l) {
        ur += P.D[x * n + l] * U[L::idx(l, y, k)];
        us += P.D[y * n + l] * U[L::idx(x, l, k)];
        ut += P.D[k * n + l] * U[L::idx(x, y, l)];
      }
      const double w3 = P.fx.wq[x] * P.fx.wq[y] * P.fx.wq[k];
      double g[6];
#pragma unroll
      for (int f = 0; f < 3; ++f) {
        const int4 c = P.fx.G[(e * 3 + f) * n3 + line + k * n2];
        g[2 * f] = ldexp(__ll2double_rn(shl(c.y, 32) + c.x), -s) * w3;
        g[2 * f + 1] = ldexp(__ll2double_rn(shl(c.w, 32) + c.z), -s) * w3;
      }
      R[L::idx(x, y, k)] = g[0] * ur + g[3] * us + g[4] * ut;
      S[L::idx(x, y, k)] = g[3] * ur + g[1] * us + g[5] * ut;
      P.w[base + k * n2] = g[4] * ur + g[5] * us + g[2] * ut;  // until u has been read
    }
  }
  __syncthreads();
  if (on)
#pragma unroll 1
    for (int k = 0; k < n; ++k) U[L::idx(x, y, k)] = P.w[base + k * n2];
  __syncthreads();
  if (on)
#pragma unroll 1
    for (int k = 0; k < n; ++k) {
      double w = 0.0;
#pragma unroll 1
      for (int l = 0; l < n; ++l)
        w += P.D[l * n + x] * R[L::idx(l, y, k)] + P.D[l * n + y] * S[L::idx(x, l, k)] + P.D[l * n + k] * U[L::idx(x, y, l)];
      w *= P.h1;
      if (P.helm) w += P.h2 * P.B[base + k * n2] * v[base + k * n2];
      P.w[base + k * n2] = w;
      pw += v[base + k * n2] * w;
    }
  return pw;
}

// Arrays of an element in shared memory: u, then the r- and s-lines' values, and for n >= 10 the t-line's while the
// thread works on the other two (24 registers at n = 12).
__host__ __device__ constexpr int line_arrays(int N) { return N >= 9 ? 4 : 3; }
__host__ __device__ constexpr int line_threads(int N, int epb) { return (epb * (N + 1) * (N + 1) + 31) / 32 * 32; }
// Resident threads per SM, by the registers a line of n values needs: 768 up to n = 9 (N = 7, E = 32,768: 287 us; 640:
// 304; 480: 362), 640 for n = 10 and 11 (N = 10: 372; 768: 521), 480 for n = 12 (478; 640: 604).
__host__ __device__ constexpr int line_blocks(int N, int epb) {
  const int r = (N <= 8 ? 768 : N <= 10 ? 640 : 480) / line_threads(N, epb);
  return r < 1 ? 1 : r;
}

template <int N, int EPB, bool FUSED>
__global__ void __launch_bounds__(line_threads(N, EPB), line_blocks(N, EPB))
    k_ax_fx(const __grid_constant__ LineParams<N> Q) {
  constexpr int n = N + 1, n2 = n * n, n3 = n2 * n;
  const AxParams<double>& P = Q.a;
  using L = LineLayout<n>;
  extern __shared__ __align__(16) unsigned char smem_raw[];
  __shared__ double sred[32];
  __shared__ int sdone;
  using Max = ElemMax<n2, EPB>;
  __shared__ int smax[3][Max::size];
  __shared__ unsigned srow[EPB][4][n];  // find_alone
  __shared__ int alone[EPB];            // a point without a good line
  __shared__ int slook, sfp64;          // in the CTA: a t-line that may not be good; elements in FP64

  const int tid = threadIdx.x;
  if (FUSED) {
    if (tid == 0) sdone = P.st->done;
    __syncthreads();
    if (sdone) return;
  }
  // the CTA's factors into L2 while u is loaded and contracted (a hint, nothing waits on it)
  if (tid == 0) {
    const int64_t e0 = (int64_t)blockIdx.x * EPB;
    const uint32_t bytes = (uint32_t)(min((int64_t)EPB, P.E - e0) * 6 * n3 * sizeof(int2));
    asm volatile("cp.async.bulk.prefetch.L2.global [%0], %1;" ::"l"(P.fx.G + e0 * 3 * n3), "r"(bytes) : "memory");
    if (P.helm && n % 2 == 0)  // (16-byte ranges)
      asm volatile("cp.async.bulk.prefetch.L2.global [%0], %1;" ::"l"(P.fx.B + e0 * n3), "r"(bytes / 6) : "memory");
  }
  for (int q = 0; q < 3; ++q) Max::clear(smax[q]);
  if (tid == 0) {
    slook = 0;
    sfp64 = P.fx.direct;
  }
  if (!Max::whole) __syncthreads();

  const int le = min(tid / n2, EPB - 1), line = tid - le * n2, x = line % n, y = line / n;
  const int64_t e = (int64_t)blockIdx.x * EPB + le;
  const bool act = line < n2 && e < P.E;
  ll* U = reinterpret_cast<ll*>(smem_raw) + (size_t)le * line_arrays(N) * L::size;
  ll* R = U + L::size;
  ll* S = R + L::size;
  ll* T = S + L::size;
  constexpr bool park = line_arrays(N) == 4;
  const int64_t base = e * n3 + line;  // the t-line's points: i = x, j = y

  ll wt[n];  // the t-line: D_t u, then (G grad u)_t, then the result
  int ehi = 0;
  {
    double v[n];
#pragma unroll
    for (int k = 0; k < n; ++k) v[k] = 0.0;
    if (act) {
      if (FUSED) {
        const double beta = P.st->beta;
        double* po = P.pout ? P.pout : P.p;
#pragma unroll
        for (int k = 0; k < n; ++k) v[k] = P.z[base + k * n2] + beta * P.p[base + k * n2];
#pragma unroll
        for (int k = 0; k < n; ++k) po[base + k * n2] = v[k];
      } else {
#pragma unroll
        for (int k = 0; k < n; ++k) v[k] = P.u[base + k * n2];
      }
    }
#pragma unroll
    for (int k = 0; k < n; ++k) ehi = max(ehi, __double2hiint(v[k]) & 0x7fffffff);
    Max::put(smax[0], le, ehi);
    __syncthreads();
    const int lhi = ehi;
    ehi = Max::get(smax[0], le);
    if (ehi == 0) ehi = 1023 << 20;  // an element of zeros
    if (act) {
      if (expo(ehi) - expo(lhi) + P.fx.range > kLineBits) slook = 1;
      if (expo(ehi) < kExpMin || expo(ehi) > kExpMax) sfp64 = 1;
    }
    if (act) {
      ll u[n];
#pragma unroll
      for (int k = 0; k < n; ++k) {
        u[k] = from_double(v[k], expo(ehi));
        U[L::idx(x, y, k)] = u[k];
      }
      contract<n>(Q.d.e, Q.d.o, u, wt);
    }
  }
  int m = 0;
#pragma unroll
  for (int k = 0; k < n; ++k) {
    if (act) m |= mag(wt[k]);
    if (park && act) T[L::idx(x, y, k)] = wt[k];
  }
  const int sG = act ? P.fx.sG[e].x : 0;
  __syncthreads();
  if (slook) {  // the same for the whole CTA
    if (find_alone<n>(U, act ? P.fx.sG[e].y : 0, act, srow[le], alone + le, x, y)) sfp64 = 1;
  }

  if (act) {
    ll v[n], g[n];
#pragma unroll
    for (int l = 0; l < n; ++l) v[l] = U[L::idx(l, x, y)];
    contract<n>(Q.d.e, Q.d.o, v, g);
#pragma unroll
    for (int l = 0; l < n; ++l) {
      R[L::idx(l, x, y)] = g[l];
      m |= mag(g[l]);
    }
#pragma unroll
    for (int l = 0; l < n; ++l) v[l] = U[L::idx(x, l, y)];
    contract<n>(Q.d.e, Q.d.o, v, g);
#pragma unroll
    for (int l = 0; l < n; ++l) {
      S[L::idx(x, l, y)] = g[l];
      m |= mag(g[l]);
    }
  }
  Max::put(smax[1], le, bits_of(m));
  // the first point's factors, [f/2][k][line] of two each
  const int4* Ge = P.fx.G + e * 3 * n3 + line;
  int4 n0, n1, n2_;
  n0 = n1 = n2_ = make_int4(0, 0, 0, 0);
  if (act) {
    n0 = __ldg(Ge);
    n1 = __ldg(Ge + n3);
    n2_ = __ldg(Ge + 2 * n3);
  }
  __syncthreads();

  // gradients to 60 bits; (wr, ws, wt) = G (ur, us, ut), g1..g6 = G_rr, G_ss, G_tt, G_rs, G_rt, G_st
  const int s1 = max(kBits - Max::get(smax[1], le), 0);
  m = 0;
  if (act) {
#pragma unroll
    for (int k = 0; k < n; ++k) {
      const int4 x0 = n0, x1 = n1, x2 = n2_;
      if (k + 1 < n) {
        n0 = __ldg(Ge + (k + 1) * n2);
        n1 = __ldg(Ge + n3 + (k + 1) * n2);
        n2_ = __ldg(Ge + 2 * n3 + (k + 1) * n2);
      }
      const int2 g1 = make_int2(x0.x, x0.y), g2 = make_int2(x0.z, x0.w), g3 = make_int2(x1.x, x1.y);
      const int2 g4 = make_int2(x1.z, x1.w), g5 = make_int2(x2.x, x2.y), g6 = make_int2(x2.z, x2.w);
      const int at = L::idx(x, y, k);
      const int2 v[3] = {split(shl(R[at], s1)), split(shl(S[at], s1)), split(shl(park ? T[at] : wt[k], s1))};
      const int2 r0[3] = {g1, g4, g5}, r1[3] = {g4, g2, g6}, r2[3] = {g5, g6, g3};
      const ll wr = dot<3, n % 2 == 0>(r0, v), ws = dot<3, n % 2 == 0>(r1, v);
      const ll w = dot<3, n % 2 == 0>(r2, v);
      R[at] = wr;
      S[at] = ws;
      if (park)
        T[at] = w;
      else
        wt[k] = w;
      m |= mag(wr) | mag(ws) | mag(w);
    }
  }
  Max::put(smax[2], le, bits_of(m));
  __syncthreads();

  const int up = kBits - Max::get(smax[2], le);
  if (act) {
    ll v[n], g[n];
#pragma unroll
    for (int l = 0; l < n; ++l) v[l] = shl(R[L::idx(l, x, y)], up);
    contract<n>(Q.d.te, Q.d.to, v, g);
#pragma unroll
    for (int l = 0; l < n; ++l) R[L::idx(l, x, y)] = g[l];
#pragma unroll
    for (int l = 0; l < n; ++l) v[l] = shl(S[L::idx(x, l, y)], up);
    contract<n>(Q.d.te, Q.d.to, v, g);
#pragma unroll
    for (int l = 0; l < n; ++l) S[L::idx(x, l, y)] = g[l];
#pragma unroll
    for (int k = 0; k < n; ++k) v[k] = shl(park ? T[L::idx(x, y, k)] : wt[k], up);
    contract<n>(Q.d.te, Q.d.to, v, wt);
  }
  int2 B[n];  // loaded together, ahead of the stores of w
#pragma unroll
  for (int k = 0; k < n; ++k) B[k] = P.helm && act ? __ldg(P.fx.B + base + k * n2) : make_int2(0, 0);
  __syncthreads();

  double pw = 0.0;  // this thread's part of <p, A_L p>
  const bool fp64 = sfp64 && (P.fx.direct || (slook && alone[le]) || expo(ehi) < kExpMin || expo(ehi) > kExpMax);
  if (act && !fp64) {
    const int eu = expo(ehi) - 1022 - kBits;    // u = value 2^eu
    int eo = eu + Q.scale - sG - s1 - up;       // the unit of a point's sum, without its weights
    MassTerm mt{Q.h2, 0};
    bool helm = P.helm, mass64 = false;
    if (helm) {
      const int sB = P.fx.sB[e], em = eu + 63 + Q.e2 - sB;
      mass64 = sG - sB > Q.mass_limit;
      helm = !mass64;
      mt.down = eo - em;
      if (helm) eo = max(eo, em);
    }
    const double* v = FUSED ? (P.pout ? P.pout : P.p) : P.u;
#pragma unroll
    for (int k = 0; k < n; ++k) {
      const int at = L::idx(x, y, k);
      ll o = wt[k] + R[at] + S[at];
      if (helm) o = mt.add(o, B[k], split(U[at]));
      // The weights and <p, A p> in FP64, whose pipe is idle.  (In integers, a CG iteration at N = 7, E = 32,768: 661 to 669 us,
      // 655 so; with p from its integers 661; a plain apply at E = 262,144 with the weights in integers 2697, 2667 so.)
      const double w = to_double(o, eo) * __ldg(P.fx.W64 + line + k * n2);
      if (FUSED) pw = fma(v[base + k * n2], w, pw);
      P.w[base + k * n2] = w;
    }
    if (mass64) {
#pragma unroll 1
      for (int k = 0; k < n; ++k) {
        const double u = v[base + k * n2], t = P.h2 * P.B[base + k * n2] * u;
        P.w[base + k * n2] += t;
        if (FUSED) pw += u * t;
      }
    }
  }
  if (sfp64) {  // the same for the whole CTA
    const double r = element_fp64<N>(P, FUSED ? (P.pout ? P.pout : P.p) : P.u, e, x, y, act && fp64,
                                     reinterpret_cast<double*>(U));
    if (act && fp64) pw = r;
  }

  if (FUSED) {  // this block's part of <p, A_L p>; k_pap_finish sums the parts in block order
    const double s = block_sum(pw, sred);
    if (tid == 0) P.partial[blockIdx.x] = s;
  }
}

template <int N>
LineTable<N> line_table() {
  constexpr int n = N + 1;
  const FxScale& f = fx_scale(N);
  LineTable<N> t{};
  auto fill = [&](auto at, long double s, auto& e, auto& o) {
    for (int r = 0; r < (n + 1) / 2; ++r) {
      for (int l = 0; l < n / 2; ++l) {
        e[r][l] = split(std::llround((at(r, l) + at(r, n - 1 - l)) / 2 * s));
        o[r][l] = split(std::llround((at(r, l) - at(r, n - 1 - l)) / 2 * s));
      }
      if (n & 1) e[r][n / 2] = split(std::llround(at(r, n / 2) * s));
    }
  };
  fill([&](int r, int l) { return f.D[r * n + l]; }, f.d, t.e, t.o);
  fill([&](int r, int l) { return f.M[r * n + l]; }, f.dt, t.te, t.to);
  return t;
}

// The forward table times mant 2^-shift (h1 without its exponent, or half of that), to half a unit.
template <class T>
void scale_table(const T& from, T& to, long long mant, int shift) {  // mant 2^-53 in (-1, 1)
  for (size_t r = 0; r < std::size(from); ++r)
    for (size_t l = 0; l < std::size(from[r]); ++l) {
      const int2 c = from[r][l];
      const __int128 p = (__int128)(((long long)c.y << 32) + c.x) * mant + ((__int128)1 << (shift - 1));
      to[r][l] = split((long long)(p >> shift));
    }
}

// Whether fx::dot's middle sums of the table's rows stay below 2^63 for all folded values (up to 2^61, so |y| <= 2^29 and
// |x| <= 2^31).
template <class T>
bool sums_fit(const T& t) {
  for (auto& row : t) {
    unsigned long long s = 1ull << 31;
    for (const int2& c : row)
      s += ((unsigned long long)std::llabs(c.x) << 29) + ((unsigned long long)std::llabs(c.y) << 31);
    if (s >> 63) return false;
  }
  return true;
}

template <int N, int EPB, bool FUSED>
cudaError_t launch_fx_t(const AxParams<double>& user, cudaStream_t s, int* grid_out) {
  constexpr int n = N + 1;
  const size_t smem = sizeof(ll) * (size_t)line_arrays(N) * EPB * LineLayout<n>::size;
  static DeviceOnce once;
  cudaError_t aerr = once.get([&](int, int*) {
    return cudaFuncSetAttribute(k_ax_fx<N, EPB, FUSED>, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem);
  });
  if (aerr != cudaSuccess) return aerr;
  // h1 or h2 outside 2^+-100: the operator with both over 2^far, and the results times 2^far by a pass of their own
  AxParams<double> p = user;
  int far = 0;
  const double top = std::max(std::fabs(p.h1), std::fabs(p.h2));
  if (!p.fx.direct && top != 0.0 && !(top >= 0x1p-100 && top <= 0x1p100)) {
    far = std::ilogb(top);
    p.h1 = std::ldexp(p.h1, -far);
    p.h2 = std::ldexp(p.h2, -far);
    p.helm = p.h2 != 0.0;
  }
  const int64_t grid = (p.E + EPB - 1) / EPB;
  if (grid_out) *grid_out = (int)grid;
  if (p.E == 0) return cudaSuccess;
  static const LineTable<N> plain = line_table<N>();
  LineParams<N> q{p, fx_scale(N).scale, make_int2(0, 0), 0, 0, plain};
  int e1 = 0;  // exponent of h1
  if (p.helm && !p.fx.direct)
    q.h2 = split(std::llround(std::ldexp(std::frexp((long double)p.h2 / fx_scale(N).kappa, &q.e2), 62)));
  if (p.h1 != 1.0 && !p.fx.direct) {
    const long long mant = (long long)std::ldexp(std::frexp(p.h1, &e1), 53);
    // The plain tables keep the sums below 0.8 2^63; a mantissa gives the entries any low halves, and then the sums of
    // N >= 9 can pass 2^63 (at worst 1.15 2^63 at N = 11, where about 4 mantissas in 10,000 allow it).  Half the mantissa
    // keeps them below 0.96 2^63, at the cost of one bit.
    for (int shift = 53; shift <= 54; ++shift) {
      scale_table(plain.e, q.d.e, mant, shift);
      scale_table(plain.o, q.d.o, mant, shift);
      q.scale = fx_scale(N).scale + e1 + shift - 53;
      if (sums_fit(q.d.e) && sums_fit(q.d.o)) break;
    }
  }
  // The mass term of a point where u is small is rounded like the element's largest; FP64 rounds it with the stiffness
  // terms of the point's lines.  It is left in fixed point up to 2^4 times the bound of those, 2 D_00^2 h1 G: beyond that
  // (h1 = 0 among them) the mass is most of the result.
  if (p.helm) {
    constexpr int d00 = N * n / 4 < 2 ? 0 : N * n / 4 < 4 ? 2 : N * n / 4 < 8 ? 4 : N * n / 4 < 16 ? 6 : N * n / 4 < 32 ? 8 : 10;
    q.mass_limit = p.h1 == 0.0 ? -100000 : e1 + d00 + 1 + 4 - q.e2;
  }
  k_ax_fx<N, EPB, FUSED><<<(unsigned)grid, line_threads(N, EPB), smem, s>>>(q);
  cudaError_t err = cudaGetLastError();
  if (far && err == cudaSuccess)
    err = launch_scale_far(p.w, p.E * n * n * n, FUSED ? p.partial : nullptr, (int)grid, far, FUSED ? p.st : nullptr, s);
  if (FUSED && err == cudaSuccess) err = launch_pap_finish(p.partial, (int)grid, p.st, s);
  return err;
}

}  // namespace fxk

// Native FP64 operator of order N: variants 0 and 1 are the register kernels on
// the FP64 pipe (ax_impl.cuh), 4 and 5 the fixed-point kernel with ~128 / ~256
// threads per CTA.
template <int N>
inline cudaError_t dispatch_fp64_n(int variant, bool fused, const AxParams<double>& p, cudaStream_t s, int* grid_out) {
  if (variant < 2) return p.G ? dispatch_ax_n<double, N>(variant, fused, p, s, grid_out) : cudaErrorNotSupported;
  if (!p.fx.G || variant < kAxFixed || variant >= kAxVariants) return cudaErrorNotSupported;
  constexpr int e2 = epb_for(N, 1), e3 = epb_for(N, 0);
  if (variant == kAxFixed)
    return fused ? fxk::launch_fx_t<N, e2, true>(p, s, grid_out) : fxk::launch_fx_t<N, e2, false>(p, s, grid_out);
  return fused ? fxk::launch_fx_t<N, e3, true>(p, s, grid_out) : fxk::launch_fx_t<N, e3, false>(p, s, grid_out);
}

}  // namespace sem
