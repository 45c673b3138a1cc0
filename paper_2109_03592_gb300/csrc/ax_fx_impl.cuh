// FP64 local operator (Alg. 1 + h2 mass term) in 64-bit fixed point on the
// integer pipe (fixed.cuh), even-odd form, for even n = N + 1.
//
// The contractions are those of ax_eo_impl.cuh: D and D^T are
// centro-antisymmetric, so with P = v[l] + v[l'], M = v[l] - v[l'] (l' = n-1-l)
//   (D v)[i], (D v)[i'] = sum_l Em[i][l] M[l] +- sum_l Ep[i][l] P[l],
// and one thread owns one 2x2x2 octant {a, n-1-a} x {b, n-1-b} x {c, n-1-c}
// ((n/2)^3 threads per element).  Three IMAD.WIDE per multiply-add and plain
// 64-bit adds replace the ~12 and ~8 FP32 instructions of the double-float form.
//
// Scaling, all powers of two: u is brought to 60 bits below the element's
// largest exponent; each thread shifts its gradients up to 60 bits (results of
// smooth fields are small against the terms of D that cancel), and after the
// factors the element's values go to 60 bits below their largest. The stored
// factors are G 2^(t + sG) with t = ti[i] + ti[j] + ti[k], 2^-ti ~ w_i / max w:
// the quadrature weights, which spread G over 2^11 within an element at N = 7,
// become part of the second shift (t is the same for a thread's eight points,
// the weights being symmetric).  Measured against 128-bit arithmetic the error is
// that of the FP64-pipe kernel to within a third at every order (N = 1..11,
// random and smooth fields; 1e-15 and 5e-14 at N = 7, most of it the table of D),
// where the double-float kernels have 1e-14 and 1e-12.
//
// An element whose values are not finite, or whose exponents lie outside the
// range that the shifts are written for (2^-500 .. 2^500), is evaluated in FP64
// directly from memory (slow_point).
//
// What bounds it: issue slots.  IMAD.WIDE, shifts and logic cost two slots each
// and do not overlap (measured), so the 3150 instructions a warp spends on 256
// points are ~4600 slots; they run at two thirds of that rate.  E = 32,768, N =
// 7: 349 us (3.9 TB/s of u, G and w), against 407 us for the even-odd double-float
// kernel and 1900 us on the FP64 pipe; N = 11 (E = 10,240): 494, 588 and 3200 us.
#pragma once

#include "ax_eo_impl.cuh"
#include "ax_fxd_impl.cuh"
#include "ax_impl.cuh"
#include "fixed.cuh"
#include "fx_common.cuh"

namespace sem {
namespace fxk {

using eo_detail::EoLayout;

// Register budget: 512 resident threads per SM (128 registers, no spills to speak of) measured fastest at N = 3 to 9
// (N = 7: 349 us at E = 32,768; 376 us at 640 threads, which spill, 375 us at 384).
constexpr int fx_min_blocks(int threads) { return 512 / threads < 1 ? 1 : 512 / threads; }

constexpr int octants(int N) { return ((N + 1) / 2) * ((N + 1) / 2) * ((N + 1) / 2); }

template <int N, int EPB, bool FUSED>
__global__ void __launch_bounds__(EPB* octants(N), fx_min_blocks(EPB* octants(N)))
    k_ax_fx(const AxParams<double> P) {
  constexpr int n = N + 1, h = n / 2, T = h * h * h, n2 = n * n, n3 = n2 * n;
  using L = EoLayout<n>;
  extern __shared__ __align__(16) unsigned char smem_raw[];
  int4* sC = reinterpret_cast<int4*>(smem_raw);  // [2][h][h]: (Ep, Em), D then D^T
  int2* sA = reinterpret_cast<int2*>(sC + 2 * h * h);
  __shared__ double sred[32];
  __shared__ int sdone;
  using Max = ElemMax<T, EPB>;
  __shared__ int smax[2][Max::size];

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
  }
  Max::clear(smax[0]);
  Max::clear(smax[1]);
  // coefficients; |h1| 2^-e1 in [1/2, 1) scales the forward ones, e1 goes into the exponent
  int e1 = 0;
  if (P.h1 == 1.0) {
    for (int q = tid; q < 2 * h * h; q += blockDim.x) sC[q] = P.fx.tab[q];
  } else {
    const double hm = P.h1 == 0.0 ? 0.0 : frexp(P.h1, &e1);
    for (int q = tid; q < 2 * h * h; q += blockDim.x) {
      const int4 c = P.fx.tab[q];
      if (q < h * h) {
        const double s = 4294967296.0;
        const int2 p = split(__double2ll_rn(hm * ((double)c.y * s + (double)c.x)));
        const int2 m = split(__double2ll_rn(hm * ((double)c.w * s + (double)c.z)));
        sC[q] = make_int4(p.x, p.y, m.x, m.y);
      } else {
        sC[q] = c;
      }
    }
  }

  const int le = tid / T, t = tid - le * T;
  const int a = t % h, b = (t / h) % h, c = t / (h * h);
  const int64_t e = (int64_t)blockIdx.x * EPB + le;
  const bool act = e < P.E;
  int2* S0 = sA + (size_t)le * 3 * L::size;
  int2* S1 = S0 + L::size;
  int2* S2 = S1 + L::size;
  const int I[2] = {a, n - 1 - a}, J[2] = {b, n - 1 - b}, K[2] = {c, n - 1 - c};
  // octant point q = da + 2 db + 4 dc is (I[da], J[db], K[dc])
  const int64_t base = e * n3;

  // u again where the mass term and <p, A_L p> need it (sixteen registers fewer in between)
  const double* uv = FUSED ? (P.pout ? P.pout : P.p) : P.u;
  auto u_at = [&](int q, int emax) {
    return split(from_double(uv[base + I[q & 1] + n * J[(q >> 1) & 1] + n2 * K[q >> 2]], emax));
  };
  ll u[8];
  int ehi = 0;
  {
    double v[8];
#pragma unroll
    for (int q = 0; q < 8; ++q) v[q] = 0.0;
    if (act) {
      if (FUSED) {
        const double beta = P.st->beta;
        double* po = P.pout ? P.pout : P.p;
#pragma unroll
        for (int q = 0; q < 8; ++q) {
          const int64_t g = base + I[q & 1] + n * J[(q >> 1) & 1] + n2 * K[q >> 2];
          v[q] = P.z[g] + beta * P.p[g];
        }
#pragma unroll
        for (int q = 0; q < 8; ++q) po[base + I[q & 1] + n * J[(q >> 1) & 1] + n2 * K[q >> 2]] = v[q];
      } else {
#pragma unroll
        for (int q = 0; q < 8; ++q) v[q] = P.u[base + I[q & 1] + n * J[(q >> 1) & 1] + n2 * K[q >> 2]];
      }
    }
#pragma unroll
    for (int q = 0; q < 8; ++q) ehi = max(ehi, __double2hiint(v[q]) & 0x7fffffff);
    if (!Max::whole) __syncthreads();  // smax is cleared
    Max::put(smax[0], le, ehi);
    __syncthreads();
    ehi = Max::get(smax[0], le);
    if (ehi == 0) ehi = 1023 << 20;  // an element of zeros
#pragma unroll
    for (int q = 0; q < 8; ++q) u[q] = from_double(v[q], expo(ehi));
  }
  const int sG = act ? P.fx.sG[e] : 0;
  const bool slow = P.fx.direct || expo(ehi) < kExpMin || expo(ehi) > kExpMax;
  const int tq = P.fx.ti[a] + P.fx.ti[b] + P.fx.ti[c];
  int ex = expo(ehi) - 1022 - kBits + e1;  // u = value 2^ex (e1 from here on)

  // pre-additions of the three directions; P at the pair's low index, M at its high one
#pragma unroll
  for (int x = 0; x < 2; ++x)
#pragma unroll
    for (int y = 0; y < 2; ++y) {
      {  // r: pairs over da, row (db, dc) = (x, y)
        const ll p = u[2 * x + 4 * y], m = u[1 + 2 * x + 4 * y];
        S0[L::idx(a, J[x], K[y])] = split(p + m);
        S0[L::idx(n - 1 - a, J[x], K[y])] = split(p - m);
      }
      {  // s: pairs over db, row (da, dc) = (x, y)
        const ll p = u[x + 4 * y], m = u[x + 2 + 4 * y];
        S1[L::idx(I[x], b, K[y])] = split(p + m);
        S1[L::idx(I[x], n - 1 - b, K[y])] = split(p - m);
      }
      {  // t: pairs over dc, row (da, db) = (x, y)
        const ll p = u[x + 2 * y], m = u[x + 2 * y + 4];
        S2[L::idx(I[x], J[y], c)] = split(p + m);
        S2[L::idx(I[x], J[y], n - 1 - c)] = split(p - m);
      }
    }
  __syncthreads();

  // one direction's contractions of this thread's four pairs: lo[q] / hi[q] = B +- A
  auto contract = [&](int d, const int4* C, int x, int y, ll& lo, ll& hi) {
    const int own = d == 0 ? a : d == 1 ? b : c;
    int2 pv[h], mv[h], ep[h], em[h];
#pragma unroll
    for (int l = 0; l < h; ++l) {
      const int4 cf = C[own * h + l];
      ep[l] = make_int2(cf.x, cf.y);
      em[l] = make_int2(cf.z, cf.w);
      if (d == 0) {
        pv[l] = S0[L::idx(l, J[x], K[y])];
        mv[l] = S0[L::idx(n - 1 - l, J[x], K[y])];
      } else if (d == 1) {
        pv[l] = S1[L::idx(I[x], l, K[y])];
        mv[l] = S1[L::idx(I[x], n - 1 - l, K[y])];
      } else {
        pv[l] = S2[L::idx(I[x], J[y], l)];
        mv[l] = S2[L::idx(I[x], J[y], n - 1 - l)];
      }
    }
    const ll A = dot<h>(ep, pv), B = dot<h>(em, mv);
    lo = B + A;
    hi = B - A;
  };

  // factors, [24][T] of two each, 3 of them per point: a point's are loaded one point ahead, the first here
  int4 n0, n1, n2_;
  n0 = n1 = n2_ = make_int4(0, 0, 0, 0);
  if (act) {
    const int4* Ge = P.fx.G + e * 3 * n3 + t;
    n0 = __ldg(Ge);
    n1 = __ldg(Ge + T);
    n2_ = __ldg(Ge + 2 * T);
  }

  // forward contractions: g[d][q] = (h1 D_d u)(point q), d = r, s, t
  ll g[3][8];
#pragma unroll
  for (int d = 0; d < 3; ++d)
#pragma unroll
    for (int x = 0; x < 2; ++x)
#pragma unroll
      for (int y = 0; y < 2; ++y) {
        const int q0 = d == 0 ? 2 * x + 4 * y : d == 1 ? x + 4 * y : x + 2 * y;
        contract(d, sC, x, y, g[d][q0], g[d][q0 + (d == 0 ? 1 : d == 1 ? 2 : 4)]);
      }
  ex += 64 - P.fx.sc[0];

  // each thread's gradients up to 60 bits: one shift for its eight points
  int m = 0;
#pragma unroll
  for (int d = 0; d < 3; ++d)
#pragma unroll
    for (int q = 0; q < 8; ++q) m |= mag(g[d][q]);
  const int s1 = max(kBits - bits_of(m), 0);
#pragma unroll
  for (int d = 0; d < 3; ++d)
#pragma unroll
    for (int q = 0; q < 8; ++q) g[d][q] = shl(g[d][q], s1);

  // (wr, ws, wt) = G (ur, us, ut); g1..g6 = G_rr, G_ss, G_tt, G_rs, G_rt, G_st
  m = 0;
  if (act) {
    const int4* Ge = P.fx.G + e * 3 * n3 + t;
#pragma unroll
    for (int q = 0; q < 8; ++q) {
      const int4 x0 = n0, x1 = n1, x2 = n2_;
      if (q < 7) {
        n0 = __ldg(Ge + (3 * q + 3) * T);
        n1 = __ldg(Ge + (3 * q + 4) * T);
        n2_ = __ldg(Ge + (3 * q + 5) * T);
      }
      const int2 g1 = make_int2(x0.x, x0.y), g2 = make_int2(x0.z, x0.w), g3 = make_int2(x1.x, x1.y);
      const int2 g4 = make_int2(x1.z, x1.w), g5 = make_int2(x2.x, x2.y), g6 = make_int2(x2.z, x2.w);
      const int2 v[3] = {split(g[0][q]), split(g[1][q]), split(g[2][q])};
      const int2 r0[3] = {g1, g4, g5}, r1[3] = {g4, g2, g6}, r2[3] = {g5, g6, g3};
      g[0][q] = dot<3>(r0, v);
      g[1][q] = dot<3>(r1, v);
      g[2][q] = dot<3>(r2, v);
      m |= mag(g[0][q]) | mag(g[1][q]) | mag(g[2][q]);
    }
  }
  // this thread's w are value 2^(64 - sG - s1 - tq): onto the element's common exponent, at 60 bits
  constexpr int kOff = 256;  // keeps the maximum positive
  Max::put(smax[1], le, bits_of(m) - s1 - tq + kOff);
  __syncthreads();  // and every forward read of S0..S2 is done
  {
    const int up = kBits + kOff - Max::get(smax[1], le);
    const int s = up - s1 - tq;
    if (s >= 0) {
#pragma unroll
      for (int d = 0; d < 3; ++d)
#pragma unroll
        for (int q = 0; q < 8; ++q) g[d][q] = shl(g[d][q], s);
    } else {
      const int r = min(-s, 63);
#pragma unroll
      for (int d = 0; d < 3; ++d)
#pragma unroll
        for (int q = 0; q < 8; ++q) g[d][q] >>= r;
    }
    ex += 64 - sG - up;
  }

#pragma unroll
  for (int x = 0; x < 2; ++x)
#pragma unroll
    for (int y = 0; y < 2; ++y) {
      {
        const ll p = g[0][2 * x + 4 * y], q = g[0][1 + 2 * x + 4 * y];
        S0[L::idx(a, J[x], K[y])] = split(p + q);
        S0[L::idx(n - 1 - a, J[x], K[y])] = split(p - q);
      }
      {
        const ll p = g[1][x + 4 * y], q = g[1][x + 2 + 4 * y];
        S1[L::idx(I[x], b, K[y])] = split(p + q);
        S1[L::idx(I[x], n - 1 - b, K[y])] = split(p - q);
      }
      {
        const ll p = g[2][x + 2 * y], q = g[2][x + 2 * y + 4];
        S2[L::idx(I[x], J[y], c)] = split(p + q);
        S2[L::idx(I[x], J[y], n - 1 - c)] = split(p - q);
      }
    }
  __syncthreads();

  // back contractions with D^T: w(point) = sum over d of (D_d^T w_d)(point)
  ll o[8];
#pragma unroll
  for (int d = 0; d < 3; ++d)
#pragma unroll
    for (int x = 0; x < 2; ++x)
#pragma unroll
      for (int y = 0; y < 2; ++y) {
        const int q0 = d == 0 ? 2 * x + 4 * y : d == 1 ? x + 4 * y : x + 2 * y;
        const int q1 = q0 + (d == 0 ? 1 : d == 1 ? 2 : 4);
        ll lo, hi;
        contract(d, sC + h * h, x, y, lo, hi);
        o[q0] = d == 0 ? lo : o[q0] + lo;
        o[q1] = d == 0 ? hi : o[q1] + hi;
      }
  ex += 64 - P.fx.sc[1];

  double pw = 0.0;  // this thread's part of <p, A_L p>
  if (act && !slow) {
    int eo = ex;
    if (P.helm) {
      MassTerm mt;
      mt.init(P.h2, P.fx.eB[e], expo(ehi));
#pragma unroll
      for (int q = 0; q < 8; ++q) {
        eo = ex;  // the same for the thread's eight points, as t is
        mt.add(o[q], eo, __ldg(P.B + base + I[q & 1] + n * J[(q >> 1) & 1] + n2 * K[q >> 2]), u_at(q, expo(ehi)), tq);
      }
      ex = eo;
    }
    ll ph = 0, pm = 0;
#pragma unroll
    for (int q = 0; q < 8; ++q) {
      P.w[base + I[q & 1] + n * J[(q >> 1) & 1] + n2 * K[q >> 2]] = to_double(o[q], ex);
      if (FUSED) {
        const int2 x = u_at(q, expo(ehi)), y = split(o[q] >> 4);
        ph = mad(ph, x.y, y.y);
        pm = mad(mad(pm, x.x, y.y), x.y, y.x);
      }
    }
    if (FUSED) pw = ldexp(__ll2double_rn(ph + (pm >> 32)), 64 + 4 + ex + expo(ehi) - 1022 - kBits);
  } else if (act) {
#pragma unroll 1
    for (int q = 0; q < 8; ++q) {
      const int i = (q & 1) ? n - 1 - a : a, j = (q & 2) ? n - 1 - b : b, k = (q & 4) ? n - 1 - c : c;
      const double r = slow_point<N>(P, uv, e, i, j, k);
      P.w[base + i + n * j + n2 * k] = r;
      if (FUSED) pw += uv[base + i + n * j + n2 * k] * r;
    }
  }

  if (FUSED) {  // this block's part of <p, A_L p>; k_pap_finish sums the parts in block order
    const double s = block_sum(pw, sred);
    if (tid == 0) P.partial[blockIdx.x] = s;
  }
}

template <int N, int EPB, bool FUSED>
cudaError_t launch_fx_t(const AxParams<double>& p, cudaStream_t s, int* grid_out) {
  constexpr int n = N + 1, h = n / 2;
  const size_t smem = sizeof(int4) * 2 * h * h + sizeof(int2) * 3ull * EPB * EoLayout<n>::size;
  static DeviceOnce once;
  cudaError_t aerr = once.get([&](int, int*) {
    return cudaFuncSetAttribute(k_ax_fx<N, EPB, FUSED>, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem);
  });
  if (aerr != cudaSuccess) return aerr;
  const int64_t grid = (p.E + EPB - 1) / EPB;
  if (grid_out) *grid_out = (int)grid;
  if (p.E == 0) return cudaSuccess;
  k_ax_fx<N, EPB, FUSED><<<(unsigned)grid, EPB * octants(N), smem, s>>>(p);
  cudaError_t err = cudaGetLastError();
  if (FUSED && err == cudaSuccess) err = launch_pap_finish(p.partial, (int)grid, p.st, s);
  return err;
}

}  // namespace fxk

// Native FP64 operator of order N: variants 0 and 1 are the register kernels on
// the FP64 pipe (ax_impl.cuh), 4 and 5 the fixed-point kernels with ~128 / ~256
// threads per CTA.
template <int N>
inline cudaError_t dispatch_fp64_n(int variant, bool fused, const AxParams<double>& p, cudaStream_t s, int* grid_out) {
  if (variant < 2) return p.G ? dispatch_ax_n<double, N>(variant, fused, p, s, grid_out) : cudaErrorNotSupported;
  if (!p.fx.G || variant < kAxFixed || variant >= kAxVariants) return cudaErrorNotSupported;
  if constexpr ((N & 1) == 1) {
    constexpr int e2 = eo_detail::epb_eo(N, 2), e3 = eo_detail::epb_eo(N, 3);
    if (variant == kAxFixed)
      return fused ? fxk::launch_fx_t<N, e2, true>(p, s, grid_out) : fxk::launch_fx_t<N, e2, false>(p, s, grid_out);
    return fused ? fxk::launch_fx_t<N, e3, true>(p, s, grid_out) : fxk::launch_fx_t<N, e3, false>(p, s, grid_out);
  } else {
    constexpr int d2 = epb_for(N, 1), d3 = epb_for(N, 0);
    if (variant == kAxFixed)
      return fused ? fxk::launch_fxd_t<N, d2, true>(p, s, grid_out) : fxk::launch_fxd_t<N, d2, false>(p, s, grid_out);
    return fused ? fxk::launch_fxd_t<N, d3, true>(p, s, grid_out) : fxk::launch_fxd_t<N, d3, false>(p, s, grid_out);
  }
}

}  // namespace sem
