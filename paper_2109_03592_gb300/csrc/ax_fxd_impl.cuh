// FP64 local operator in 64-bit fixed point (fixed.cuh), direct form, for odd
// n = N + 1.  Scaling, accuracy and the FP64 evaluation of out-of-range
// elements as in ax_fx_impl.cuh; the thread mapping is that of the register
// kernels (ax_impl.cuh): a thread owns one (i, j) column, the t-direction
// stays in its registers, r and s go through shared memory.  Bound by issue slots
// like the even-odd form, with twice its multiply-adds: N = 8, E = 23,040: 674 us,
// against 793 us for the direct double-float kernel and 2220 us on the FP64 pipe;
// N = 10, E = 12,288: 752, 1001 and 2570 us.
#pragma once

#include "ax_impl.cuh"
#include "fixed.cuh"
#include "fx_common.cuh"

namespace sem {
namespace fxk {

template <int N, int EPB, bool FUSED>
__global__ void __launch_bounds__(EPB*(N + 1) * (N + 1)) k_ax_fxd(const AxParams<double> P) {
  constexpr int n = N + 1, n2 = n * n, n3 = n2 * n;
  constexpr int RP = n + 1, PL = n * RP;  // padded row / plane strides in shared memory
  extern __shared__ __align__(16) unsigned char smem_raw[];
  int2* sD = reinterpret_cast<int2*>(smem_raw);  // [2][n][RP]: D and D^T
  int2* sA = sD + 2 * n * RP;                    // [EPB][2][n PL]: u (first), then w_r and w_s
  __shared__ double sred[32];
  __shared__ int sdone;
  using Max = ElemMax<n2, EPB>;
  __shared__ int smax[3][Max::size];

  const int tid = threadIdx.x;
  if (FUSED) {
    if (tid == 0) sdone = P.st->done;
    __syncthreads();
    if (sdone) return;
  }
  for (int q = 0; q < 3; ++q) Max::clear(smax[q]);
  int e1 = 0;
  const double hm = P.h1 == 0.0 ? 0.0 : frexp(P.h1, &e1);
  if (P.h1 == 1.0) e1 = 0;
  {
    const int2* tab = reinterpret_cast<const int2*>(P.fx.tab);
    for (int q = tid; q < 2 * n2; q += blockDim.x) {
      int2 c = tab[q];
      if (q < n2 && P.h1 != 1.0) c = split(__double2ll_rn(hm * ((double)c.y * 4294967296.0 + (double)c.x)));
      sD[(q / n) * RP + q % n] = c;
    }
  }

  const int le = tid / n2, ij = tid - le * n2, i = ij % n, j = ij / n;
  const int64_t e = (int64_t)blockIdx.x * EPB + le;
  const bool act = e < P.E;
  int2* S0 = sA + (size_t)le * 2 * n * PL;
  int2* S1 = S0 + n * PL;
  const int64_t base = e * n3 + ij;

  int2 ru[n];  // u of the column, in fixed point
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
    if (!Max::whole) __syncthreads();  // smax is cleared
    Max::put(smax[0], le, ehi);
    __syncthreads();
    ehi = Max::get(smax[0], le);
    if (ehi == 0) ehi = 1023 << 20;  // an element of zeros
#pragma unroll
    for (int k = 0; k < n; ++k) {
      ru[k] = split(from_double(v[k], expo(ehi)));
      S0[k * PL + j * RP + i] = ru[k];
    }
  }
  const int sG = act ? P.fx.sG[e] : 0;
  const bool slow = P.fx.direct || expo(ehi) < kExpMin || expo(ehi) > kExpMax;
  const int tij = P.fx.ti[i] + P.fx.ti[j];
  int ex = expo(ehi) - 1022 - kBits + e1;  // u = value 2^ex (e1 from here on)
  __syncthreads();

  // forward contractions: g[d][k] = (h1 D_d u)(i, j, k)
  ll g[3][n];
#pragma unroll
  for (int k = 0; k < n; ++k) {
    Dot r, s, t;
#pragma unroll
    for (int l = 0; l < n; ++l) {
      r.add(sD[i * RP + l], S0[k * PL + j * RP + l]);
      s.add(sD[j * RP + l], S0[k * PL + l * RP + i]);
      t.add(sD[k * RP + l], ru[l]);
    }
    g[0][k] = r.get();
    g[1][k] = s.get();
    g[2][k] = t.get();
  }
  ex += 64 - P.fx.sc[0];
  int m = 0;
#pragma unroll
  for (int k = 0; k < n; ++k)
    m = max(m, bits_of(mag(g[0][k]) | mag(g[1][k]) | mag(g[2][k])) - tij - P.fx.ti[k] + 64);
  Max::put(smax[1], le, m);
  __syncthreads();  // and every forward read of S0 is done
  const int up1 = kBits + 64 - Max::get(smax[1], le);  // |g| 2^(up1 - t) < 2^60
  ex -= up1;

  // (wr, ws, wt) = G (ur, us, ut); g1..g6 = G_rr, G_ss, G_tt, G_rs, G_rt, G_st
  m = 0;
  if (act) {
    const int4* Ge = P.fx.G + e * 3 * n3 + ij;
#pragma unroll
    for (int k = 0; k < n; ++k) {
      const int4 x0 = __ldg(Ge + k * n2), x1 = __ldg(Ge + n3 + k * n2), x2 = __ldg(Ge + 2 * n3 + k * n2);
      const int s = up1 - tij - P.fx.ti[k];
      const int2 v[3] = {split(shift(g[0][k], s)), split(shift(g[1][k], s)), split(shift(g[2][k], s))};
      const int2 g1 = make_int2(x0.x, x0.y), g2 = make_int2(x0.z, x0.w), g3 = make_int2(x1.x, x1.y);
      const int2 g4 = make_int2(x1.z, x1.w), g5 = make_int2(x2.x, x2.y), g6 = make_int2(x2.z, x2.w);
      const int2 r0[3] = {g1, g4, g5}, r1[3] = {g4, g2, g6}, r2[3] = {g5, g6, g3};
      g[0][k] = dot<3>(r0, v);
      g[1][k] = dot<3>(r1, v);
      g[2][k] = dot<3>(r2, v);
      m |= mag(g[0][k]) | mag(g[1][k]) | mag(g[2][k]);
    }
  }
  Max::put(smax[2], le, bits_of(m));
  __syncthreads();
  const int up2 = kBits - Max::get(smax[2], le);
  ex += 64 - sG - up2;
  int2 wt[n];
#pragma unroll
  for (int k = 0; k < n; ++k) {
    S0[k * PL + j * RP + i] = split(shl(g[0][k], up2));
    S1[k * PL + j * RP + i] = split(shl(g[1][k], up2));
    wt[k] = split(shl(g[2][k], up2));
  }
  __syncthreads();

  ex += 64 - P.fx.sc[1];
  const int2* sT = sD + n * RP;
  double pw = 0.0;  // this thread's part of <p, A_L p>
  if (act && !slow) {
    ll ph = 0, pm = 0;
    MassTerm mt;
    int ec = ex;  // the column's coarsest unit
    if (P.helm) {
      mt.init(P.h2, P.fx.eB[e], expo(ehi));
      ec = max(ex, mt.em - tij);
    }
#pragma unroll
    for (int k = 0; k < n; ++k) {
      // the three directions separately: each sum has the headroom of its own row
      Dot r, s, t;
#pragma unroll
      for (int l = 0; l < n; ++l) {
        r.add(sT[i * RP + l], S0[k * PL + j * RP + l]);
        s.add(sT[j * RP + l], S1[k * PL + l * RP + i]);
        t.add(sT[k * RP + l], wt[l]);
      }
      ll o = r.get() + s.get() + t.get();
      int eo = ex;
      if (P.helm) mt.add(o, eo, __ldg(P.B + base + k * n2), ru[k], tij + P.fx.ti[k]);
      P.w[base + k * n2] = to_double(o, eo);
      if (FUSED) {
        const int2 y = split((o >> 5) >> min(ec - eo, 58));
        ph = mad(ph, ru[k].y, y.y);
        pm = mad(mad(pm, ru[k].x, y.y), ru[k].y, y.x);
      }
    }
    if (FUSED) pw = ldexp(__ll2double_rn(ph + (pm >> 32)), 64 + 5 + ec + expo(ehi) - 1022 - kBits);
  } else if (act) {
    const double* v = FUSED ? (P.pout ? P.pout : P.p) : P.u;
#pragma unroll 1
    for (int k = 0; k < n; ++k) {
      const double r = slow_point<N>(P, v, e, i, j, k);
      P.w[base + k * n2] = r;
      if (FUSED) pw += v[base + k * n2] * r;
    }
  }

  if (FUSED) {  // this block's part of <p, A_L p>; k_pap_finish sums the parts in block order
    const double s = block_sum(pw, sred);
    if (tid == 0) P.partial[blockIdx.x] = s;
  }
}

template <int N, int EPB, bool FUSED>
cudaError_t launch_fxd_t(const AxParams<double>& p, cudaStream_t s, int* grid_out) {
  constexpr int n = N + 1;
  const size_t smem = sizeof(int2) * (2ull * n * (n + 1) + 2ull * EPB * n * n * (n + 1));
  static DeviceOnce once;
  cudaError_t aerr = once.get([&](int, int*) {
    return cudaFuncSetAttribute(k_ax_fxd<N, EPB, FUSED>, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem);
  });
  if (aerr != cudaSuccess) return aerr;
  const int64_t grid = (p.E + EPB - 1) / EPB;
  if (grid_out) *grid_out = (int)grid;
  if (p.E == 0) return cudaSuccess;
  k_ax_fxd<N, EPB, FUSED><<<(unsigned)grid, EPB * n * n, smem, s>>>(p);
  cudaError_t err = cudaGetLastError();
  if (FUSED && err == cudaSuccess) err = launch_pap_finish(p.partial, (int)grid, p.st, s);
  return err;
}

}  // namespace fxk
}  // namespace sem
