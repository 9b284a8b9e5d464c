// The diquark factor of the nucleon's Wick contractions, shared by the
// two-point function (nucleon_kernels.cuh) and its derivative
// (nucleon_grad.cuh).
//
// With S^{ab} the 4x4 spin matrices of one site's propagator (a sink, b source
// colour), Y^ = G Y G' (G = C g5 = diag(J, J), G' = -G, J = [[0,-1],[1,0]], so
// Y^_{ij} = g(i) g(j) Y_{i^1, j^1}, g = -1 for even and +1 for odd indices) and
// u = d, both Wick terms of eq. Nop,
//   tr[P G] = eps eps' { tr[P S^{cc'}] tr[S^{aa'T} S^{bb'}^] - tr[P S^{ca'} S^{bb'}^T S^{ac'}] },
// contain the same sums over two of the three quark lines: summed over the
// colours, tr[P G] = - sum_{cc'} ( tr R tr[P S^{cc'}] + tr[P R S^{cc'}] ) with
//   R^{cc'} = S^{21'} S^{12'}^T - S^{22'} S^{11'}^T - S^{11'} S^{22'}^T + S^{12'} S^{21'}^T
// (1, 2 = c+1, c+2 and 1', 2' = c'+1, c'+2 mod 3).  The last two products are
// the first two with rows and columns exchanged by j -> i^1, so
//   R_{ij} = g(j) W_{i, j^1},   W_{uv} = -W_{vu}
//   W_{uv} = sum_k g(k) ( X1_{uk} Y2_{v,k^1} - X1_{vk} Y2_{u,k^1} - X2_{uk} Y1_{v,k^1} + X2_{vk} Y1_{u,k^1} )
// with X1 = S^{21'}, X2 = S^{22'}, Y1 = S^{11'}, Y2 = S^{12'}: six numbers per
// colour pair from 96 complex multiply-adds.  (The 36 colour permutations of the
// two epsilons need 4032 a site; this form about 1000.)
#pragma once

#include "qcd_internal.cuh"

namespace diquark {
namespace {

// acc -= a * b
template <typename R>
__device__ inline void cmsub(Cplx<R>& acc, Cplx<R> a, Cplx<R> b) {
  acc.re = rfma(-a.re, b.re, acc.re);
  acc.re = rfma(a.im, b.im, acc.re);
  acc.im = rfma(-a.re, b.im, acc.im);
  acc.im = rfma(-a.im, b.re, acc.im);
}

// the entries (i, j) of R that determine it (R_{j^1, i^1} = g(i) g(j) R_{ij}, R_{i, i^1} = 0)
__host__ __device__ constexpr int r_row(int m) { return m < 3 ? 0 : m < 5 ? 1 : 2; }
__host__ __device__ constexpr int r_col(int m) { return m == 0 ? 0 : (m == 2 || m == 4) ? 3 : 2; }
__host__ __device__ constexpr int gsgn(int b) { return (b & 1) ? 1 : -1; }

// R_{r_row(m), r_col(m)} of the colour pair (c, cp); get(al, a, alp, ap) reads S.  FP32:
// four products at a time, since one chain of 16 made the correlator's rounding error 1.25
// times that of the 36 permutations (1.18e-7 of the rms on random propagators; 0.93e-7 so).
// FP64 has no use for the additions, which it would take 12 % longer for.
template <typename R, typename Get>
__device__ inline void diquark_r(Get get, int c, int cp, Cplx<R> (&r)[6]) {
  const int x1 = c == 2 ? 0 : c + 1, x2 = c == 0 ? 2 : c - 1;
  const int y1 = cp == 2 ? 0 : cp + 1, y2 = cp == 0 ? 2 : cp - 1;
#pragma unroll
  for (int m = 0; m < 6; m++) r[m] = cmk((R)0, (R)0);
  constexpr bool single = sizeof(R) == 4;
#pragma unroll
  for (int k = 0; k < 4; k++) {
    Cplx<R> X1[4], X2[4], Y1[4], Y2[4];
#pragma unroll
    for (int u = 0; u < 4; u++) {
      X1[u] = get(u, x2, k, y1);
      X2[u] = get(u, x2, k, y2);
      Y1[u] = get(u, x1, k ^ 1, y1);
      Y2[u] = get(u, x1, k ^ 1, y2);
    }
#pragma unroll
    for (int m = 0; m < 6; m++) {
      const int u = r_row(m), v = r_col(m) ^ 1;
      Cplx<R> s = single ? cmk((R)0, (R)0) : r[m];
      if (gsgn(k) * gsgn(r_col(m)) > 0) {
        cmac(s, X1[u], Y2[v]);
        cmsub(s, X1[v], Y2[u]);
        cmsub(s, X2[u], Y1[v]);
        cmac(s, X2[v], Y1[u]);
      } else {
        cmsub(s, X1[u], Y2[v]);
        cmac(s, X1[v], Y2[u]);
        cmac(s, X2[u], Y1[v]);
        cmsub(s, X2[v], Y1[u]);
      }
      r[m] = single ? r[m] + s : s;
    }
  }
}

}  // namespace
}  // namespace diquark
