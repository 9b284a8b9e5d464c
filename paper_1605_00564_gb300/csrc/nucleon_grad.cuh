// Derivative of the projected nucleon two-point contraction with respect to
// the point-source propagators of its quark lines, per site.  Shared by the
// Feynman-Hellmann gradient (fh.cu, weights over all time-slices) and the
// sequential sources of the three-point functions (threept.cu, one sink
// time-slice).
//
// C(x) = tr[P(t) G(x)] with G(x) = F(S_u, S_d, S_u)(x) the trilinear Wick
// form of eq. Nop (the diquark's u quark, the d quark, the third quark; the
// two Wick terms differ in which u-bar each u meets) and P(t) a 4x4 complex
// matrix per time-slice.  The kernel writes, for f = u and d,
//     H_f(x) = conj( dC(x) / dS_f(x) )          (12 x 12 per site)
// summed over the slots of flavour f, in the propagator's layout (field
// rhs = 3 alpha' + colour', component 3 alpha + colour).
//
// In the diquark form (nucleon_diquark.cuh), with the u and d propagators kept
// apart,
//   C = - sum_{cc'} tr[ R^{cc'} N^{cc'} ],  N^{cc'} = tr[P U^{cc'}] 1 + U^{cc'} P,
//   R^{cc'} = - sum_{x != c, x' != c'} s s' U^{xx'} D^{yy'}^T   (hat on D),
// y, y' the remaining colours and s = +1 if x follows c cyclically, else -1 (s'
// likewise).  At U = D = S its derivatives are, per colour pair (x, x'),
//   dC/dU^{xx'} = [ - tr R^{xx'} P - P R^{xx'} + sum s s' S^{yy'}^T N^{cc'} ]^T
//   dC/dD^{xx'} = hat( sum s s' N^{cc'} S^{yy'} )
// (sums over the four (c, c') with c != x, c' != x'): eight 4x4 products a pair,
// about 6,300 complex multiply-adds a site against 16,600 of the sum over the 36
// colour permutations with its repeated products.  Bound by the FP64 pipe; that form
// also spilled its 4x4 blocks and took 143 ms on 16^3x32 (all time-slices), this one
// about 10 (the gradient call 296 -> 114 ms with the faster SAP sweep).
//
// P(t) has entries (k, k) and (k, k^2) only: true of P+-, of P+- g5 g3 and of
// any combination of them (g0 and g3 both couple spin k to k^2).
#pragma once

#include "nucleon_diquark.cuh"

namespace nucleon_grad {
namespace {

using C64 = Cplx<double>;
using diquark::cmsub;

// sites of one CTA: the largest power of two <= MAX_SITES dividing the spatial volume
constexpr int MAX_SITES = 16;
inline int sites_per_cta(long long L3) {
  int ns = MAX_SITES;
  while (L3 % ns) ns >>= 1;
  return ns;
}
inline int cta_threads(int ns) { return 9 * ns; }
// S and N of the CTA's sites
inline size_t cta_smem(int ns) { return (size_t)2 * 144 * ns * sizeof(C64); }

// a * +-1 by the sign bit (integer units; the FP64 pipe is the bound)
__device__ inline double flip_sign(double a, int mask) {
  return __hiloint2double(__double2hiint(a) ^ mask, __double2loint(a));
}
__device__ inline C64 flip_sign(C64 a, int mask) { return cmk(flip_sign(a.re, mask), flip_sign(a.im, mask)); }

// H_f for ns sites per CTA, the CTAs covering the sites site0, site0 + 1, ...;
// thread = (site i, colour pair (x, x')), first flavour u, then d.  pmat[t]: the
// 4x4 complex matrix P(t) (row major) of time-slice t.  prop: internal FP64
// layout, 12 fields; H: internal FP64 layout, 24 fields (u then d),
// rhs = 3 alpha' + x'.
__global__ void __launch_bounds__(144) k_dC_dS(const double2* __restrict__ prop, const double2* __restrict__ pmat,
                                               int V, int L3, int ns, int site0, double2* __restrict__ H) {
  extern __shared__ __align__(16) unsigned char smem_raw[];
  C64* S_s = (C64*)smem_raw;
  C64* N_s = S_s + (size_t)144 * ns;
  const int s0 = site0 + blockIdx.x * ns;
  for (int idx = threadIdx.x; idx < 144 * ns; idx += blockDim.x) {
    const int i = idx % ns, e = idx / ns;
    const double2 v = __ldg(prop + (size_t)e * V + s0 + i);
    S_s[idx] = cmk(v.x, v.y);
  }
  __syncthreads();
  const int i = threadIdx.x % ns, o = threadIdx.x / ns;
  const int x = o / 3, xp = o - 3 * x;
  auto get = [&](int al, int a, int alp, int ap) { return S_s[(12 * (3 * alp + ap) + 3 * al + a) * ns + i]; };
  const int t = (s0 + i) / L3;
  C64 pd[4], po[4];   // P_kk and P_{k, k^2}
#pragma unroll
  for (int k = 0; k < 4; k++) {
    const double2 u = pmat[16 * t + 5 * k], v = pmat[16 * t + 4 * k + (k ^ 2)];
    pd[k] = cmk(u.x, u.y);
    po[k] = cmk(v.x, v.y);
  }
  // acc[j][k] = dC/dS_u(j, k): the third quark's part, -(tr R P + P R)_{kj}
  C64 acc[4][4];
#pragma unroll
  for (int j = 0; j < 4; j++)
#pragma unroll
    for (int k = 0; k < 4; k++) acc[j][k] = cmk(0.0, 0.0);
  {
    C64 r[6];
    diquark::diquark_r<double>(get, x, xp, r);
    const C64 tr = 2.0 * (r[0] + r[5]);
#pragma unroll
    for (int k = 0; k < 4; k++) {
      cmsub(acc[k][k], tr, pd[k]);
      cmsub(acc[k ^ 2][k], tr, po[k]);
    }
    // R entry (a, j) = rv: (P R)_{aj} takes P_aa, (P R)_{a^2, j} takes P_{a^2, a}
    auto add = [&](int a, int j, C64 rv) {
      cmsub(acc[j][a], pd[a], rv);
      cmsub(acc[j][a ^ 2], po[a ^ 2], rv);
    };
#pragma unroll
    for (int m = 0; m < 6; m++) {
      const int a = diquark::r_row(m), j = diquark::r_col(m);
      add(a, j, r[m]);
      add(j ^ 1, a ^ 1, diquark::gsgn(a) * diquark::gsgn(j) > 0 ? r[m] : -r[m]);
    }
  }
  {
    // N = tr[P S] 1 + S P
    C64 Z[4][4], n[4][4], tr = cmk(0.0, 0.0);
#pragma unroll
    for (int a = 0; a < 4; a++)
#pragma unroll
      for (int b = 0; b < 4; b++) Z[a][b] = get(a, x, b, xp);
#pragma unroll
    for (int k = 0; k < 4; k++) {
      cmac(tr, pd[k], Z[k][k]);
      cmac(tr, po[k], Z[k ^ 2][k]);
    }
#pragma unroll
    for (int a = 0; a < 4; a++)
#pragma unroll
      for (int b = 0; b < 4; b++) {
        n[a][b] = a == b ? tr : cmk(0.0, 0.0);
        cmac(n[a][b], Z[a][b], pd[b]);
        cmac(n[a][b], Z[a][b ^ 2], po[b ^ 2]);
        N_s[(16 * o + 4 * a + b) * ns + i] = n[a][b];
      }
  }
  __syncthreads();
  // the diquark parts: the four (c, c') with c = x + 1, x + 2 and c' likewise; the
  // sign is that of the two cyclic steps, y and y' the remaining colours
#pragma unroll 1
  for (int q = 0; q < 4; q++) {
    const int dc = 1 + (q & 1), dp = 1 + (q >> 1);
    const int c = (x + dc) % 3, cp = (xp + dp) % 3, y = 3 - x - c, yp = 3 - xp - cp;
    const int mask = dc != dp ? (int)0x80000000 : 0;
    const C64* n = N_s + (size_t)(16 * (3 * c + cp)) * ns + i;
#pragma unroll
    for (int a = 0; a < 4; a++) {
      // (S^{yy'}^T N)_{kj} += g(a) g(k) S_{a^1, k^1} N_{aj}
      C64 nr[4], sr[4];
#pragma unroll
      for (int j = 0; j < 4; j++) nr[j] = flip_sign(n[(4 * a + j) * ns], mask);
#pragma unroll
      for (int k = 0; k < 4; k++) sr[k] = get(a ^ 1, y, k ^ 1, yp);
#pragma unroll
      for (int k = 0; k < 4; k++)
#pragma unroll
        for (int j = 0; j < 4; j++) {
          if (diquark::gsgn(a) * diquark::gsgn(k) > 0) cmac(acc[j][k], sr[k], nr[j]);
          else cmsub(acc[j][k], sr[k], nr[j]);
        }
    }
  }
  // H = conj(dC/dS): entry (al, al') -> field rhs = 3 al' + x', component 3 al + x
#pragma unroll
  for (int al = 0; al < 4; al++)
#pragma unroll
    for (int alp = 0; alp < 4; alp++)
      H[((size_t)(3 * alp + xp) * 12 + 3 * al + x) * V + s0 + i] = make_double2(acc[al][alp].re, -acc[al][alp].im);
#pragma unroll
  for (int j = 0; j < 4; j++)
#pragma unroll
    for (int k = 0; k < 4; k++) acc[j][k] = cmk(0.0, 0.0);
#pragma unroll 1
  for (int q = 0; q < 4; q++) {
    const int dc = 1 + (q & 1), dp = 1 + (q >> 1);
    const int c = (x + dc) % 3, cp = (xp + dp) % 3, y = 3 - x - c, yp = 3 - xp - cp;
    const int mask = dc != dp ? (int)0x80000000 : 0;
    const C64* n = N_s + (size_t)(16 * (3 * c + cp)) * ns + i;
#pragma unroll
    for (int k = 0; k < 4; k++) {
      C64 nc[4], sr[4];
#pragma unroll
      for (int a = 0; a < 4; a++) nc[a] = flip_sign(n[(4 * a + k) * ns], mask);
#pragma unroll
      for (int b = 0; b < 4; b++) sr[b] = get(k, y, b, yp);
#pragma unroll
      for (int a = 0; a < 4; a++)
#pragma unroll
        for (int b = 0; b < 4; b++) cmac(acc[a][b], nc[a], sr[b]);
    }
  }
  double2* Hd = H + (size_t)144 * V;
#pragma unroll
  for (int al = 0; al < 4; al++)
#pragma unroll
    for (int alp = 0; alp < 4; alp++) {
      const C64 z = acc[al ^ 1][alp ^ 1];
      const double sg = (double)(diquark::gsgn(al) * diquark::gsgn(alp));
      Hd[((size_t)(3 * alp + xp) * 12 + 3 * al + x) * V + s0 + i] = make_double2(sg * z.re, -sg * z.im);
    }
}

}  // namespace
}  // namespace nucleon_grad
