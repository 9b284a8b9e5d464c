// Kernels of the nucleon two-point function (eq. Nop and the P+- projections
// of Sec. 2.3), shared by qcd_nucleon_2pt (internal propagator layout) and
// qcd_nucleon_2pt_noalloc (canonical layout).
//
// N_alpha = eps^{abc} (u^a^T G d^b) u^c_alpha, G = C g5, C = g0 g2; with u = d
// and one point-source propagator S (12x12 per site, S^{a a'}_{alpha alpha'}),
// the Wick contractions give
//   G(x) = eps^{abc} eps^{a'b'c'} { S^{cc'} tr[S^{aa'T} G S^{bb'} G']
//                                   - S^{ca'} G'^T S^{bb'T} G^T S^{ac'} },
// G' = g0 G^+ g0^T.  In the chiral basis G = diag(J, J), J = [[0,-1],[1,0]],
// and G' = -G, so both are signed permutations: G_{b, b^1} = g(b) and
// G'_{b^1, b} = g(b) with g(b) = -1 for even b, +1 for odd b.  Hence
//   tr[S^{aa'T} G S^{bb'} G'] = sum_{b,b'} g(b) g(b') S^{aa'}_{b b'} S^{bb'}_{b^1 b'^1}
//   (G'^T S^{bb'T} G^T)_{ij} = g(i) g(j) S^{bb'}_{j^1 i^1}
// and with P+- = (1 +- g0)/2, tr[P+- Z] = (1/2) sum_l (Z_{ll} -+ Z_{l^2, l}).
//
// Evaluated in the diquark form (nucleon_diquark.cuh):
//   tr[P+- G] = - sum_{cc'} ( tr R^{cc'} tr[P+- S^{cc'}] + tr[P+- R^{cc'} S^{cc'}] ).
//
// Layout: 9 threads per site, one per colour pair (c, c').  A CTA covers NS
// consecutive sites of one timeslice (NS a power of two dividing the spatial
// volume, so a CTA never straddles two timeslices); the propagator of those
// sites is staged in shared memory (the 144 complex entries of a site are read
// by its 9 threads; entry stride NS + 1, so that the canonical layout, whose
// consecutive words are the components of one site, stages without bank
// conflicts).  The CTA has 9 NS threads rounded up to whole warps; the padding
// threads stage but contribute zero to the sums, so every warp of the
// shuffle reduction is full.  The CTA's sum over its sites is written to a
// partial; a second kernel sums the partials of each timeslice in a fixed
// order, re-references the time to the source and applies the boundary sign
// of wrapped sink times.
//
// FP64 is bound by the FP64 pipe (1.25 TFLOP/s), so the operation count sets the
// time: 24^3x48 in 31.3 ms summed over the 36 colour permutations, 5.2 ms in this
// form (the whole call, reading the canonical propagator); the pipe is active 95 % of
// the time.  FP32 has the same bound, from the conversions of the FP64 propagator's 288
// words a site and the sums across threads (pipe active 77 %, DRAM at 25 % of its rate).
#pragma once

#include "nucleon_diquark.cuh"

// an unnamed namespace: each translation unit that includes this header
// gets its own copy of the kernels
namespace nucleon {
namespace {

// threads of a CTA covering ns sites: 9 ns rounded up to a multiple of 32
inline int cta_threads(int ns) { return (9 * ns + 31) & ~31; }
// dynamic shared memory of a CTA
template <typename R>
inline size_t cta_smem(int ns) { return (size_t)144 * (ns + 1) * sizeof(Cplx<R>); }

// CANONICAL = true: prop is [rhs][site][spin][colour] complex FP64 (the C-ABI
// layout); false: the internal FP64 spinor layout double2 [rhs][12][V].
template <typename R, bool CANONICAL>
__global__ void __launch_bounds__(288) k_sites(const double2* __restrict__ prop, int V, int ns,
                                               double2* __restrict__ part) {
  extern __shared__ __align__(16) unsigned char smem_raw[];
  Cplx<R>* S_s = (Cplx<R>*)smem_raw;
  const int s0 = blockIdx.x * ns, st = ns + 1;
  // stage: entry e = 12 rhs + comp of site s0 + i at S_s[e * st + i]
  for (int idx = threadIdx.x; idx < 144 * ns; idx += blockDim.x) {
    int i, e;
    double2 v;
    if (CANONICAL) {
      const int rhs = idx / (12 * ns), rem = idx - rhs * 12 * ns;
      i = rem / 12;
      e = 12 * rhs + rem - 12 * i;
      v = __ldg(prop + ((size_t)rhs * V + s0) * 12 + rem);
    } else {
      i = idx % ns;
      e = idx / ns;
      v = __ldg(prop + (size_t)e * V + s0 + i);
    }
    S_s[e * st + i] = cmk((R)v.x, (R)v.y);
  }
  __syncthreads();

  Cplx<R> accp = cmk((R)0, (R)0), accm = cmk((R)0, (R)0);
  if (threadIdx.x < 9 * ns) {
    const int i = threadIdx.x % ns;
    const int o = threadIdx.x / ns;
    const int c = o / 3, cp = o - 3 * c;
    auto get = [&](int al, int a, int alp, int ap) { return S_s[(12 * (3 * alp + ap) + 3 * al + a) * st + i]; };
    Cplx<R> r[6];
    diquark::diquark_r<R>(get, c, cp, r);
    Cplx<R> Z[4][4];
#pragma unroll
    for (int l = 0; l < 4; l++)
#pragma unroll
      for (int k = 0; k < 4; k++) Z[l][k] = get(l, c, k, cp);
    // tr S, tr[g0 S] = -o, tr[R S] and tr[g0 R S] = -zo over the independent entries of R
    Cplx<R> d = Z[0][0], q = Z[2][0], zd = cmk((R)0, (R)0), zo = cmk((R)0, (R)0);
#pragma unroll
    for (int l = 1; l < 4; l++) {
      d = d + Z[l][l];
      q = q + Z[l ^ 2][l];
    }
#pragma unroll
    for (int m = 0; m < 6; m++) {
      const int ii = diquark::r_row(m), j = diquark::r_col(m);
      if (diquark::gsgn(ii) * diquark::gsgn(j) > 0) {
        cmac(zd, r[m], Z[j][ii] + Z[ii ^ 1][j ^ 1]);
        cmac(zo, r[m], Z[j][ii ^ 2] + Z[ii ^ 1][j ^ 3]);
      } else {
        cmac(zd, r[m], Z[j][ii] - Z[ii ^ 1][j ^ 1]);
        cmac(zo, r[m], Z[j][ii ^ 2] - Z[ii ^ 1][j ^ 3]);
      }
    }
    // tr R / 2 = R_00 + R_22; tr[P+- X] = (tr X +- tr[g0 X]) / 2
    const Cplx<R> tr = r[0] + r[5];
    if constexpr (sizeof(R) == 4) {   // (fewer roundings; FP64 keeps its bits)
      accp = (R)0.5 * (zo - zd);
      accm = (R)-0.5 * (zd + zo);
      cmac(accp, -tr, d - q);
      cmac(accm, -tr, d + q);
    } else {
      accp = -(tr * (d - q) + (R)0.5 * (zd - zo));
      accm = -(tr * (d + q) + (R)0.5 * (zd + zo));
    }
  }
  // CTA sum (fixed order): warp shuffles over full warps, then one thread
  // over the warp sums
  __shared__ double red[4][32];
  double v[4] = {(double)accp.re, (double)accp.im, (double)accm.re, (double)accm.im};
#pragma unroll
  for (int k = 0; k < 4; k++)
#pragma unroll
    for (int off = 16; off > 0; off >>= 1) v[k] += __shfl_xor_sync(0xffffffffu, v[k], off);
  const int w = threadIdx.x >> 5, lane = threadIdx.x & 31, nw = blockDim.x >> 5;
  if (lane == 0)
    for (int k = 0; k < 4; k++) red[k][w] = v[k];
  __syncthreads();
  if (threadIdx.x == 0) {
    double t[4] = {0, 0, 0, 0};
    for (int ww = 0; ww < nw; ww++)
      for (int k = 0; k < 4; k++) t[k] += red[k][ww];
    part[2 * (size_t)blockIdx.x] = make_double2(t[0], t[1]);
    part[2 * (size_t)blockIdx.x + 1] = make_double2(t[2], t[3]);
  }
}

// one CTA of 256 threads per timeslice: corr[p][trel] = sign * sum of the
// partials of timeslice t
__global__ void k_timeslices(const double2* __restrict__ part, int per_t, int T, int t0, int bc3,
                             double2* __restrict__ corr) {
  const int t = blockIdx.x;
  __shared__ double2 sh[2][256];
  double2 ap = make_double2(0, 0), am = make_double2(0, 0);
  for (int k = threadIdx.x; k < per_t; k += blockDim.x) {
    const double2 p = part[2 * ((size_t)t * per_t + k)], m = part[2 * ((size_t)t * per_t + k) + 1];
    ap.x += p.x; ap.y += p.y; am.x += m.x; am.y += m.y;
  }
  sh[0][threadIdx.x] = ap;
  sh[1][threadIdx.x] = am;
  __syncthreads();
  for (int st = blockDim.x / 2; st > 0; st >>= 1) {
    if (threadIdx.x < st) {
      sh[0][threadIdx.x].x += sh[0][threadIdx.x + st].x; sh[0][threadIdx.x].y += sh[0][threadIdx.x + st].y;
      sh[1][threadIdx.x].x += sh[1][threadIdx.x + st].x; sh[1][threadIdx.x].y += sh[1][threadIdx.x + st].y;
    }
    __syncthreads();
  }
  if (threadIdx.x == 0) {
    const int trel = (t - t0 + T) % T;
    const double sg = (t < t0) ? (double)bc3 : 1.0;
    corr[trel] = make_double2(sg * sh[0][0].x, sg * sh[0][0].y);
    corr[T + trel] = make_double2(sg * sh[1][0].x, sg * sh[1][0].y);
  }
}

// sites per CTA: the largest power of two <= MAX_SITES dividing the spatial volume
constexpr int MAX_SITES = 32;
inline int sites_per_cta(long long L3) {
  int ns = MAX_SITES;
  while (L3 % ns) ns >>= 1;
  return ns;
}

}  // namespace
}  // namespace nucleon
