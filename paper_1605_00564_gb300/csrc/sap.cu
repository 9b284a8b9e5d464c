// Schwarz alternating procedure (Sec. 2.2).
//
// The lattice is split into blocks of extent b = (bt, bx, by, bz) coloured
// as a checkerboard (colour = parity of the block coordinates); D_Omega is the
// operator restricted to the black blocks with the hops that leave a block
// dropped (Dirichlet), D_dOmega* the hops from Omega into the white blocks.
// n_cy cycles, each visiting all black then all white blocks, applied to
// psi = 0 give M_SAP = K sum_{nu<n_cy} (1 - D K)^nu.
//
// Residual form of a half-cycle on colour c (rho = eta - D psi):
//   on every block L of colour c:  x = approx D_L^-1 rho_L (n_mr MR steps from 0),
//                                   psi_L += x,  rho_L = rho_L - D_L x,  delta_L = x
//   on the neighbouring sites y of the other colour: rho(y) -= (D delta)(y)
// The last line touches only blocks of the other colour, which are the next
// half-cycle's blocks, so it is applied there as a gather at the start of the
// next sweep: each site at a block face adds kappa * hop(delta) from the
// neighbouring block (delta of the previous half-cycle).  No two CTAs write
// the same word, so the result does not depend on scheduling.
//
// One CTA per block and right-hand side, one thread per block site; the
// block's residual lives in shared memory across the MR steps, the solution
// increment x in registers.
#include <string.h>

#include <type_traits>

#include <cooperative_groups.h>
#include <cuda_bf16.h>
#include <cuda_fp16.h>

#include "spin_pair.cuh"

namespace {

struct SapGeom {
  int b[4];     // block extents by direction (t, x, y, z)
  int nb[4];    // blocks per direction
  int lst[4];   // local stride of direction mu inside a block
  int vb;       // block volume
};

// the blk-th block of a colour
__device__ __forceinline__ void block_of(const SapGeom& sg, int colour, int blk, int bc[4]) {
  const int nbx2 = sg.nb[1] >> 1;
  int q = blk / nbx2;
  const int j = blk - q * nbx2;
  bc[2] = q % sg.nb[2];
  q /= sg.nb[2];
  bc[3] = q % sg.nb[3];
  bc[0] = q / sg.nb[3];
  bc[1] = 2 * j + ((colour + bc[0] + bc[3] + bc[2]) & 1);
}
// its number within its colour
__device__ __forceinline__ int block_number(const SapGeom& sg, const int bc[4]) {
  return ((bc[0] * sg.nb[3] + bc[3]) * sg.nb[2] + bc[2]) * (sg.nb[1] >> 1) + (bc[1] >> 1);
}

template <typename R>
__device__ inline Spinor<R> smem_load(const Cplx<R>* r_s, int vb, int l) {
  Spinor<R> o;
#pragma unroll
  for (int k = 0; k < 12; k++) o.c[k] = r_s[k * vb + l];
  return o;
}
template <typename R>
__device__ inline void smem_store(Cplx<R>* r_s, int vb, int l, const Spinor<R>& v) {
#pragma unroll
  for (int k = 0; k < 12; k++) r_s[k * vb + l] = v.c[k];
}

// p += scale * (hops of the block operator inside the block, applied to r_s)
template <typename F, int MU>
__device__ inline void block_hop(Spinor<typename F::R>& p, const Cplx<typename F::R>* r_s, const SapGeom& sg,
                                 const void* gauge, const Geom& g, int s, int l, const int lc[4],
                                 typename F::R scale) {
  using R = typename F::R;
  if (lc[MU] < sg.b[MU] - 1) {
    HalfSpinor<R> h = project<MU, -1>(smem_load(r_s, sg.vb, l + sg.lst[MU]));
    h = su3_mul(F::load_link(gauge, g.V, MU, s), h);
    accum_recon<MU, -1>(p, h, scale);
  }
  if (lc[MU] > 0) {
    HalfSpinor<R> h = project<MU, +1>(smem_load(r_s, sg.vb, l - sg.lst[MU]));
    h = su3_dag_mul(F::load_link(gauge, g.V, MU, s - g.stride[MU]), h);
    accum_recon<MU, +1>(p, h, scale);
  }
}

// r += scale * (hops from delta on the neighbouring blocks, across this block's faces)
template <typename F, int MU>
__device__ inline void face_hop(Spinor<typename F::R>& hop, const char* delta, const SapGeom& sg, const void* gauge,
                                const Geom& g, int s, const int c[4], const int lc[4], typename F::R scale) {
  using R = typename F::R;
  if (lc[MU] == sg.b[MU] - 1) {
    int sf = site_fwd(g, s, c, MU);
    R sign = (MU == 0 && c[0] == g.L[0] - 1) ? (R)g.bc_t * scale : scale;
    HalfSpinor<R> h = project<MU, -1>(F::load_spinor(delta, g.V, sf));
    h = su3_mul(F::load_link(gauge, g.V, MU, s), h);
    accum_recon<MU, -1>(hop, h, sign);
  }
  if (lc[MU] == 0) {
    int sb = site_bwd(g, s, c, MU);
    R sign = (MU == 0 && c[0] == 0) ? (R)g.bc_t * scale : scale;
    HalfSpinor<R> h = project<MU, +1>(F::load_spinor(delta, g.V, sb));
    h = su3_dag_mul(F::load_link(gauge, g.V, MU, sb), h);
    accum_recon<MU, +1>(hop, h, sign);
  }
}

template <typename R>
__device__ inline R warp_sum(R v) {
#pragma unroll
  for (int o = 16; o > 0; o >>= 1) v += __shfl_xor_sync(0xffffffffu, v, o);
  return v;
}

template <typename F, int MAXT, int MINB>
__global__ void __launch_bounds__(MAXT, MINB) k_sap_sweep(const char* __restrict__ rho_src, char* __restrict__ rho,
                                                          char* __restrict__ psi, char* __restrict__ delta,
                            const void* __restrict__ gauge, const void* __restrict__ clover, Geom g, SapGeom sg,
                            int colour, int gather, int psi_init, typename F::R kappa, int nmr, int nrhs,
                            const int* mask) {
  using R = typename F::R;
  extern __shared__ __align__(16) unsigned char smem_raw[];
  Cplx<R>* r_s = (Cplx<R>*)smem_raw;
  __shared__ R red[3][32];

  // the RHS index runs fastest over the grid: the CTAs of one block (all RHS)
  // are resident together and share its links and clover term through L2
  const int rhs = blockIdx.x % nrhs;
  const int blk = blockIdx.x / nrhs;
  if (mask && !mask[rhs]) return;
  const size_t off = (size_t)rhs * F::spinor_bytes * g.V;
  rho_src += off;
  rho += off;
  psi += off;
  delta += off;

  // which block: the blk-th block of this colour
  const int nbx2 = sg.nb[1] >> 1;
  int q = blk / nbx2;
  const int j = blk - q * nbx2;
  const int by = q % sg.nb[2];
  q /= sg.nb[2];
  const int bz = q % sg.nb[3];
  const int bt = q / sg.nb[3];
  const int bx = 2 * j + ((colour + bt + bz + by) & 1);

  const int l = threadIdx.x;
  int lc[4], c[4];
  {
    int r = l;
    lc[1] = r % sg.b[1]; r /= sg.b[1];
    lc[2] = r % sg.b[2]; r /= sg.b[2];
    lc[3] = r % sg.b[3];
    lc[0] = r / sg.b[3];
  }
  c[0] = bt * sg.b[0] + lc[0];
  c[1] = bx * sg.b[1] + lc[1];
  c[2] = by * sg.b[2] + lc[2];
  c[3] = bz * sg.b[3] + lc[3];
  const int s = ((c[0] * g.L[3] + c[3]) * g.L[2] + c[2]) * g.L[1] + c[1];

  // pending boundary update from the previous half-cycle
  Spinor<R> r = F::load_spinor(rho_src, g.V, s);
  if (gather) {
    face_hop<F, 0>(r, delta, sg, gauge, g, s, c, lc, kappa);
    face_hop<F, 1>(r, delta, sg, gauge, g, s, c, lc, kappa);
    face_hop<F, 2>(r, delta, sg, gauge, g, s, c, lc, kappa);
    face_hop<F, 3>(r, delta, sg, gauge, g, s, c, lc, kappa);
  }
  smem_store(r_s, sg.vb, l, r);

  Spinor<R> x;
#pragma unroll
  for (int k = 0; k < 12; k++) x.c[k] = cmk((R)0, (R)0);

  const int warp = l >> 5, lane = l & 31, nw = (sg.vb + 31) >> 5;
  for (int step = 0; step < nmr; step++) {
    __syncthreads();
    // p = D_L r
    Spinor<R> p = clover_apply<F>(clover, g.V, s, r);
    block_hop<F, 0>(p, r_s, sg, gauge, g, s, l, lc, -kappa);
    block_hop<F, 1>(p, r_s, sg, gauge, g, s, l, lc, -kappa);
    block_hop<F, 2>(p, r_s, sg, gauge, g, s, l, lc, -kappa);
    block_hop<F, 3>(p, r_s, sg, gauge, g, s, l, lc, -kappa);
    // alpha = (p, r) / (p, p) over the block
    Cplx<R> pr = cmk((R)0, (R)0);
    R pp = 0;
#pragma unroll
    for (int k = 0; k < 12; k++) {
      cmac_conj(pr, p.c[k], r.c[k]);
      pp = rfma(p.c[k].re, p.c[k].re, pp);
      pp = rfma(p.c[k].im, p.c[k].im, pp);
    }
    R pr_re = pr.re, pr_im = pr.im;
    pr_re = warp_sum(pr_re);
    pr_im = warp_sum(pr_im);
    pp = warp_sum(pp);
    if (lane == 0) {
      red[0][warp] = pr_re;
      red[1][warp] = pr_im;
      red[2][warp] = pp;
    }
    __syncthreads();
    R a_re = 0, a_im = 0, n2 = 0;
    for (int w = 0; w < nw; w++) {
      a_re += red[0][w];
      a_im += red[1][w];
      n2 += red[2][w];
    }
    Cplx<R> alpha = n2 > (R)0 ? cmk(a_re / n2, a_im / n2) : cmk((R)0, (R)0);
    const Cplx<R> malpha = -alpha;
#pragma unroll
    for (int k = 0; k < 12; k++) {
      cmac(x.c[k], alpha, r.c[k]);
      cmac(r.c[k], malpha, p.c[k]);
    }
    __syncthreads();
    smem_store(r_s, sg.vb, l, r);
  }

  if (psi_init) {
    F::store_spinor(psi, g.V, s, x);
  } else {
    Spinor<R> y = F::load_spinor(psi, g.V, s);
#pragma unroll
    for (int k = 0; k < 12; k++) y.c[k] = y.c[k] + x.c[k];
    F::store_spinor(psi, g.V, s, y);
  }
  F::store_spinor(rho, g.V, s, r);
  F::store_spinor(delta, g.V, s, x);
}

// ---------------------------------------------------------------------------
// FP64, 4^4 blocks.  The FP64 pipe is the bound (a warp instruction takes the SM 16
// cycles, with however few lanes active), so no warp runs with idle lanes: hops are
// tasks, numbered over the sites that have a neighbour in the block (3/4 of them
// in every direction) or over the sites of a face (boundary term), and their
// results are added to the site's sum in shared memory, one direction and sign
// per round.  Per MR step and block 48 hops of a warp instead of 60 with one
// thread per site, in the boundary term 16 instead of 64.
//
// A block is spread over a cluster of two CTAs (time-slices 0-1 and 2-3) that read
// each other's residual through distributed shared memory: the units of work are
// coarse (8^3x16 with 12 RHS: 192 on 152 SMs).  Per half-cycle, one thread per site on
// one CTA -> tasks on one CTA -> tasks on two: 8^3x16, 12 RHS 770 -> 669 -> 531 us, one
// RHS 388 -> 337 -> 215; 16^3x32, 12 RHS 8.11 -> 7.12 -> 6.65 ms.  (Four CTAs of one
// time-slice leave half-empty warps again: 598 us and 7.96 ms.)
// ---------------------------------------------------------------------------
using CD = Cplx<double>;

__device__ __forceinline__ Spinor<double> sm_ld(const CD* b, int n, int l) {
  Spinor<double> o;
#pragma unroll
  for (int k = 0; k < 12; k++) {
    const double2 v = *(const double2*)(b + k * n + l);
    o.c[k] = cmk(v.x, v.y);
  }
  return o;
}
__device__ __forceinline__ void sm_st(CD* b, int n, int l, const Spinor<double>& v) {
#pragma unroll
  for (int k = 0; k < 12; k++) *(double2*)(b + k * n + l) = make_double2(v.c[k].re, v.c[k].im);
}

// o += scale * hop of r over link MU at site sl
template <int MU, bool FWD>
__device__ __forceinline__ void hop_d(Spinor<double>& o, const Spinor<double>& r, const void* gauge, int V, int sl,
                                      double scale) {
  HalfSpinor<double> h = project<MU, FWD ? -1 : +1>(r);
  if (FWD) h = su3_mul(FieldsD::load_link(gauge, V, MU, sl), h);
  else h = su3_dag_mul(FieldsD::load_link(gauge, V, MU, sl), h);
  accum_recon<MU, FWD ? -1 : +1>(o, h, scale);
}

struct BlockD {   // what the tasks need to know about the CTA's half of a block
  static constexpr int N = 128, NT = 2;   // sites, time-slices
  CD *r_s, *p_s;          // [12][N] residual and operator sum
  const CD* other;        // the other CTA's r_s
  const void* gauge;
  int co[4], t0, rank;    // first site of the block, first local time-slice
};
__device__ __forceinline__ int site_of(const BlockD& B, const Geom& g, int t, int x, int y, int z) {
  return (((B.co[0] + t) * g.L[3] + B.co[3] + z) * g.L[2] + B.co[2] + y) * g.L[1] + B.co[1] + x;
}

// one round of the block operator: p_s += scale * (hops in direction MU, one sign)
template <int MU, bool FWD>
__device__ __forceinline__ void hop_round(const BlockD& B, const Geom& g, int i, double scale) {
  constexpr int N = BlockD::N, NT = BlockD::NT;
  // sites with a neighbour: x, y, z: three of four coordinates; t: those whose
  // neighbour is in the block (here or in the other CTA)
  int x, y, z, t;   // t local to the CTA
  if (MU == 0) {
    const bool edge = FWD ? B.rank == 1 : B.rank == 0;   // the block ends on this side
    if (i >= 64 * (edge ? NT - 1 : NT)) return;
    x = i & 3; y = (i >> 2) & 3; z = (i >> 4) & 3; t = (i >> 6) + (!FWD && edge ? 1 : 0);
  } else {
    if (i >= N / 4 * 3) return;
    const int d = i / (N / 4), e = i % (N / 4), v = d + (FWD ? 0 : 1);   // the coordinate in MU, the others
    const int a = e & 3, b = (e >> 2) & 3;
    t = e >> 4;
    x = MU == 1 ? v : a;
    y = MU == 2 ? v : MU == 1 ? a : b;
    z = MU == 3 ? v : b;
  }
  const int l = ((t * 4 + z) * 4 + y) * 4 + x;
  constexpr int st = MU == 0 ? 64 : MU == 1 ? 1 : MU == 2 ? 4 : 16;
  int ln = l + (FWD ? st : -st);
  const CD* rb = B.r_s;
  if (MU == 0 && (ln < 0 || ln >= N)) {
    rb = B.other;
    ln += ln < 0 ? N : -N;
  }
  const int s = site_of(B, g, B.t0 + t, x, y, z);
  Spinor<double> p = sm_ld(B.p_s, N, l);
  hop_d<MU, FWD>(p, sm_ld(rb, N, ln), B.gauge, g.V, FWD ? s : s - g.stride[MU], scale);
  sm_st(B.p_s, N, l, p);
}

// boundary term of one direction: the hops from delta across the two MU faces
template <int MU>
__device__ __forceinline__ void gather_round(const BlockD& B, const Geom& g, const char* delta, int i,
                                             double kappa) {
  constexpr int N = BlockD::N, NT = BlockD::NT;
  constexpr int nf = MU == 0 ? 64 : N / 4;   // sites of one face in this CTA
  if (i >= 2 * nf) return;
  const bool fwd = i >= nf;
  const int e = fwd ? i - nf : i, a = e & 3, b = (e >> 2) & 3, d = e >> 4;
  int t, x, y, z;
  if (MU == 0) {
    if (fwd ? B.rank != 1 : B.rank != 0) return;
    x = a; y = b; z = d; t = fwd ? NT - 1 : 0;
  } else {
    const int v = fwd ? 3 : 0;
    t = d;
    x = MU == 1 ? v : a;
    y = MU == 2 ? v : MU == 1 ? a : b;
    z = MU == 3 ? v : b;
  }
  const int l = ((t * 4 + z) * 4 + y) * 4 + x, s = site_of(B, g, B.t0 + t, x, y, z);
  const int c[4] = {B.co[0] + B.t0 + t, B.co[1] + x, B.co[2] + y, B.co[3] + z};
  Spinor<double> r = sm_ld(B.r_s, N, l);
  if (fwd) {
    const double sc = (MU == 0 && c[0] == g.L[0] - 1) ? g.bc_t * kappa : kappa;
    hop_d<MU, true>(r, FieldsD::load_spinor(delta, g.V, site_fwd(g, s, c, MU)), B.gauge, g.V, s, sc);
  } else {
    const int sb = site_bwd(g, s, c, MU);
    const double sc = (MU == 0 && c[0] == 0) ? g.bc_t * kappa : kappa;
    hop_d<MU, false>(r, FieldsD::load_spinor(delta, g.V, sb), B.gauge, g.V, sb, sc);
  }
  sm_st(B.r_s, N, l, r);
}

// both CTAs of the block
__device__ __forceinline__ void sync_block() { cooperative_groups::this_cluster().sync(); }

// RES: CTAs that share an SM.  Three (168 registers, 300 bytes of spills) where two leave
// the last wave with one CTA per SM, whose four warps the FP64 pipe waits for; two (254
// registers) on up to 2 CTAs per SM in all, and on 3 to 4, where 2 + 2 beats 3 + 1.
// Measured with RES = 2 and 3, 8^3x16: 8 RHS (256 CTAs) 334 and 336 us, 10 to 14 (320 to
// 448) 531 and 494, 16 (512) 660 and 684, 20 (640) 853 and 816; 16^3x32: one RHS (512) 671
// and 693, two (1,024) 1,183 and 1,164, 12 6,646 and 6,551.
inline bool d4_three(unsigned ctas) {
  const unsigned per_sm = (ctas + 151) / 152;
  return per_sm > 2 && per_sm != 4;
}
template <int RES>
__global__ void __cluster_dims__(2, 1, 1) __launch_bounds__(128, RES)
    k_sap_sweep_d4(const char* __restrict__ rho_src, char* __restrict__ rho, char* __restrict__ psi,
                   char* __restrict__ delta, const void* __restrict__ gauge, const void* __restrict__ clover, Geom g,
                   SapGeom sg, int colour, int gather, int psi_init, int last, double kappa, int nmr, int nrhs,
                   const int* mask) {
  constexpr int N = BlockD::N, NW = N / 32;
  extern __shared__ __align__(16) unsigned char smem_raw[];
  __shared__ double red[2][3][NW];
  const int unit = blockIdx.x / 2;
  const int rhs = unit % nrhs;   // RHS fastest, as in k_sap_sweep
  const int blk = unit / nrhs;
  if (mask && !mask[rhs]) return;   // both CTAs of a cluster
  const size_t off = (size_t)rhs * FieldsD::spinor_bytes * g.V;
  rho_src += off;
  rho += off;
  psi += off;
  delta += off;
  int bc[4];
  block_of(sg, colour, blk, bc);
  BlockD B;
  B.r_s = (CD*)smem_raw;
  B.p_s = B.r_s + 12 * N;
  B.gauge = gauge;
  B.rank = blockIdx.x % 2;
  B.other = cooperative_groups::this_cluster().map_shared_rank(B.r_s, 1 - B.rank);
#pragma unroll
  for (int mu = 0; mu < 4; mu++) B.co[mu] = 4 * bc[mu];
  B.t0 = 2 * B.rank;
  const int l = threadIdx.x;
  const int s = site_of(B, g, B.t0 + (l >> 6), l & 3, (l >> 2) & 3, (l >> 4) & 3);

  Spinor<double> r = FieldsD::load_spinor(rho_src, g.V, s);
  sm_st(B.r_s, N, l, r);
  if (gather) {
    __syncthreads();
    gather_round<0>(B, g, delta, l, kappa);
    __syncthreads();
    gather_round<1>(B, g, delta, l, kappa);
    __syncthreads();
    gather_round<2>(B, g, delta, l, kappa);
    __syncthreads();
    gather_round<3>(B, g, delta, l, kappa);
    __syncthreads();
    r = sm_ld(B.r_s, N, l);
  }
  Spinor<double> x;
#pragma unroll
  for (int k = 0; k < 12; k++) x.c[k] = cmk(0.0, 0.0);
  const int warp = l >> 5, lane = l & 31;
  for (int step = 0; step < nmr; step++) {
    sm_st(B.p_s, N, l, clover_apply<FieldsD>(clover, g.V, s, r));
    sync_block();   // the residual of both CTAs and the sums are in place
    hop_round<0, true>(B, g, l, -kappa);
    __syncthreads();
    hop_round<0, false>(B, g, l, -kappa);
    __syncthreads();
    hop_round<1, true>(B, g, l, -kappa);
    __syncthreads();
    hop_round<1, false>(B, g, l, -kappa);
    __syncthreads();
    hop_round<2, true>(B, g, l, -kappa);
    __syncthreads();
    hop_round<2, false>(B, g, l, -kappa);
    __syncthreads();
    hop_round<3, true>(B, g, l, -kappa);
    __syncthreads();
    hop_round<3, false>(B, g, l, -kappa);
    __syncthreads();
    const Spinor<double> p = sm_ld(B.p_s, N, l);
    CD pr = cmk(0.0, 0.0);
    double pp = 0;
#pragma unroll
    for (int k = 0; k < 12; k++) {
      cmac_conj(pr, p.c[k], r.c[k]);
      pp = fma(p.c[k].re, p.c[k].re, pp);
      pp = fma(p.c[k].im, p.c[k].im, pp);
    }
    pr.re = warp_sum(pr.re);
    pr.im = warp_sum(pr.im);
    pp = warp_sum(pp);
    // two buffers: the other CTA may still read the last step's sums
    double(*rd)[NW] = red[step & 1];
    if (lane == 0) {
      rd[0][warp] = pr.re;
      rd[1][warp] = pr.im;
      rd[2][warp] = pp;
    }
    sync_block();   // also: both CTAs have read the other's residual
    double a[3] = {0, 0, 0};
#pragma unroll
    for (int q = 0; q < 2; q++) {   // CTA 0's sums first, for both
      const double* src = cooperative_groups::this_cluster().map_shared_rank(&rd[0][0], q);
#pragma unroll
      for (int k = 0; k < 3; k++)
#pragma unroll
        for (int w = 0; w < NW; w++) a[k] += src[k * NW + w];
    }
    const CD alpha = a[2] > 0 ? cmk(a[0] / a[2], a[1] / a[2]) : cmk(0.0, 0.0);
    const CD malpha = -alpha;
#pragma unroll
    for (int k = 0; k < 12; k++) {
      cmac(x.c[k], alpha, r.c[k]);
      cmac(r.c[k], malpha, p.c[k]);
    }
    sm_st(B.r_s, N, l, r);
  }
  if (psi_init) {
    FieldsD::store_spinor(psi, g.V, s, x);
  } else {
    Spinor<double> y = FieldsD::load_spinor(psi, g.V, s);
#pragma unroll
    for (int k = 0; k < 12; k++) y.c[k] = y.c[k] + x.c[k];
    FieldsD::store_spinor(psi, g.V, s, y);
  }
  // the last cycle's residuals and the last half-cycle's delta have no reader
  if (last < 1) FieldsD::store_spinor(rho, g.V, s, r);
  if (last < 2) FieldsD::store_spinor(delta, g.V, s, x);
  sync_block();   // the other CTA's last reads of this shared memory
}

// ---------------------------------------------------------------------------
// FP32 sweeps in two-lane arithmetic (spin_pair.cuh).
//
// Links and clover term come from a block image: for each block (all black
// blocks first, blk-th block of a colour as in the sweep) its sites' words in
// the order of the local index, so a block is one contiguous run.  Read from the
// lexicographic fields a warp's 32 sites of a 4^4 block are eight pieces of 64
// bytes in as many lines, and every word of a site is another page: such loads
// took 22,000 of the 56,000 clock cycles of a CTA.  S selects the image and how
// the MR steps use it:
//   __half     16-bit copies (uint4 [4][vb] entries 0-3 of the four links, uint4
//              [4][vb] entries 4-7, half2 [4][vb] entry 8, uint4 [9][vb] clover;
//              288 B a site), staged whole in shared memory.  The preconditioner
//              is then a slightly different operator, which the flexible outer
//              GCR tolerates;
//   float      FP32 (float4 [12][vb] link rows 0 and 1, float4 [18][vb] clover in
//              the order of CloverPairs; 480 B a site): links staged, clover
//              read from the image (L2) at every step.  With both staged a 4^4
//              block takes 147 KB and an SM holds one CTA, whose loads and
//              barriers nothing hides;
//   FromImage  the FP32 image read from L2 at every step (blocks of 257 to 512
//              sites, whose copies exceed shared memory, and blocks with an extent
//              of 1; 8 x 4^3 blocks have the sweep of their own below);
//   FromField  the same from the lexicographic fields, where there is no memory
//              for an image.
// Either staged form leaves room for two CTAs of a 4^4 block per SM.  Blocks of more
// than 512 sites stay with k_sap_sweep: at the 64 registers that 1024 threads leave it,
// the two-lane sweep spills 1.3 KB (8 x 8 x 4 x 4 blocks, 16^3x32, 2 cycles: 12 RHS
// 3.05 ms against 2.48, one RHS 540 us against 442).
// ---------------------------------------------------------------------------
struct FromImage {};
struct FromField {};

template <typename S>
struct Stage {   // bytes of shared memory per site for links and clover term
  static constexpr int bytes = std::is_same<S, __half>::value ? 288 : std::is_same<S, float>::value ? 192 : 0;
};

// where a block's links and clover term are (the members S uses)
struct BlockFields {
  const void* lk;         // links: shared memory or the block's image
  const void* cl;         // clover: likewise
  const float4* gauge;    // lexicographic fields (FromField)
  const float4* clover;
};

__device__ __forceinline__ void cp_async16(void* smem, const void* gmem) {
  asm volatile("cp.async.cg.shared.global [%0], [%1], 16;" ::"r"((unsigned)__cvta_generic_to_shared(smem)), "l"(gmem)
               : "memory");
}
__device__ __forceinline__ void cp_async_wait() { asm volatile("cp.async.wait_all;" ::: "memory"); }
__device__ __forceinline__ void prefetch_l2(const void* p) { asm volatile("prefetch.global.L2 [%0];" ::"l"(p)); }

// The block residual shared between neighbouring threads, six records q = 3 c + a
// (chirality, colour) per site at [q * vb + l]: (re0, re1, im0, im1) of the two
// spins as FP32 (one 128-bit load), or as bf16 (FP32 exponent range, 8-bit
// mantissa, 64 bits; each thread keeps its own residual in FP32 registers,
// only the neighbours' contributions to p = D_L r see the rounding).
template <bool BF>
__device__ __forceinline__ float4 rs_rec(const void* r_s, int vb, int l, int q) {
  if (BF) {
    const uint2 w = ((const uint2*)r_s)[q * vb + l];
    const float2 re = __bfloat1622float2(*reinterpret_cast<const __nv_bfloat162*>(&w.x));
    const float2 im = __bfloat1622float2(*reinterpret_cast<const __nv_bfloat162*>(&w.y));
    return make_float4(re.x, re.y, im.x, im.y);
  }
  return ((const float4*)r_s)[q * vb + l];
}
template <bool BF>
__device__ __forceinline__ void rs_put(void* r_s, int vb, int l, int q, float4 v) {
  if (BF) {
    const __nv_bfloat162 re = __floats2bfloat162_rn(v.x, v.y), im = __floats2bfloat162_rn(v.z, v.w);
    ((uint2*)r_s)[q * vb + l] =
        make_uint2(*reinterpret_cast<const unsigned*>(&re), *reinterpret_cast<const unsigned*>(&im));
  } else {
    ((float4*)r_s)[q * vb + l] = v;
  }
}
template <bool BF>
__device__ __forceinline__ void rs_store(void* r_s, int vb, int l, const PairSpinor& v) {
#pragma unroll
  for (int q = 0; q < 6; q++) rs_put<BF>(r_s, vb, l, q, pair_rec(v, q));
}

// o = A r at site l of the block (s of the lattice)
template <typename S>
__device__ __forceinline__ void block_clover(const BlockFields& f, int V, int s, int vb, int l, const PairSpinor& r,
                                             PairSpinor& o) {
#pragma unroll
  for (int c = 0; c < 2; c++) {
    if constexpr (std::is_same<S, __half>::value) {
      uint4 h[5];   // words 18 c .. 18 c + 17 of the site's 36
#pragma unroll
      for (int k = 0; k < 5; k++) h[k] = ((const uint4*)f.cl)[(4 * c + k) * vb + l];
      pair_clover_block(clover_pairs([&](int j) {
                          const int w = j + 2 * c;
                          const uint4 v = h[w >> 2];
                          return __half22float2(bits_h2((w & 3) == 0 ? v.x : (w & 3) == 1 ? v.y : (w & 3) == 2 ? v.z : v.w));
                        }),
                        c, r, o);
    } else if constexpr (std::is_same<S, FromField>::value) {
      float4 h[9];
#pragma unroll
      for (int k = 0; k < 9; k++) h[k] = __ldg(f.clover + (size_t)(9 * c + k) * V + s);
      pair_clover_block(
          clover_pairs([&](int j) { return (j & 1) ? p2(h[j >> 1].z, h[j >> 1].w) : p2(h[j >> 1].x, h[j >> 1].y); }), c,
          r, o);
    } else {
      float4 h[9];
#pragma unroll
      for (int k = 0; k < 9; k++) h[k] = __ldg((const float4*)f.cl + (9 * c + k) * vb + l);
      auto pr = [&](int j) { return (j & 1) ? p2(h[j >> 1].z, h[j >> 1].w) : p2(h[j >> 1].x, h[j >> 1].y); };
      CloverPairs m;
#pragma unroll
      for (int k = 0; k < 3; k++) {
        m.d[k] = pr(k);
        m.lr[k] = pr(3 + k);
        m.li[k] = pr(6 + k);
        m.e[k] = pr(9 + k);
        m.orr[k] = pr(12 + k);
        m.oi[k] = pr(15 + k);
      }
      pair_clover_block(m, c, r, o);
    }
  }
}

// p += scale * (1 + SIGN gamma_MU) U r(ln): the hop from block site ln over
// link MU of block site ll (lattice site sl), U or U^+
template <typename S, bool BF, int MU, int SIGN, bool DAG>
__device__ __forceinline__ void block_hop_pair(PairSpinor& p, const void* r_s, const BlockFields& f, int V, int vb,
                                               int ln, int ll, int sl, float scale) {
  auto rec = [&](int q) { return rs_rec<BF>(r_s, vb, ln, q); };
  if constexpr (std::is_same<S, __half>::value) {
    // entries 0-3, 4-7 and 8 as (re, im) halves
    const uint4* lk = (const uint4*)f.lk + MU * vb + ll;
    const uint4 a = lk[0], b = lk[4 * vb];
    const unsigned e8 = ((const unsigned*)((const uint4*)f.lk + 8 * vb))[MU * vb + ll];
    const unsigned w[9] = {a.x, a.y, a.z, a.w, b.x, b.y, b.z, b.w, e8};
    pair_hop<MU, SIGN, DAG>(p, rec, [&](int k) { return __half22float2(bits_h2(w[k])); }, scale);
  } else if constexpr (std::is_same<S, FromField>::value) {
    const float4* lk = f.gauge + (size_t)3 * MU * V + sl;
    const LinkRows U = link_rows(__ldg(lk), __ldg(lk + V), __ldg(lk + 2 * (size_t)V));
    pair_hop<MU, SIGN, DAG>(p, rec, [&](int k) { return U.m[k]; }, scale);
  } else {
    const float4* lk = (const float4*)f.lk + 3 * MU * vb + ll;
    const LinkRows U = link_rows(lk[0], lk[vb], lk[2 * vb]);
    pair_hop<MU, SIGN, DAG>(p, rec, [&](int k) { return U.m[k]; }, scale);
  }
}

template <typename S, bool BF, int MU>
__device__ __forceinline__ void block_hops(PairSpinor& p, const void* r_s, const BlockFields& f, const SapGeom& sg,
                                           const Geom& g, int s, int l, const int lc[4], float scale) {
  if (lc[MU] < sg.b[MU] - 1)
    block_hop_pair<S, BF, MU, -1, false>(p, r_s, f, g.V, sg.vb, l + sg.lst[MU], l, s, scale);
  if (lc[MU] > 0)
    block_hop_pair<S, BF, MU, +1, true>(p, r_s, f, g.V, sg.vb, l - sg.lst[MU], l - sg.lst[MU], s - g.stride[MU],
                                        scale);
}

// n_mr minimal-residual steps on a block from x = 0: r the site's residual (in
// r_s too, behind a barrier that this function begins with), x the increment
template <typename S, bool BF>
__device__ __forceinline__ void mr_steps(PairSpinor& r, PairSpinor& x, void* r_s, const BlockFields& f,
                                         const SapGeom& sg, const Geom& g, int s, int l, const int lc[4], float kappa,
                                         int nmr, float4* red) {
  const int vb = sg.vb;
#pragma unroll
  for (int b = 0; b < 2; b++)
#pragma unroll
    for (int a = 0; a < 3; a++) x.re[b][a] = x.im[b][a] = p2(0.f, 0.f);
  const int warp = l >> 5, lane = l & 31, nw = (vb + 31) >> 5;
  for (int step = 0; step < nmr; step++) {
    __syncthreads();
    PairSpinor p;
    block_clover<S>(f, g.V, s, vb, l, r, p);
    block_hops<S, BF, 0>(p, r_s, f, sg, g, s, l, lc, -kappa);
    block_hops<S, BF, 1>(p, r_s, f, sg, g, s, l, lc, -kappa);
    block_hops<S, BF, 2>(p, r_s, f, sg, g, s, l, lc, -kappa);
    block_hops<S, BF, 3>(p, r_s, f, sg, g, s, l, lc, -kappa);
    float2 prr = p2(0.f, 0.f), pri = p2(0.f, 0.f), ppp = p2(0.f, 0.f);
#pragma unroll
    for (int b = 0; b < 2; b++)
#pragma unroll
      for (int a = 0; a < 3; a++) {
        prr = pfma(p.re[b][a], r.re[b][a], prr);
        prr = pfma(p.im[b][a], r.im[b][a], prr);
        pri = pfma(p.re[b][a], r.im[b][a], pri);
        pri = pfma(pneg(p.im[b][a]), r.re[b][a], pri);
        ppp = pfma(p.re[b][a], p.re[b][a], ppp);
        ppp = pfma(p.im[b][a], p.im[b][a], ppp);
      }
    const float pr_re = warp_sum(prr.x + prr.y), pr_im = warp_sum(pri.x + pri.y), pp = warp_sum(ppp.x + ppp.y);
    if (lane == 0) red[warp] = make_float4(pr_re, pr_im, pp, 0.f);
    __syncthreads();
    float a_re = 0, a_im = 0, n2 = 0;
#pragma unroll 8   // (all 16 sums of a 512-site block at once would spill)
    for (int w = 0; w < nw; w++) {
      const float4 v = red[w];
      a_re += v.x;
      a_im += v.y;
      n2 += v.z;
    }
    // a quotient, not a reciprocal: far from a point source both sums can be
    // denormal, where 1 / n2 overflows but a_re / n2 stays finite
    const float al_re = n2 > 0.f ? a_re / n2 : 0.f, al_im = n2 > 0.f ? a_im / n2 : 0.f;
#pragma unroll
    for (int b = 0; b < 2; b++)
#pragma unroll
      for (int a = 0; a < 3; a++) {
        x.re[b][a] = pfma(pbc(al_re), r.re[b][a], x.re[b][a]);
        x.re[b][a] = pfma(pbc(-al_im), r.im[b][a], x.re[b][a]);
        x.im[b][a] = pfma(pbc(al_re), r.im[b][a], x.im[b][a]);
        x.im[b][a] = pfma(pbc(al_im), r.re[b][a], x.im[b][a]);
        r.re[b][a] = pfma(pbc(-al_re), p.re[b][a], r.re[b][a]);
        r.re[b][a] = pfma(pbc(al_im), p.im[b][a], r.re[b][a]);
        r.im[b][a] = pfma(pbc(-al_re), p.im[b][a], r.im[b][a]);
        r.im[b][a] = pfma(pbc(-al_im), p.re[b][a], r.im[b][a]);
      }
    // every thread read its neighbours' residual for p before the barrier
    // above, so the new residual can be stored now; the next step's first
    // barrier orders the store (and the reads of red[]) before any later use
    if (step + 1 < nmr) rs_store<BF>(r_s, vb, l, r);
  }
}

// r += scale * (hop from delta at lattice site sn over link MU of site sl)
template <int MU, int SIGN, bool DAG>
__device__ __forceinline__ void delta_hop(PairSpinor& r, const char* delta, const float4* gauge, int V, int sn, int sl,
                                          float scale) {
  const PairSpinor d = pair_load(delta, V, sn);
  const float4* lk = gauge + (size_t)3 * MU * V + sl;
  const LinkRows U = link_rows(__ldg(lk), __ldg(lk + V), __ldg(lk + 2 * (size_t)V));
  pair_hop<MU, SIGN, DAG>(r, [&](int q) { return pair_rec(d, q); }, [&](int k) { return U.m[k]; }, scale);
}

// the boundary term of one direction for this thread's own site
template <int MU>
__device__ __forceinline__ void own_gather_dir(PairSpinor& r, const SapGeom& sg, const Geom& g, const char* delta,
                                               const float4* gauge, int s, const int c[4], const int lc[4],
                                               float kappa) {
  if (lc[MU] == sg.b[MU] - 1)
    delta_hop<MU, -1, false>(r, delta, gauge, g.V, site_fwd(g, s, c, MU), s,
                             (MU == 0 && c[0] == g.L[0] - 1) ? (float)g.bc_t * kappa : kappa);
  if (lc[MU] == 0) {
    const int sb = site_bwd(g, s, c, MU);
    delta_hop<MU, +1, true>(r, delta, gauge, g.V, sb, sb, (MU == 0 && c[0] == 0) ? (float)g.bc_t * kappa : kappa);
  }
}

// One direction of the boundary gather with the block residual in shared
// memory (FP32): every site on the +MU face and every site on the -MU face
// (disjoint sets for b_MU >= 2) receives the hop from the neighbouring block's
// delta.  One thread per face site, so all lanes of the busy warps work; the
// site's residual is read, updated and written back by that thread, in the
// same arithmetic as a per-site update.  co: the block's first site.
template <int MU>
__device__ inline void smem_gather_dir(void* r_s, const SapGeom& sg, const Geom& g, const char* delta,
                                       const float4* gauge, const int co[4], int l, float kappa) {
  const int nface = sg.vb / sg.b[MU];
  if (l >= 2 * nface) return;
  const bool fwd = l < nface;
  int t = fwd ? l : l - nface;
  int lc[4], c[4];
#pragma unroll
  for (int k = 0; k < 4; k++) {
    const int nu = (k + 1) & 3;   // x, y, z, then t
    if (nu == MU) {
      lc[nu] = fwd ? sg.b[MU] - 1 : 0;
    } else {
      lc[nu] = t % sg.b[nu];
      t /= sg.b[nu];
    }
  }
  const int ls = lc[0] * sg.lst[0] + lc[1] * sg.lst[1] + lc[2] * sg.lst[2] + lc[3] * sg.lst[3];
#pragma unroll
  for (int mu = 0; mu < 4; mu++) c[mu] = co[mu] + lc[mu];
  const int s = ((c[0] * g.L[3] + c[3]) * g.L[2] + c[2]) * g.L[1] + c[1];
  PairSpinor r;
#pragma unroll
  for (int q = 0; q < 6; q++) {
    const float4 v = rs_rec<false>(r_s, sg.vb, ls, q);
    r.re[q / 3][q % 3] = p2(v.x, v.y);
    r.im[q / 3][q % 3] = p2(v.z, v.w);
  }
  if (fwd) {
    delta_hop<MU, -1, false>(r, delta, gauge, g.V, site_fwd(g, s, c, MU), s,
                             (MU == 0 && c[0] == g.L[0] - 1) ? (float)g.bc_t * kappa : kappa);
  } else {
    const int sb = site_bwd(g, s, c, MU);
    delta_hop<MU, +1, true>(r, delta, gauge, g.V, sb, sb, (MU == 0 && c[0] == 0) ? (float)g.bc_t * kappa : kappa);
  }
  rs_store<false>(r_s, sg.vb, ls, r);
}

// Any block shape: rho, psi and delta in the lexicographic layout.  img: the
// block image of S.
template <typename S, bool BF, int MAXT, int MINB>
__global__ void __launch_bounds__(MAXT, MINB)
    k_sap_sweep_pair(const char* __restrict__ rho_src, char* __restrict__ rho, char* __restrict__ psi,
                     char* __restrict__ delta, const float4* __restrict__ gauge, const float4* __restrict__ clover,
                     const unsigned char* __restrict__ img, Geom g, SapGeom sg, int colour, int gather, int psi_init,
                     int last, float kappa, int nmr, int nrhs, const int* mask) {
  extern __shared__ __align__(16) unsigned char smem_raw[];
  const int vb = sg.vb;
  void* r_s = smem_raw;
  unsigned char* lk_s = smem_raw + (size_t)vb * (BF ? 48 : 96);
  __shared__ float4 red[32];   // per warp: (p, r) re, im, (p, p)

  const int rhs = blockIdx.x % nrhs;   // RHS fastest, as in k_sap_sweep
  const int blk = blockIdx.x / nrhs;
  if (mask && !mask[rhs]) return;
  const size_t off = (size_t)rhs * FieldsF::spinor_bytes * g.V;
  rho_src += off;
  rho += off;
  psi += off;
  delta += off;

  int bc[4];
  block_of(sg, colour, blk, bc);
  const int l = threadIdx.x;
  int lc[4], c[4];
  {
    int r = l;
    lc[1] = r % sg.b[1]; r /= sg.b[1];
    lc[2] = r % sg.b[2]; r /= sg.b[2];
    lc[3] = r % sg.b[3];
    lc[0] = r / sg.b[3];
  }
#pragma unroll
  for (int mu = 0; mu < 4; mu++) c[mu] = bc[mu] * sg.b[mu] + lc[mu];
  const int s = ((c[0] * g.L[3] + c[3]) * g.L[2] + c[2]) * g.L[1] + c[1];

  BlockFields f = {nullptr, nullptr, gauge, clover};
  const size_t bidx = (size_t)colour * (gridDim.x / nrhs) + blk;
  if constexpr (std::is_same<S, __half>::value) {
    img += bidx * 288 * vb;
#pragma unroll
    for (int k = 0; k < 18; k++) cp_async16(lk_s + 16 * (k * vb + l), img + 16 * (k * vb + l));
    f.lk = lk_s;
    f.cl = lk_s + 144 * vb;
  } else if constexpr (!std::is_same<S, FromField>::value) {
    img += bidx * 480 * vb;
    f.lk = img;
    f.cl = img + 192 * vb;
    if constexpr (std::is_same<S, float>::value) {
#pragma unroll
      for (int k = 0; k < 12; k++) cp_async16(lk_s + 16 * (k * vb + l), img + 16 * (k * vb + l));
      f.lk = lk_s;
    }
  }

  PairSpinor r = pair_load(rho_src, g.V, s);
  if (BF || Stage<S>::bytes == 0) {
    // the site's own residual stays FP32 in registers
    if (gather) {
      own_gather_dir<0>(r, sg, g, delta, gauge, s, c, lc, kappa);
      own_gather_dir<1>(r, sg, g, delta, gauge, s, c, lc, kappa);
      own_gather_dir<2>(r, sg, g, delta, gauge, s, c, lc, kappa);
      own_gather_dir<3>(r, sg, g, delta, gauge, s, c, lc, kappa);
    }
    rs_store<BF>(r_s, vb, l, r);
  } else {
    rs_store<BF>(r_s, vb, l, r);
    if (gather) {
      // boundary term in four rounds (one direction each, both faces at once)
      const int co[4] = {c[0] - lc[0], c[1] - lc[1], c[2] - lc[2], c[3] - lc[3]};
      __syncthreads();
      smem_gather_dir<0>(r_s, sg, g, delta, gauge, co, l, kappa);
      __syncthreads();
      smem_gather_dir<1>(r_s, sg, g, delta, gauge, co, l, kappa);
      __syncthreads();
      smem_gather_dir<2>(r_s, sg, g, delta, gauge, co, l, kappa);
      __syncthreads();
      smem_gather_dir<3>(r_s, sg, g, delta, gauge, co, l, kappa);
      __syncthreads();
#pragma unroll
      for (int k = 0; k < 6; k++) {
        const float4 v = rs_rec<BF>(r_s, vb, l, k);
        r.re[k / 3][k % 3] = p2(v.x, v.y);
        r.im[k / 3][k % 3] = p2(v.z, v.w);
      }
    }
  }
  cp_async_wait();   // this thread's copies; the barrier of the first MR step covers the others'

  PairSpinor x;
  mr_steps<S, BF>(r, x, r_s, f, sg, g, s, l, lc, kappa, nmr, red);

  if (psi_init) {
    pair_store(psi, g.V, s, x);
  } else {
    PairSpinor y = pair_load(psi, g.V, s);
    pair_add(y, x);
    pair_store(psi, g.V, s, y);
  }
  // the last cycle's residuals and the last half-cycle's delta have no reader
  if (last < 1) pair_store(rho, g.V, s, r);
  if (last < 2) pair_store(delta, g.V, s, x);
}

// Blocks of T x 4^3 sites, T = 4 or 8 in time.  Between the first and the last
// cycle everything a CTA reads and writes is a contiguous run of its block:
//   rho_b, psi_b  [rhs][block][record q][64 T] float4, the residual and the sum
//                 of the increments (the first cycle reads the caller's
//                 lexicographic residual, the last one writes its psi);
//   faces         what the neighbours of the other colour need of delta: per
//                 block of a colour, face f = 2 mu + side (side 0: the sites at
//                 -mu, 1: at +mu) and colour a the half spinors of the face
//                 sites (64 in time, 16 T in space), [rhs][colour][block][face]
//                 [3][site] float4, projected with 1 - gamma_mu (side 0, for the
//                 block at -mu) or 1 + gamma_mu;
//   flinks        the FP32 links across a block's own faces in the same order,
//                 [block][face][link row word 3][site] float4.
// Boundary term: the face sites are 4 + 6 T / 2 tasks of a warp, at most two per
// warp (task k of warp k mod 2 T, faces in order): read the
// neighbour's half spinor and the link, multiply, leave the product in shared
// memory; after a barrier every site adds those of the faces it lies on, in the
// order t, x, y, z.  The products take the block residual's place before it is
// stored.  All loads of a CTA are issued before the first wait.
//
// Bound by the FP32 pipe: per site and MR step 1,242 multiply-adds of the operator
// and the MR update and 207 conversions of 16-bit words, which only half of the
// pipe takes.  Measured against the same sweep on lexicographic vectors in
// scalar arithmetic: 32^3x64, 12 RHS, 16-bit copies 44.4 -> 33.7 ms per
// application (5 cycles); 24^3x48, one RHS, FP32 copies 225 -> 119 us per
// half-cycle.  (Two-lane arithmetic alone, still loading lexicographic pieces, gave
// nothing: the loads were the bound.)  T = 8, one CTA of 512 threads per SM, against
// the general sweep on FromImage: 24^3x48, 12 RHS 2050 -> 1375 us per half-cycle;
// 48x24x8x16, 5 RHS 191 -> 141, one RHS 37 -> 30 (the 4^4 block: 1180, 123, 29).  A
// block on a cluster of two CTAs, hops across the middle from the other's shared
// memory: 1453, 155 and 35.
struct SapB4 {
  const char* rho_src;
  float4 *rho_b, *psi_b, *faces;
  char* psi;
  const unsigned char* img;
  const float4* flinks;
  int colour, gather, first, last, accumulate;   // last: 1 the last cycle, 2 its second half
};

template <int MU>
__device__ __forceinline__ int face_site_of(int l) {   // index of site l on a mu face (the other three coordinates)
  return MU == 0 ? (l & 63) : MU == 1 ? (l >> 2) : MU == 2 ? ((l & 3) | ((l >> 4) << 2)) : ((l & 15) | ((l >> 6) << 4));
}
// sites of a mu face and the first site of face f = 2 mu + side in the order of
// the faces; 128 + 96 T in all (at most 2 per site of the block)
template <int NT>
__host__ __device__ constexpr int face_sites(int mu) { return NT == 4 || mu == 0 ? 64 : 16 * NT; }
template <int NT>
__host__ __device__ constexpr int face_first(int f) { return NT == 4 || f < 2 ? 64 * f : 128 + (f - 2) * 16 * NT; }
template <int NT>
__host__ __device__ constexpr int all_face_sites() { return 128 + 96 * NT; }

template <int NT, int MU>
__device__ __forceinline__ void face_add(PairSpinor& r, const float4* buf, const Geom& g, int t, const int lc[4], int l,
                                         float kappa) {
  const int tf = face_site_of<MU>(l);
  constexpr int n = face_sites<NT>(MU);
  if (lc[MU] == (MU == 0 ? NT : 4) - 1) {
    const float s = (MU == 0 && t == g.L[0] - 1) ? (float)g.bc_t * kappa : kappa;
#pragma unroll
    for (int a = 0; a < 3; a++) {
      const float4 v = buf[3 * face_first<NT>(2 * MU + 1) + a * n + tf];
      pair_recon<MU, -1>(r, a, p2(v.x, v.y), p2(v.z, v.w), s);
    }
  }
  if (lc[MU] == 0) {
    const float s = (MU == 0 && t == 0) ? (float)g.bc_t * kappa : kappa;
#pragma unroll
    for (int a = 0; a < 3; a++) {
      const float4 v = buf[3 * face_first<NT>(2 * MU) + a * n + tf];
      pair_recon<MU, +1>(r, a, p2(v.x, v.y), p2(v.z, v.w), s);
    }
  }
}
// the projections of delta = x the neighbours will read
template <int NT, int MU>
__device__ __forceinline__ void face_store(float4* out, const PairSpinor& x, const int lc[4], int l) {
  const int tf = face_site_of<MU>(l);
  constexpr int n = face_sites<NT>(MU);
  float2 hr, hi;
  if (lc[MU] == 0) {
#pragma unroll
    for (int a = 0; a < 3; a++) {
      pair_project<MU, -1>(x.re[0][a], x.im[0][a], x.re[1][a], x.im[1][a], hr, hi);
      out[3 * face_first<NT>(2 * MU) + a * n + tf] = make_float4(hr.x, hr.y, hi.x, hi.y);
    }
  }
  if (lc[MU] == (MU == 0 ? NT : 4) - 1) {
#pragma unroll
    for (int a = 0; a < 3; a++) {
      pair_project<MU, +1>(x.re[0][a], x.im[0][a], x.re[1][a], x.im[1][a], hr, hi);
      out[3 * face_first<NT>(2 * MU + 1) + a * n + tf] = make_float4(hr.x, hr.y, hi.x, hi.y);
    }
  }
}
// U h (side 1) or U^+ h (side 0) of a half spinor in three records, n apart in out
__device__ __forceinline__ void face_mul(const float4 (&h)[3], const float4 (&u)[3], int side, float4* out, int n) {
  const LinkRows U = link_rows(u[0], u[1], u[2]);
  auto mul = [&](auto link) {
#pragma unroll
    for (int a = 0; a < 3; a++) {
      float2 gr = p2(0.f, 0.f), gi = p2(0.f, 0.f);
#pragma unroll
      for (int b = 0; b < 3; b++) {
        const float2 w = link(a, b), hr = p2(h[b].x, h[b].y), hi = p2(h[b].z, h[b].w);
        gr = pfma(pbc(w.x), hr, gr);
        gr = pfma(pbc(-w.y), hi, gr);
        gi = pfma(pbc(w.x), hi, gi);
        gi = pfma(pbc(w.y), hr, gi);
      }
      out[a * n] = make_float4(gr.x, gr.y, gi.x, gi.y);
    }
  };
  if (side) mul([&](int a, int b) { return U.m[3 * a + b]; });
  else mul([&](int a, int b) { return p2(U.m[3 * b + a].x, -U.m[3 * b + a].y); });
}

template <typename S, bool BF, int NT>
__global__ void __launch_bounds__(64 * NT, 8 / NT)
    k_sap_sweep_b4(SapB4 A, Geom g, SapGeom sg, float kappa, int nmr, int nrhs, const int* mask) {
  constexpr int VB = 64 * NT, NW = VB / 32, FS = all_face_sites<NT>();
  sg.b[0] = NT;
  sg.b[1] = sg.b[2] = sg.b[3] = 4;
  sg.lst[1] = 1;
  sg.lst[2] = 4;
  sg.lst[3] = 16;
  sg.lst[0] = 64;
  sg.vb = VB;
  extern __shared__ __align__(16) unsigned char smem_raw[];
  void* r_s = smem_raw;                          // boundary products, then the residual
  unsigned char* lk_s = smem_raw + 96 * VB;
  __shared__ float4 red[NW];

  launch_dependents();
  const int rhs = blockIdx.x % nrhs;   // RHS fastest, as in k_sap_sweep
  const int blk = blockIdx.x / nrhs;
  // (without a dependency_wait: the CTAs of an active right-hand side, of which every
  // application has one, wait, so the grid does not end before the previous one)
  if (mask && !mask[rhs]) return;
  const int nhalf = gridDim.x / nrhs;
  const size_t bidx = (size_t)A.colour * nhalf + blk;
  const int l = threadIdx.x;

  BlockFields f = {lk_s, lk_s + 144 * VB, nullptr, nullptr};
  {
    const unsigned char* img = A.img + bidx * (size_t)((std::is_same<S, __half>::value ? 288 : 480) * VB);
#pragma unroll
    for (int k = 0; k < (std::is_same<S, __half>::value ? 18 : 12); k++)
      cp_async16(lk_s + 16 * (k * VB + l), img + 16 * (k * VB + l));
    if (!std::is_same<S, __half>::value) f.cl = img + 192 * VB;
  }
  int bc[4];
  block_of(sg, A.colour, blk, bc);
  const int lc[4] = {l >> 6, l & 3, (l >> 2) & 3, (l >> 4) & 3};
  const int t = NT * bc[0] + lc[0];
  const int s = ((t * g.L[3] + 4 * bc[3] + lc[3]) * g.L[2] + 4 * bc[2] + lc[2]) * g.L[1] + 4 * bc[1] + lc[1];

  const size_t voff = ((size_t)rhs * 2 * nhalf + bidx) * 6 * VB + l;   // block-ordered vectors
  float4* rho_b = A.rho_b + voff;
  float4* psi_b = A.psi_b + voff;
  // above: the mask, the links and the clover term, which no half-cycle writes;
  // from here on, the previous half-cycle's results
  dependency_wait();
  if (!A.first) {
#pragma unroll
    for (int q = 0; q < 6; q++) prefetch_l2(psi_b + q * VB);
  }

  float4 rw[6];
  if (A.first) {
    load_words(A.rho_src + (size_t)rhs * FieldsF::spinor_bytes * g.V, g.V, s, rw);
  } else {
#pragma unroll
    for (int q = 0; q < 6; q++) rw[q] = rho_b[q * VB];
  }
  auto residual = [&]() {
    if (A.first) return pair_from_words(rw);
    PairSpinor o;
#pragma unroll
    for (int q = 0; q < 6; q++) {
      o.re[q / 3][q % 3] = p2(rw[q].x, rw[q].y);
      o.im[q / 3][q % 3] = p2(rw[q].z, rw[q].w);
    }
    return o;
  };
  PairSpinor r;
  if (A.gather) {
    float4* buf = (float4*)r_s;
    constexpr int NTASK = FS / 32;
    // task i of this warp: its face 2 mu + side and its 32 sites of it, from tf on
    const int w = l >> 5, side4 = (w >> 1) & 1, tf4 = ((w & 1) << 5) | (l & 31);   // (T = 4)
    auto task = [&](int i, int& mu, int& side, int& tf) {
      if (NT == 4) {
        mu = 2 * i + (w >> 2);
        side = side4;
        tf = tf4;
        return true;
      }
      const int k = i * NW + w;
      const bool time = i == 0 && k < 4;   // (2 T > 4 warps)
      const int per_face = time ? 2 : NT / 2, j = time ? k : (k - 4) % NT;
      mu = time ? 0 : 1 + (k - 4) / NT;
      side = j / per_face;
      tf = (j % per_face) * 32 + (l & 31);
      return k < NTASK;
    };
    float4 h[2][3], u[2][3];
    int mu, side, tf;
#pragma unroll
    for (int i = 0; i < 2; i++) {
      if (!task(i, mu, side, tf)) continue;
      int nbc[4] = {bc[0], bc[1], bc[2], bc[3]};
#pragma unroll
      for (int m = 0; m < 4; m++)
        if (m == mu) nbc[m] = side ? (bc[m] == sg.nb[m] - 1 ? 0 : bc[m] + 1) : (bc[m] == 0 ? sg.nb[m] - 1 : bc[m] - 1);
      const int n = face_sites<NT>(mu);
      const float4* hp = A.faces + (((size_t)rhs * 2 + 1 - A.colour) * nhalf + block_number(sg, nbc)) * (3 * FS) +
                         3 * face_first<NT>(2 * mu + 1 - side) + tf;
      const float4* up = A.flinks + bidx * (3 * FS) + 3 * face_first<NT>(2 * mu + side) + tf;
#pragma unroll
      for (int a = 0; a < 3; a++) {
        h[i][a] = hp[a * n];
        u[i][a] = __ldg(up + a * n);
      }
    }
#pragma unroll
    for (int i = 0; i < 2; i++)
      if (task(i, mu, side, tf))
        face_mul(h[i], u[i], side, buf + 3 * face_first<NT>(2 * mu + side) + tf, face_sites<NT>(mu));
    __syncthreads();
    r = residual();
    face_add<NT, 0>(r, buf, g, t, lc, l, kappa);
    face_add<NT, 1>(r, buf, g, t, lc, l, kappa);
    face_add<NT, 2>(r, buf, g, t, lc, l, kappa);
    face_add<NT, 3>(r, buf, g, t, lc, l, kappa);
    __syncthreads();   // the products are read before the residual takes their place
  } else {
    r = residual();
  }
  rs_store<BF>(r_s, VB, l, r);
  cp_async_wait();   // this thread's copies; the barrier of the first MR step covers the others'

  PairSpinor x;
  mr_steps<S, BF>(r, x, r_s, f, sg, g, s, l, lc, kappa, nmr, red);

  if (A.last < 2) {
    float4* out = A.faces + (((size_t)rhs * 2 + A.colour) * nhalf + blk) * (3 * FS);
    face_store<NT, 0>(out, x, lc, l);
    face_store<NT, 1>(out, x, lc, l);
    face_store<NT, 2>(out, x, lc, l);
    face_store<NT, 3>(out, x, lc, l);
  }
  if (A.last < 1) {
#pragma unroll
    for (int q = 0; q < 6; q++) rho_b[q * VB] = pair_rec(r, q);
  }
  if (!A.first) {
    PairSpinor y;
#pragma unroll
    for (int q = 0; q < 6; q++) {
      const float4 v = psi_b[q * VB];
      y.re[q / 3][q % 3] = p2(v.x, v.y);
      y.im[q / 3][q % 3] = p2(v.z, v.w);
    }
    pair_add(x, y);
  }
  if (A.last < 1) {
#pragma unroll
    for (int q = 0; q < 6; q++) psi_b[q * VB] = pair_rec(x, q);
  } else {
    char* psi = A.psi + (size_t)rhs * FieldsF::spinor_bytes * g.V;
    if (A.accumulate) pair_add(x, pair_load(psi, g.V, s));
    pair_store(psi, g.V, s, x);
  }
}

// ---------------------------------------------------------------------------
// The block images (built when a sweep first needs them, again after a new
// gauge field or block shape).  One thread per site, in image order.
// ---------------------------------------------------------------------------
template <typename S>
__global__ void k_block_image(const float4* __restrict__ gauge, const float4* __restrict__ clover, Geom g, SapGeom sg,
                              unsigned char* __restrict__ img) {
  const int i = blockIdx.x * blockDim.x + threadIdx.x;
  if (i >= g.V) return;
  const int bidx = i / sg.vb, l = i - bidx * sg.vb, nhalf = g.V / sg.vb / 2, vb = sg.vb;
  int bc[4], r = l;
  block_of(sg, bidx >= nhalf, bidx >= nhalf ? bidx - nhalf : bidx, bc);
  const int x = r % sg.b[1]; r /= sg.b[1];
  const int y = r % sg.b[2]; r /= sg.b[2];
  const int z = r % sg.b[3], t = r / sg.b[3];
  const int s = (((bc[0] * sg.b[0] + t) * g.L[3] + bc[3] * sg.b[3] + z) * g.L[2] + bc[2] * sg.b[2] + y) * g.L[1] +
                bc[1] * sg.b[1] + x;
  if constexpr (std::is_same<S, __half>::value) {
    img += (size_t)bidx * 288 * vb;
    uint4* o = (uint4*)img;
    unsigned* o8 = (unsigned*)(o + 8 * vb);
#pragma unroll
    for (int mu = 0; mu < 4; mu++) {
      const SU3<float> U = FieldsF::load_link(gauge, g.V, mu, s);
      unsigned h[9];
#pragma unroll
      for (int k = 0; k < 9; k++) h[k] = h2_bits(__floats2half2_rn(U.m[k / 3][k % 3].re, U.m[k / 3][k % 3].im));
      o[mu * vb + l] = make_uint4(h[0], h[1], h[2], h[3]);
      o[(4 + mu) * vb + l] = make_uint4(h[4], h[5], h[6], h[7]);
      o8[mu * vb + l] = h[8];
    }
#pragma unroll
    for (int k = 0; k < 9; k++) {
      const float4 a = clover[(size_t)(2 * k) * g.V + s], b = clover[(size_t)(2 * k + 1) * g.V + s];
      o[(9 + k) * vb + l] =
          make_uint4(h2_bits(__floats2half2_rn(a.x, a.y)), h2_bits(__floats2half2_rn(a.z, a.w)),
                     h2_bits(__floats2half2_rn(b.x, b.y)), h2_bits(__floats2half2_rn(b.z, b.w)));
    }
  } else {
    float4* o = (float4*)(img + (size_t)bidx * 480 * vb);
#pragma unroll
    for (int k = 0; k < 12; k++) o[k * vb + l] = gauge[(size_t)k * g.V + s];
#pragma unroll
    for (int c = 0; c < 2; c++) {
      float4 h[9];
#pragma unroll
      for (int k = 0; k < 9; k++) h[k] = clover[(size_t)(9 * c + k) * g.V + s];
      const CloverPairs m = clover_pairs(
          [&](int j) { return (j & 1) ? p2(h[j >> 1].z, h[j >> 1].w) : p2(h[j >> 1].x, h[j >> 1].y); });
      const float2 w[18] = {m.d[0], m.d[1], m.d[2], m.lr[0], m.lr[1], m.lr[2], m.li[0], m.li[1], m.li[2],
                            m.e[0], m.e[1], m.e[2], m.orr[0], m.orr[1], m.orr[2], m.oi[0], m.oi[1], m.oi[2]};
#pragma unroll
      for (int k = 0; k < 9; k++)
        o[(12 + 9 * c + k) * vb + l] = make_float4(w[2 * k].x, w[2 * k].y, w[2 * k + 1].x, w[2 * k + 1].y);
    }
  }
}

// flinks: one thread per (block, face, face site)
template <int NT>
__global__ void k_face_links(const float4* __restrict__ gauge, Geom g, SapGeom sg, float4* __restrict__ out) {
  constexpr int FS = all_face_sites<NT>();
  const int nblocks = g.V / (64 * NT);
  const size_t i = (size_t)blockIdx.x * blockDim.x + threadIdx.x;
  if (i >= (size_t)nblocks * FS) return;
  const int bidx = (int)(i / FS), j = (int)(i % FS), nhalf = nblocks / 2;
  const int f = j < 128 ? j >> 6 : 2 + (j - 128) / (16 * NT), tf = j - face_first<NT>(f);
  const int mu = f >> 1, side = f & 1, e = side ? (mu == 0 ? NT : 4) - 1 : 0;
  int bc[4], c[4];
  block_of(sg, bidx >= nhalf, bidx >= nhalf ? bidx - nhalf : bidx, bc);
  const int a = tf & 3, b = (tf >> 2) & 3, d = tf >> 4;
  c[0] = NT * bc[0] + (mu == 0 ? e : d);
  c[1] = 4 * bc[1] + (mu == 1 ? e : a);
  c[2] = 4 * bc[2] + (mu == 2 ? e : mu == 1 ? a : b);
  c[3] = 4 * bc[3] + (mu == 3 ? e : mu == 0 ? d : b);
  int s = ((c[0] * g.L[3] + c[3]) * g.L[2] + c[2]) * g.L[1] + c[1];
  if (!side) s = site_bwd(g, s, c, mu);
#pragma unroll
  for (int k = 0; k < 3; k++)
    out[(size_t)bidx * (3 * FS) + 3 * face_first<NT>(f) + k * face_sites<NT>(mu) + tf] =
        gauge[(size_t)(3 * mu + k) * g.V + s];
}

// blocks of k_sap_sweep_b4
bool face_blocks(const int b[4]) { return b[1] == 4 && b[2] == 4 && b[3] == 4 && (b[0] == 4 || b[0] == 8); }

// whether the FP32 sweep stages links (and clover term) of such blocks, and whether
// as 16-bit copies
bool stageable(const qcd_solver_params& P, const int b[4]) {
  const bool thin = b[0] == 1 || b[1] == 1 || b[2] == 1 || b[3] == 1;
  return b[0] * b[1] * b[2] * b[3] <= 256 && (!thin || P.sap_half == 2);
}
bool sap_uses_half(const qcd_solver_params& P, const int b[4]) { return P.sap_half && stageable(P, b); }
// whether the FP32 sweep is one in two-lane arithmetic
bool two_lane(int vb) { return vb <= 512; }

// Brings the context's block image for these blocks up to date, and with faces (blocks
// of T x 4^3, T = 4 or 8) the face links; nullptr for what there is no memory for.
qcd_status block_image(qcd_ctx* c, const SapGeom& sg, bool half, bool faces, const unsigned char** img,
                       const float4** flinks) {
  SapImage& m = half ? c->sap_img16 : c->sap_img32;
  const size_t V = c->g.V;
  bool same = m.gauge_id == c->gauge_id && m.buf.p;
  for (int mu = 0; mu < 4; mu++) same = same && m.block[mu] == sg.b[mu];
  *img = nullptr;
  *flinks = nullptr;
  if (!same) {
    m.gauge_id = 0;
    const qcd_status st = devbuf_ensure(m.buf, V * (half ? 288 : 480));
    if (st == QCD_ERR_OOM) return QCD_OK;
    QCD_TRY(st);
    ProfScope ps(c, FAM_LAYOUT, (double)V * (480 + (half ? 288 : 480)), 0.0);
    const unsigned grid = (unsigned)((V + 127) / 128);
    if (half)
      k_block_image<__half><<<grid, 128, 0, c->stream>>>((const float4*)c->gaugeF.p, (const float4*)c->cloverF.p, c->g,
                                                         sg, (unsigned char*)m.buf.p);
    else
      k_block_image<float><<<grid, 128, 0, c->stream>>>((const float4*)c->gaugeF.p, (const float4*)c->cloverF.p, c->g,
                                                        sg, (unsigned char*)m.buf.p);
    QCD_CUDA_OK(cudaGetLastError());
    for (int mu = 0; mu < 4; mu++) m.block[mu] = sg.b[mu];
    m.gauge_id = c->gauge_id;
  }
  *img = (const unsigned char*)m.buf.p;
  if (faces && (c->flinks_id != c->gauge_id || c->flinks_nt != sg.b[0])) {
    c->flinks_id = 0;
    const qcd_status st = devbuf_ensure(c->flinks, V * 96);
    if (st == QCD_ERR_OOM) return QCD_OK;
    QCD_TRY(st);
    ProfScope ps(c, FAM_LAYOUT, (double)V * 192, 0.0);
    // (at most two face sites per site of a block)
    auto kern = sg.b[0] == 4 ? k_face_links<4> : k_face_links<8>;
    kern<<<(unsigned)((2 * V + 255) / 256), 256, 0, c->stream>>>((const float4*)c->gaugeF.p, c->g, sg,
                                                                 (float4*)c->flinks.p);
    QCD_CUDA_OK(cudaGetLastError());
    c->flinks_nt = sg.b[0];
    c->flinks_id = c->gauge_id;
  }
  if (faces) *flinks = (const float4*)c->flinks.p;
  return QCD_OK;
}

template <typename F>
qcd_status launch_sweeps(qcd_ctx* c, const char* rho_src, char* rho, char* psi, char* delta, const void* gauge,
                         const void* clover, int nrhs, const int* mask, int nactive, int accumulate) {
  const qcd_solver_params& P = c->params;
  SapGeom sg;
  sg.vb = 1;
  for (int mu = 0; mu < 4; mu++) {
    sg.b[mu] = P.block[mu];
    sg.nb[mu] = c->g.L[mu] / sg.b[mu];
    sg.vb *= sg.b[mu];
    // (qcd_set_params checks this, but a lattice that the default blocks do not fit
    // starts with 2^4 ones unchecked: with an odd number of blocks in a direction
    // block_of counts past the lattice)
    if (c->g.L[mu] % sg.b[mu] != 0 || sg.nb[mu] % 2 != 0) {
      qcd_set_error("SAP: %d sites in direction %d are no even number of blocks of %d; set the block shape", c->g.L[mu],
                    mu, sg.b[mu]);
      return QCD_ERR_ARG;
    }
  }
  sg.lst[1] = 1;
  sg.lst[2] = sg.b[1];
  sg.lst[3] = sg.b[1] * sg.b[2];
  sg.lst[0] = sg.b[1] * sg.b[2] * sg.b[3];
  const int nblocks = sg.nb[0] * sg.nb[1] * sg.nb[2] * sg.nb[3];
  const dim3 grid((unsigned)(nblocks / 2) * (unsigned)nrhs);
  // Algorithmic cost of one half-cycle (the minimum each launch must move):
  // per active site and RHS, rho read and written, psi read and written (only
  // written in the first cycle), delta written, and the other colour's delta
  // read once for every site that lies on a block face (fraction f_face of
  // the sites); per active site, once per launch, its 4 links and its clover
  // term.  Flops per active site and RHS: per MR step the block operator
  // (its internal hops and the clover term) plus the MR update (24 complex
  // multiply-adds), and one hop per face direction for the gather.
  double face = 0, inner = 1;
  for (int mu = 0; mu < 4; mu++) {
    face += 2.0 / sg.b[mu];
    inner *= 1.0 - 2.0 / sg.b[mu];
  }
  const double f_face = 1.0 - (inner > 0 ? inner : 0.0);
  const double sb = (double)F::spinor_bytes, lb = (double)F::link_bytes, cb = (double)F::clover_bytes;
  const double half = c->g.V / 2.0;
  const double flops_gather = 165.0 * face;
  const double flops_site = P.nmr * (1320.0 * (1.0 - face / 8.0) + 504.0 + 192.0) + flops_gather;
  const int fam = sizeof(typename F::R) == 8 ? FAM_SAP_D : FAM_SAP_F;
  constexpr bool f32 = sizeof(typename F::R) == 4;
  const bool b4 = face_blocks(sg.b) && (f32 || sg.b[0] == 4);
  // FP32 blocks of at most 256 sites are staged in shared memory, unless an extent is
  // 1: the two faces of such a direction are the same sites, which smem_gather_dir does
  // not serve (the bf16 residual's and the unstaged sweeps gather per site; a second
  // pass of smem_gather_dir cost the other shapes 1 to 5 %).  Without memory for the
  // FP32 image (FromField), or for the face links or block-ordered vectors of a block of
  // 4 or 8 x 4^3, the sweep runs on the lexicographic fields or vectors
  const bool h16 = f32 && sap_uses_half(P, sg.b);
  const unsigned char* img = nullptr;
  SapB4 A = {};
  bool use_b4 = false;
  const bool pair = f32 && two_lane(sg.vb);
  if (pair) {
    QCD_TRY(block_image(c, sg, h16, b4, &img, &A.flinks));
    if (h16 && !img) return QCD_ERR_OOM;
    if (b4 && img && A.flinks) {
      // psi_b, and rho_b where the caller's residual is its own working copy
      const size_t vec = (size_t)c->g.V * 96 * nrhs;
      const bool own = rho_src != rho;
      const qcd_status st = devbuf_ensure(c->sap_vec, own ? vec : 2 * vec);
      if (st != QCD_OK && st != QCD_ERR_OOM) return st;
      use_b4 = st == QCD_OK;
      A.rho_src = rho_src;
      A.psi_b = (float4*)c->sap_vec.p;
      A.rho_b = own ? (float4*)rho : A.psi_b + vec / 16;
      A.faces = (float4*)delta;
      A.psi = psi;
      A.img = img;
      A.accumulate = accumulate;
    }
  }
  const bool staged = f32 && stageable(P, sg.b) && img;
  // the register budget per thread follows from the block volume
  auto kernD = k_sap_sweep<F, 1024, 1>;
  if constexpr (!f32) kernD = sg.vb <= 256 ? k_sap_sweep<F, 256, 1> : sg.vb <= 512 ? k_sap_sweep<F, 512, 1> : kernD;
  auto kernB = sg.b[0] == 8    ? k_sap_sweep_b4<float, false, 8>
               : !h16            ? k_sap_sweep_b4<float, false, 4>
               : P.sap_half == 2 ? k_sap_sweep_b4<__half, true, 4>
                                 : k_sap_sweep_b4<__half, false, 4>;
  auto kernF = staged ? (!h16              ? k_sap_sweep_pair<float, false, 256, 2>
                         : P.sap_half == 2 ? k_sap_sweep_pair<__half, true, 256, 2>
                                           : k_sap_sweep_pair<__half, false, 256, 2>)
               : img  ? k_sap_sweep_pair<FromImage, false, 512, 1>
                      : k_sap_sweep_pair<FromField, false, 512, 1>;
  const size_t smem = (size_t)sg.vb * (!f32                 ? 192
                                       : !staged && !use_b4 ? 96
                                       : !h16               ? 96 + Stage<float>::bytes
                                              : (P.sap_half == 2 && !use_b4 ? 48 : 96) + Stage<__half>::bytes);
  // links and clover term read per active site and launch: their FP16 copies
  // (36 B per link, 144 B clover) for the 16-bit staged blocks, else FP32
  const double gcb = h16 ? 4 * 36.0 + 144.0 : 4 * lb + cb;
  // the largest block that the chosen kernel serves
  const int most = use_b4 ? sg.vb : sg.vb <= 256 && (staged || !f32) ? 256 : sg.vb <= 512 ? 512 : 1024;
  QCD_CUDA_OK(use_b4 ? allow_smem(kernB, smem)
              : pair ? allow_smem(kernF, smem / sg.vb * most)
                     : allow_smem(kernD, smem / sg.vb * most));
  const size_t smem_d4 = (size_t)2 * 12 * BlockD::N * sizeof(double2);
  auto kernC = d4_three(2 * grid.x) ? k_sap_sweep_d4<3> : k_sap_sweep_d4<2>;
  if (!f32 && b4)
    QCD_CUDA_OK(allow_smem(kernC, smem_d4));
  auto issue = [&]() -> qcd_status {
    for (int cy = 0; cy < P.ncy; cy++)
      for (int col = 0; col < 2; col++) {
        const int first = cy == 0 && !accumulate;
        const int gather = !(cy == 0 && col == 0);   // no boundary term before the first half-cycle
        const double bytes_rhs = sb * (2 + (first ? 1 : 2) + 1 + (gather ? f_face : 0.0));
        const int last = cy < P.ncy - 1 ? 0 : 1 + col;   // 1: the last cycle, 2: its second half
        ProfScope ps(c, fam, half * (nactive * bytes_rhs + gcb),
                     half * nactive * (flops_site - (gather ? 0.0 : flops_gather)));
        const char* rin = cy == 0 ? rho_src : rho;   // the first cycle reads the caller's residual
        if (pair) {
          if (use_b4) {
            A.colour = col;
            A.gather = gather;
            A.first = cy == 0;
            A.last = last;
            // Every half-cycle but the first overlaps the previous one's last wave with
            // its launch and the staging of its fields.  Measured per half-cycle, FP16
            // fields, one RHS: 24^3x48 108.8 -> 105.2 us, 16^3x32 25.2 -> 24.1; 12 RHS:
            // 1095 -> 1093 and 229.5 -> 228.5.
            QCD_CUDA_OK(launch_after(c->stream, gather, grid, sg.vb, smem, kernB, A, c->g, sg, (float)c->kappa, P.nmr,
                                     nrhs, mask));
          } else {
            kernF<<<grid, sg.vb, smem, c->stream>>>(rin, rho, psi, delta, (const float4*)gauge, (const float4*)clover,
                                                    img, c->g, sg, col, gather, first, last, (float)c->kappa, P.nmr,
                                                    nrhs, mask);
          }
        }
        else if (b4) {
          kernC<<<2 * grid.x, BlockD::N, smem_d4, c->stream>>>(rin, rho, psi, delta, gauge, clover, c->g, sg,
                                                                        col, gather, first, last, c->kappa, P.nmr,
                                                                        nrhs, mask);
        } else
          kernD<<<grid, sg.vb, smem, c->stream>>>(rin, rho, psi, delta, gauge, clover, c->g, sg, col, gather, first,
                                                  (typename F::R)c->kappa, P.nmr, nrhs, mask);
        QCD_CUDA_OK(cudaGetLastError());
      }
    return QCD_OK;
  };
  if (!P.graphs || c->stream == nullptr) return issue();
  // replay the whole application from a cached CUDA graph
  SapGraph key;
  key.rho_src = rho_src;
  key.rho = rho; key.psi = psi; key.delta = delta; key.gauge = gauge; key.clover = clover; key.mask = mask;
  key.img = img; key.flinks = A.flinks; key.vec = use_b4 ? c->sap_vec.p : nullptr;
  key.nrhs = nrhs; key.ncy = P.ncy; key.nmr = P.nmr; key.accumulate = accumulate; key.half = P.sap_half;
  key.prec = (int)sizeof(typename F::R);
  key.bc_t = c->g.bc_t;   // in the captured launches' Geom; a new field may change it
  for (int mu = 0; mu < 4; mu++) key.block[mu] = P.block[mu];
  key.kappa = c->kappa;
  cudaGraphExec_t exec = nullptr;
  for (auto& gph : c->sap_graphs)
    if (gph.rho_src == key.rho_src && gph.rho == key.rho && gph.psi == key.psi && gph.delta == key.delta && gph.gauge == key.gauge &&
        gph.clover == key.clover && gph.mask == key.mask && gph.img == key.img && gph.flinks == key.flinks &&
        gph.vec == key.vec && gph.nrhs == key.nrhs && gph.ncy == key.ncy &&
        gph.nmr == key.nmr && gph.accumulate == key.accumulate && gph.half == key.half && gph.prec == key.prec &&
        gph.bc_t == key.bc_t && gph.kappa == key.kappa && memcmp(gph.block, key.block, sizeof(key.block)) == 0) {
      exec = gph.exec;
      break;
    }
  if (!exec) {
    cudaGraph_t graph = nullptr;
    QCD_CUDA_OK(cudaStreamBeginCapture(c->stream, cudaStreamCaptureModeThreadLocal));
    c->prof_suspend++;
    qcd_status st = issue();
    c->prof_suspend--;
    cudaError_t e = cudaStreamEndCapture(c->stream, &graph);
    if (st != QCD_OK) return st;
    QCD_CUDA_OK(e);
    e = cudaGraphInstantiate(&exec, graph, 0);
    cudaGraphDestroy(graph);
    QCD_CUDA_OK(e);
    if (c->sap_graphs.size() >= 64) {
      cudaGraphExecDestroy(c->sap_graphs.front().exec);
      c->sap_graphs.erase(c->sap_graphs.begin());
    }
    key.exec = exec;
    c->sap_graphs.push_back(key);
  }
  double bytes = 0, flops = 0;
  for (int cy = 0; cy < P.ncy; cy++)
    for (int col = 0; col < 2; col++) {
      const int first = cy == 0 && !accumulate;
      const int gather = !(cy == 0 && col == 0);
      bytes += half * (nactive * sb * (2 + (first ? 1 : 2) + 1 + (gather ? f_face : 0.0)) + gcb);
      flops += half * nactive * (flops_site - (gather ? 0.0 : flops_gather));
    }
  ProfScope ps(c, fam, bytes, flops, 2 * P.ncy);
  QCD_CUDA_OK(cudaGraphLaunch(exec, c->stream));
  return QCD_OK;
}

}  // namespace

// Allocates what the SAP of the caller's parameters keeps per gauge field, so that its
// first application does not stop for it (60 us an allocation: a first application on
// 16x8x8x16, two RHS, 626 -> 543 us), and gives back what was taken for earlier ones
// and never used.  block_image tries again where there is no memory now.  (Not called
// before the caller has set parameters: a context that never applies the SAP keeps none
// of this.)
void sap_reserve(qcd_ctx* c) {
  const int* b = c->params.block;
  const bool f32 = c->params.precision == QCD_PREC_F32 && two_lane(b[0] * b[1] * b[2] * b[3]);
  const bool h16 = f32 && sap_uses_half(c->params, b);
  const bool faces = f32 && face_blocks(b);
  if ((!f32 || h16) && c->sap_img32.gauge_id == 0) devbuf_free(c->sap_img32.buf);
  if (!h16 && c->sap_img16.gauge_id == 0) devbuf_free(c->sap_img16.buf);
  if (!faces && c->flinks_id == 0) devbuf_free(c->flinks);
  if (f32) devbuf_ensure(h16 ? c->sap_img16.buf : c->sap_img32.buf, (size_t)c->g.V * (h16 ? 288 : 480));
  if (faces) devbuf_ensure(c->flinks, (size_t)c->g.V * 96);
}

qcd_status sap_apply(qcd_ctx* c, void* rho, void* psi, void* delta, int prec, int nrhs, const int* mask,
                     int nactive, int accumulate, const void* rho_src) {
  const char* src = rho_src ? (const char*)rho_src : (const char*)rho;
  if (prec == QCD_PREC_F64)
    return launch_sweeps<FieldsD>(c, src, (char*)rho, (char*)psi, (char*)delta, c->gaugeD.p, c->cloverD.p, nrhs,
                                  mask, nactive, accumulate);
  return launch_sweeps<FieldsF>(c, src, (char*)rho, (char*)psi, (char*)delta, c->gaugeF.p, c->cloverF.p, nrhs, mask,
                                nactive, accumulate);
}
