// The Wilson-clover operator D (Sec. 2.2, the Dirac equation D psi = eta):
//   D psi(x) = A(x) psi(x) - kappa sum_mu [(1 - g_mu) U_mu(x) psi(x+mu) + (1 + g_mu) U_mu(x-mu)^+ psi(x-mu)]
// with A(x) = 1 + clover term; D^+ exchanges the two spin projectors.
//
// One thread per site and right-hand side (FP32: per site and two of them).  The
// CTAs of all right-hand sides that cover the same run of sites are adjacent in
// launch order, so the gauge and clover words of those sites are reused from L2.
// Every (1 -+ g_mu) projection halves the spinor before the SU(3) multiply.
//
// Traversal order with several RHS: a run of DSLASH_TPB sites is part of one
// (t, z) plane; runs are visited slab by slab, a slab being zw consecutive z
// planes, and within a slab time-slice by time-slice.  A site's neighbours in
// t are then zw planes (zw X Y sites) away in launch order instead of a whole
// time-slice: with 12 RHS a time-slice of 32^3 sites moves ~75 MB, more than
// L2 keeps, while a slab of 8 planes moves ~20 MB, so the t-neighbours'
// spinors are still in L2 when they are read.
#include <type_traits>

#include "spin_pair.cuh"

namespace {

constexpr int DSLASH_TPB = 128;   // sites of a run, threads of a CTA

struct Canonical {};   // output [rhs][site][12] FP64, the caller's layout

// cp: runs of DSLASH_TPB sites per (t, z) plane (0: plain lexicographic
// order); zw: z planes per slab
struct RunOrder {
  int cp, zw;
};

// first site of run q
__device__ inline int run_base(const Geom& g, RunOrder o, int q) {
  if (o.cp == 0) return q * DSLASH_TPB;
  const int per_t = o.zw * o.cp;
  const int per_slab = g.L[0] * per_t;
  const int zb = q / per_slab;
  int r = q - zb * per_slab;
  const int t = r / per_t;
  r -= t * per_t;
  const int z = zb * o.zw + r / o.cp;
  const int run = r % o.cp;
  return (t * g.L[3] + z) * g.L[2] * g.L[1] + run * DSLASH_TPB;
}

// ---------------------------------------------------------------------------
// FP64
// ---------------------------------------------------------------------------
template <int MU, int DAGGER>
__device__ inline void hop_dir(Spinor<double>& acc, const void* in, const void* gauge, const Geom& g, int s,
                               const int c[4], double scale) {
  using F = FieldsD;
  constexpr int SF = DAGGER ? +1 : -1;   // projector sign for the forward hop
  constexpr int SB = -SF;                // and for the backward hop
  const int V = g.V;
  // acc += scale * (1 SF g_mu) U_mu(x) psi(x + mu)
  {
    int sf = site_fwd(g, s, c, MU);
    double sign = (MU == 0 && c[0] == g.L[0] - 1) ? g.bc_t * scale : scale;
    HalfSpinor<double> h = project<MU, SF>(F::load_spinor(in, V, sf));
    h = su3_mul(F::load_link(gauge, V, MU, s), h);
    accum_recon<MU, SF>(acc, h, sign);
  }
  // acc += scale * (1 SB g_mu) U_mu(x - mu)^+ psi(x - mu)
  {
    int sb = site_bwd(g, s, c, MU);
    double sign = (MU == 0 && c[0] == 0) ? g.bc_t * scale : scale;
    HalfSpinor<double> h = project<MU, SB>(F::load_spinor(in, V, sb));
    h = su3_dag_mul(F::load_link(gauge, V, MU, sb), h);
    accum_recon<MU, SB>(acc, h, sign);
  }
}

// The canonical output of a CTA is one contiguous run: the ns sites of sm
// ([component][ld], FP32 or FP64) written with consecutive threads on consecutive
// words.  An export of its own read the result back: operator and export, FP32,
// 32^3x64, 12 RHS 3.02 -> 2.43 ms; FP64, 24^3x48, 4 RHS 5.33 -> 5.11 ms, 8^3x16, one
// RHS one launch of two less.
template <typename T>
__device__ __forceinline__ void store_canonical(double2* p, const T* sm, int ld, int ns) {
  __syncthreads();
  for (int i = threadIdx.x; i < 12 * ns; i += blockDim.x) {
    const T v = sm[(i % 12) * ld + i / 12];
    __stcs(p + i, make_double2(v.x, v.y));   // (read by the caller: not to displace the spinors in L2)
  }
}

template <typename O, int DAGGER>
__global__ void __launch_bounds__(DSLASH_TPB, 3) k_dslash(const char* __restrict__ in, char* __restrict__ out,
                                                       const void* __restrict__ gauge, const void* __restrict__ clover,
                                                       Geom g, double kappa, int nrhs, const int* mask, RunOrder ord) {
  constexpr bool canon = std::is_same<O, Canonical>::value;
  __shared__ double2 sm[canon ? 12 * (DSLASH_TPB + 1) : 1];
  const int rhs = blockIdx.x % nrhs;
  const int base = run_base(g, ord, blockIdx.x / nrhs), s = base + threadIdx.x;
  if (!canon && s >= g.V) return;
  if (mask && !mask[rhs]) return;
  const size_t off = (size_t)rhs * FieldsD::spinor_bytes * g.V;
  if (s < g.V) {
    const void* src = in + off;
    int c[4];
    site_coords(g, s, c);
    Spinor<double> o = clover_apply<FieldsD>(clover, g.V, s, FieldsD::load_spinor(src, g.V, s));
    hop_dir<0, DAGGER>(o, src, gauge, g, s, c, -kappa);
    hop_dir<1, DAGGER>(o, src, gauge, g, s, c, -kappa);
    hop_dir<2, DAGGER>(o, src, gauge, g, s, c, -kappa);
    hop_dir<3, DAGGER>(o, src, gauge, g, s, c, -kappa);
    if constexpr (canon) {
#pragma unroll
      for (int k = 0; k < 12; k++) sm[k * (DSLASH_TPB + 1) + threadIdx.x] = make_double2(o.c[k].re, o.c[k].im);
    } else {
      FieldsD::store_spinor(out + off, g.V, s, o);
    }
  }
  if constexpr (canon)
    store_canonical((double2*)(out + off) + (size_t)12 * base, sm, DSLASH_TPB + 1, min(DSLASH_TPB, g.V - base));
}

// FP64 on small lattices: a site's operator split over two warps.  The FP64 unit of
// an SM quarter takes 64 cycles for an instruction of a warp, however few lanes are
// active, so a warp's 1,130 operations cost 35 us however many units idle beside it.
// Two warps per 32 sites take two directions and one chirality of the clover term
// each and exchange half of their sums through shared memory.
constexpr int SPLIT_SITES = 64;   // sites per CTA of 128 threads
// Lattices whose half warps' work still finds a free SM quarter each (608 of them).
// Measured, one RHS: 8^3x16 44.7 -> 26.2 us; at twice the volume 44.7 -> 45.1 (12 RHS:
// 229 -> 217 and 415 -> 409), at four times 79.9 -> 83.0.
constexpr int SPLIT_MAX_V = 4 * 152 * 16;

template <typename O, int DAGGER>
__global__ void __launch_bounds__(2 * SPLIT_SITES) k_dslash_split(const char* __restrict__ in, char* __restrict__ out,
                                                                  const void* __restrict__ gauge,
                                                                  const void* __restrict__ clover, Geom g, double kappa,
                                                                  int nrhs, const int* mask) {
  constexpr bool canon = std::is_same<O, Canonical>::value;
  __shared__ double2 sh[2][6][SPLIT_SITES + 1];
  const int rhs = blockIdx.x % nrhs;
  const int i = threadIdx.x % SPLIT_SITES, part = threadIdx.x / SPLIT_SITES;
  const int s = (int)(blockIdx.x / nrhs) * SPLIT_SITES + i;
  if (mask && !mask[rhs]) return;
  const size_t off = (size_t)rhs * FieldsD::spinor_bytes * g.V;
  const void* src = in + off;
  Spinor<double> o;
#pragma unroll
  for (int k = 0; k < 12; k++) o.c[k] = cmk(0.0, 0.0);
  if (s < g.V) {
    int c[4];
    site_coords(g, s, c);
    double cl[36];
    FieldsD::load_clover_block(clover, g.V, s, part, cl);
    Cplx<double> v[6], w[6];
    const double2* p = (const double2*)src + (size_t)6 * part * g.V + s;
#pragma unroll
    for (int k = 0; k < 6; k++) {
      const double2 x = __ldg(p + (size_t)k * g.V);
      v[k] = cmk(x.x, x.y);
    }
    clover_block_apply(cl, 0, v, w);
    if (part == 0) {
#pragma unroll
      for (int k = 0; k < 6; k++) o.c[k] = w[k];
      hop_dir<0, DAGGER>(o, src, gauge, g, s, c, -kappa);
      hop_dir<1, DAGGER>(o, src, gauge, g, s, c, -kappa);
    } else {
#pragma unroll
      for (int k = 0; k < 6; k++) o.c[6 + k] = w[k];
      hop_dir<2, DAGGER>(o, src, gauge, g, s, c, -kappa);
      hop_dir<3, DAGGER>(o, src, gauge, g, s, c, -kappa);
    }
  }
  // part 0 finishes components 0-5, part 1 components 6-11
#pragma unroll
  for (int k = 0; k < 6; k++) {
    const Cplx<double> v = part == 0 ? o.c[6 + k] : o.c[k];
    sh[part][k][i] = make_double2(v.re, v.im);
  }
  __syncthreads();
  Cplx<double> w[6];
#pragma unroll
  for (int k = 0; k < 6; k++) {
    const double2 v = sh[1 - part][k][i];
    const Cplx<double> u = part == 0 ? o.c[k] : o.c[6 + k];
    w[k] = cmk(u.re + v.x, u.im + v.y);
  }
  if constexpr (canon) {
    __syncthreads();
#pragma unroll
    for (int k = 0; k < 6; k++) sh[part][k][i] = make_double2(w[k].re, w[k].im);
    store_canonical((double2*)(out + off) + (size_t)12 * (s - i), &sh[0][0][0], SPLIT_SITES + 1,
                    min(SPLIT_SITES, g.V - (s - i)));
  } else if (s < g.V) {
    double2* q = (double2*)(out + off) + (size_t)6 * part * g.V + s;
#pragma unroll
    for (int k = 0; k < 6; k++) q[(size_t)k * g.V] = make_double2(w[k].re, w[k].im);
  }
}

// ---------------------------------------------------------------------------
// FP32, in two-lane arithmetic with the real and imaginary part of a component in
// the lanes, as the words of the fields hold them.  u v = u.re v + i (u.im v): the
// products with u.re and with u.im are summed apart, broadcasts of u cost nothing,
// and one multiply-add by (-1, 1) with exchanged lanes joins the sums.  A thread
// applies the operator to NR right-hand sides of a site with one read of the links
// and the clover term.
//
// Bound by the latency of L2: a site and right-hand side reads its four neighbours
// in z and t, itself and its share of the links from L2, about 900 bytes (1,200 with
// NR = 1), and the 16 to 20 warps that the registers leave an SM hide no more (16^3x32, 12
// RHS: a warp waits 4.3 of its 8 cycles per instruction for loads, L2 is at 45 % of its
// rate, the FMA pipe at 59 %, DRAM at 36 %).  24^3x48
// against scalar arithmetic and one right-hand side per thread: 12 RHS 634 -> 602 us,
// one RHS 84 -> 80.  (12 RHS, caller's layout: NR = 2 on 4 CTAs per SM 814 us, on 3 1002,
// on 5 891; NR = 1 on 5 836, on 8 905.)
// ---------------------------------------------------------------------------
// y +- i x
__device__ __forceinline__ float2 add_ix(float2 y, float2 x) { return pfma(psw(x), p2(-1.f, 1.f), y); }
__device__ __forceinline__ float2 sub_ix(float2 y, float2 x) { return pfma(psw(x), p2(1.f, -1.f), y); }
__device__ __forceinline__ float2 add_c(float2 y, float2 x) { return __fadd2_rn(y, x); }
__device__ __forceinline__ float2 sub_c(float2 y, float2 x) { return pfma(x, pbc(-1.f), y); }

// h = the two upper spins of (1 + SIGN gamma_mu) w (component 3 spin + colour)
template <int MU, int SIGN>
__device__ __forceinline__ void c_project(const float2 (&w)[12], float2 (&h)[6]) {
#pragma unroll
  for (int a = 0; a < 3; a++) {
    const float2 u0 = w[a], u1 = w[3 + a], d0 = w[6 + a], d1 = w[9 + a];
    if (MU == 0) { h[a] = SIGN < 0 ? add_c(u0, d0) : sub_c(u0, d0); h[3 + a] = SIGN < 0 ? add_c(u1, d1) : sub_c(u1, d1); }
    if (MU == 1) { h[a] = SIGN < 0 ? add_ix(u0, d1) : sub_ix(u0, d1); h[3 + a] = SIGN < 0 ? add_ix(u1, d0) : sub_ix(u1, d0); }
    if (MU == 2) { h[a] = SIGN < 0 ? add_c(u0, d1) : sub_c(u0, d1); h[3 + a] = SIGN < 0 ? sub_c(u1, d0) : add_c(u1, d0); }
    if (MU == 3) { h[a] = SIGN < 0 ? add_ix(u0, d0) : sub_ix(u0, d0); h[3 + a] = SIGN < 0 ? sub_ix(u1, d1) : add_ix(u1, d1); }
  }
}
// o += all four spins of (1 + SIGN gamma_mu) from the upper two, colour a
template <int MU, int SIGN>
__device__ __forceinline__ void c_recon(float2 (&o)[12], int a, float2 h0, float2 h1) {
  o[a] = add_c(o[a], h0);
  o[3 + a] = add_c(o[3 + a], h1);
  float2 &d0 = o[6 + a], &d1 = o[9 + a];
  if (MU == 0) { d0 = SIGN < 0 ? add_c(d0, h0) : sub_c(d0, h0); d1 = SIGN < 0 ? add_c(d1, h1) : sub_c(d1, h1); }
  if (MU == 1) { d0 = SIGN < 0 ? sub_ix(d0, h1) : add_ix(d0, h1); d1 = SIGN < 0 ? sub_ix(d1, h0) : add_ix(d1, h0); }
  if (MU == 2) { d0 = SIGN < 0 ? sub_c(d0, h1) : add_c(d0, h1); d1 = SIGN < 0 ? add_c(d1, h0) : sub_c(d1, h0); }
  if (MU == 3) { d0 = SIGN < 0 ? sub_ix(d0, h0) : add_ix(d0, h0); d1 = SIGN < 0 ? add_ix(d1, h1) : sub_ix(d1, h1); }
}
__device__ __forceinline__ void c_load(const float4* p, size_t V, float2 (&w)[12]) {
#pragma unroll
  for (int k = 0; k < 6; k++) {
    const float4 v = __ldg(p + k * V);
    w[2 * k] = p2(v.x, v.y);
    w[2 * k + 1] = p2(v.z, v.w);
  }
}

// acc += bc (1 + SIGN gamma_mu) U psi of site sn (DAG: U^+ psi), over link MU of site sl;
// src: the right-hand sides' spinors
template <int MU, int SIGN, bool DAG, int NR>
__device__ __forceinline__ void c_hop(float2 (&acc)[NR][12], const float4* const (&src)[NR], const float4* gauge,
                                      size_t V, int sn, int sl, float bc) {
  const float4* lk = gauge + 3 * MU * V + sl;
  LinkRows U = link_rows(__ldg(lk), __ldg(lk + V), __ldg(lk + 2 * V));
  if (MU == 0) {
#pragma unroll
    for (int k = 0; k < 9; k++) U.m[k] = pmul(U.m[k], pbc(bc));
  }
#pragma unroll
  for (int r = 0; r < NR; r++) {
    float2 w[12], h[6];
    c_load(src[r] + sn, V, w);
    c_project<MU, SIGN>(w, h);
#pragma unroll
    for (int a = 0; a < 3; a++) {
      float2 g[2];
#pragma unroll
      for (int sp = 0; sp < 2; sp++) {
        float2 x, y;   // sums of the products with the real and the imaginary parts
#pragma unroll
        for (int b = 0; b < 3; b++) {
          const float2 u = DAG ? U.m[3 * b + a] : U.m[3 * a + b];
          x = b == 0 ? pmul(pbc(u.x), h[3 * sp]) : pfma(pbc(u.x), h[3 * sp + b], x);
          y = b == 0 ? pmul(pbc(u.y), h[3 * sp]) : pfma(pbc(u.y), h[3 * sp + b], y);
        }
        g[sp] = DAG ? sub_ix(x, y) : add_ix(x, y);
      }
      c_recon<MU, SIGN>(acc[r], a, g[0], g[1]);
    }
  }
}

template <int MU, int DAGGER, int NR>
__device__ __forceinline__ void c_hops(float2 (&acc)[NR][12], const float4* const (&src)[NR], const float4* gauge,
                                       const Geom& g, int s, const int c[4]) {
  constexpr int SF = DAGGER ? +1 : -1;
  c_hop<MU, SF, false>(acc, src, gauge, g.V, site_fwd(g, s, c, MU), s,
                       MU == 0 && c[0] == g.L[0] - 1 ? (float)g.bc_t : 1.f);
  const int sb = site_bwd(g, s, c, MU);
  c_hop<MU, -SF, true>(acc, src, gauge, g.V, sb, sb, MU == 0 && c[0] == 0 ? (float)g.bc_t : 1.f);
}

// o = A psi - kappa acc for NR right-hand sides of a site, in place of acc
template <int NR>
__device__ __forceinline__ void c_finish(float2 (&acc)[NR][12], const float4* const (&src)[NR], const float4* clover,
                                         size_t V, int s, float kappa) {
#pragma unroll
  for (int ch = 0; ch < 2; ch++) {
    float2 m[18];   // the block's 36 reals: 6 of the diagonal, then entry (i, j) at 3 + i (i - 1) / 2 + j
#pragma unroll
    for (int k = 0; k < 9; k++) {
      const float4 v = __ldg(clover + (9 * ch + k) * V + s);
      m[2 * k] = p2(v.x, v.y);
      m[2 * k + 1] = p2(v.z, v.w);
    }
#pragma unroll
    for (int r = 0; r < NR; r++) {
      float2 v[6], x[6], y[6];
#pragma unroll
      for (int k = 0; k < 3; k++) {
        const float4 q = __ldg(src[r] + (3 * ch + k) * V + s);
        v[2 * k] = p2(q.x, q.y);
        v[2 * k + 1] = p2(q.z, q.w);
      }
#pragma unroll
      for (int i = 0; i < 6; i++) {
        x[i] = pmul(pbc((i & 1) ? m[i >> 1].y : m[i >> 1].x), v[i]);
        y[i] = p2(0.f, 0.f);
      }
#pragma unroll
      for (int i = 1; i < 6; i++)
#pragma unroll
        for (int j = 0; j < i; j++) {
          const float2 e = m[3 + i * (i - 1) / 2 + j];
          x[i] = pfma(pbc(e.x), v[j], x[i]);
          y[i] = pfma(pbc(e.y), v[j], y[i]);
          x[j] = pfma(pbc(e.x), v[i], x[j]);
          y[j] = pfma(pbc(-e.y), v[i], y[j]);
        }
#pragma unroll
      for (int i = 0; i < 6; i++)
        acc[r][6 * ch + i] = add_ix(pfma(pbc(-kappa), acc[r][6 * ch + i], x[i]), y[i]);
    }
  }
}

template <typename O, int DAGGER, int NR>
__device__ __forceinline__ void dslash_f32_site(const char* in, char* out, const float4* gauge, const float4* clover,
                                                const Geom& g, float kappa, int base, const int (&rhs)[NR],
                                                float2* sm) {
  constexpr bool canon = std::is_same<O, Canonical>::value;
  const int s = base + threadIdx.x;
  const size_t V = g.V;
  float2 acc[NR][12];
  if (s < g.V) {
    const float4* src[NR];
#pragma unroll
    for (int r = 0; r < NR; r++) {
      src[r] = (const float4*)in + 6 * V * rhs[r];
#pragma unroll
      for (int k = 0; k < 12; k++) acc[r][k] = p2(0.f, 0.f);
    }
    int c[4];
    site_coords(g, s, c);
    c_hops<0, DAGGER>(acc, src, gauge, g, s, c);
    c_hops<1, DAGGER>(acc, src, gauge, g, s, c);
    c_hops<2, DAGGER>(acc, src, gauge, g, s, c);
    c_hops<3, DAGGER>(acc, src, gauge, g, s, c);
    c_finish(acc, src, clover, V, s, kappa);
    if constexpr (!canon) {
#pragma unroll
      for (int r = 0; r < NR; r++) {
        Spinor<float> o;
#pragma unroll
        for (int k = 0; k < 12; k++) o.c[k] = cmk(acc[r][k].x, acc[r][k].y);
        O::store_spinor(out + (size_t)rhs[r] * O::spinor_bytes * V, g.V, s, o);
      }
    }
  }
  if constexpr (canon) {
#pragma unroll
    for (int r = 0; r < NR; r++) {
      if (r > 0) __syncthreads();   // the previous one's words are written
#pragma unroll
      for (int k = 0; k < 12; k++) sm[k * (DSLASH_TPB + 1) + threadIdx.x] = acc[r][k];
      store_canonical((double2*)out + 12 * (V * rhs[r] + base), sm, DSLASH_TPB + 1, min(DSLASH_TPB, g.V - base));
    }
  }
}

// NR right-hand sides per thread; where fewer than NR are left or active, one each
template <typename O, int DAGGER, int NR>
__global__ void __launch_bounds__(DSLASH_TPB, NR == 2 ? 4 : 5) k_dslash_f32(const char* __restrict__ in, char* __restrict__ out,
                                                           const float4* __restrict__ gauge,
                                                           const float4* __restrict__ clover, Geom g, float kappa,
                                                           int nrhs, const int* mask, RunOrder ord) {
  __shared__ float2 sm[std::is_same<O, Canonical>::value ? 12 * (DSLASH_TPB + 1) : 1];
  const int ng = (nrhs + NR - 1) / NR;
  const int base = run_base(g, ord, blockIdx.x / ng), r0 = blockIdx.x % ng * NR;
  const bool a0 = !mask || mask[r0];
  if constexpr (NR == 1) {
    const int one[1] = {r0};
    if (a0) dslash_f32_site<O, DAGGER, 1>(in, out, gauge, clover, g, kappa, base, one, sm);
  } else {
    static_assert(NR == 2, "one or two right-hand sides per thread");
    const bool a1 = r0 + 1 < nrhs && (!mask || mask[r0 + 1]);
    const int two[2] = {r0, r0 + 1}, one[1] = {a0 ? r0 : r0 + 1};
    if (a0 && a1)
      dslash_f32_site<O, DAGGER, 2>(in, out, gauge, clover, g, kappa, base, two, sm);
    else if (a0 || a1)
      dslash_f32_site<O, DAGGER, 1>(in, out, gauge, clover, g, kappa, base, one, sm);
  }
}

// slab order with several RHS when a (t, z) plane holds whole runs
RunOrder run_order(const Geom& g, int nrhs) {
  RunOrder ord = {0, 1};
  const int plane = g.L[1] * g.L[2];
  if (nrhs > 1 && plane % DSLASH_TPB == 0) {
    ord.cp = plane / DSLASH_TPB;
    ord.zw = g.L[3] % 8 == 0 ? 8 : g.L[3] % 4 == 0 ? 4 : g.L[3] % 2 == 0 ? 2 : 1;
  }
  return ord;
}

template <typename O>
qcd_status launch_f64(qcd_ctx* c, const void* in, void* out, int nrhs, int dagger, const int* mask) {
  // (by the volume alone: a right-hand side gives the same bits in any batch)
  if (c->g.V <= SPLIT_MAX_V) {
    const unsigned grid = (unsigned)((c->g.V + SPLIT_SITES - 1) / SPLIT_SITES) * nrhs;
    auto kern = dagger ? k_dslash_split<O, 1> : k_dslash_split<O, 0>;
    kern<<<grid, 2 * SPLIT_SITES, 0, c->stream>>>((const char*)in, (char*)out, c->gaugeD.p, c->cloverD.p, c->g,
                                                  c->kappa, nrhs, mask);
  } else {
    const unsigned grid = (unsigned)((c->g.V + DSLASH_TPB - 1) / DSLASH_TPB) * nrhs;
    auto kern = dagger ? k_dslash<O, 1> : k_dslash<O, 0>;
    kern<<<grid, DSLASH_TPB, 0, c->stream>>>((const char*)in, (char*)out, c->gaugeD.p, c->cloverD.p, c->g, c->kappa,
                                             nrhs, mask, run_order(c->g, nrhs));
  }
  QCD_CUDA_OK(cudaGetLastError());
  return QCD_OK;
}

template <typename O>
qcd_status launch_f32(qcd_ctx* c, const void* in, void* out, int nrhs, int dagger, const int* mask) {
  const unsigned nb = (unsigned)((c->g.V + DSLASH_TPB - 1) / DSLASH_TPB);
  const bool two = nrhs > 1;
  auto kern = two ? (dagger ? k_dslash_f32<O, 1, 2> : k_dslash_f32<O, 0, 2>)
                  : (dagger ? k_dslash_f32<O, 1, 1> : k_dslash_f32<O, 0, 1>);
  kern<<<nb * (two ? (nrhs + 1) / 2 : 1), DSLASH_TPB, 0, c->stream>>>(
      (const char*)in, (char*)out, (const float4*)c->gaugeF.p, (const float4*)c->cloverF.p, c->g, (float)c->kappa, nrhs,
      mask, run_order(c->g, nrhs));
  QCD_CUDA_OK(cudaGetLastError());
  return QCD_OK;
}

}  // namespace

// Algorithmic cost per site: each input spinor read once, the output written
// once, the 4 links of the site and its clover term read once per launch;
// 1320 flops for the eight spin-projected hops and 504 for the clover term.
// out_prec = QCD_PREC_H16 (FP32 input only): the output is stored as FP16 with
// a per-site scale; DSLASH_CANONICAL: in the caller's layout, FP64.
qcd_status dslash_apply(qcd_ctx* c, const void* in, void* out, int prec, int nrhs, int dagger, const int* mask,
                        int nactive, int out_prec) {
  const double V = c->g.V;
  const bool canon = out_prec == DSLASH_CANONICAL;
  if (prec == QCD_PREC_F64) {
    ProfScope ps(c, FAM_DSLASH_D, V * (nactive * 2.0 * 192 + 4 * 144 + 576), V * nactive * 1824.0);
    return canon ? launch_f64<Canonical>(c, in, out, nrhs, dagger, mask)
                 : launch_f64<FieldsD>(c, in, out, nrhs, dagger, mask);
  }
  const double ob = canon ? 192 : out_prec == QCD_PREC_H16 ? (double)FieldsH::spinor_bytes : 96;
  ProfScope ps(c, FAM_DSLASH_F, V * (nactive * (96.0 + ob) + 4 * 48 + 288), V * nactive * 1824.0);
  return canon                       ? launch_f32<Canonical>(c, in, out, nrhs, dagger, mask)
         : out_prec == QCD_PREC_H16 ? launch_f32<FieldsH>(c, in, out, nrhs, dagger, mask)
                                    : launch_f32<FieldsF>(c, in, out, nrhs, dagger, mask);
}
