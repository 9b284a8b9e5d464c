// Local deflation (Sec. 2.2): deflation subspace, little Dirac operator
// (eq. little), its diagonal-block inverses, and the low-mode solve used by
// the deflated preconditioner M rho = Phi A^-1 Phi^+ rho + M_SAP(P_L rho).
//
// The deflation blocks are the SAP blocks (the paper takes the two block
// sizes equal).  Phi is stored as N_s FP32 global fields in the internal
// spinor layout; the restriction of field k to block b is phi_k^b.  Little
// vectors are float2 [rhs][block][k].  The little operator is stored per
// block as 9 N_s x N_s complex matrices: part 0 couples the block to itself,
// part 1 + 2 mu to the block at +mu and part 2 + 2 mu to the block at -mu:
//   A[b][0][k][l]      = (phi_k^b, D phi_l^b)
//   A[b][1+2mu][k][l]  = (phi_k^b, D phi_l^{b+mu})   (hops across the +mu face)
//   A[b][2+2mu][k][l]  = (phi_k^b, D phi_l^{b-mu})
#include <math.h>

#include <vector>

#include "spin_pair.cuh"

namespace {

constexpr int MAX_NS = 32;   // deflation fields (checked at qcd_deflation_setup)

struct BlkGeom {
  int b[4], nb[4], lst[4], vb, nblk;
};

BlkGeom blk_geom(const qcd_ctx* c) {
  BlkGeom bg;
  bg.vb = 1;
  bg.nblk = 1;
  for (int mu = 0; mu < 4; mu++) {
    bg.b[mu] = c->params.block[mu];
    bg.nb[mu] = c->g.L[mu] / bg.b[mu];
    bg.vb *= bg.b[mu];
    bg.nblk *= bg.nb[mu];
  }
  bg.lst[1] = 1;
  bg.lst[2] = bg.b[1];
  bg.lst[3] = bg.b[1] * bg.b[2];
  bg.lst[0] = bg.b[1] * bg.b[2] * bg.b[3];
  return bg;
}

// block coordinates of block number blk: blk = ((bt*nbz + bz)*nby + by)*nbx + bx
__device__ inline void blk_coords(const BlkGeom& bg, int blk, int bc[4]) {
  bc[1] = blk % bg.nb[1];
  int r = blk / bg.nb[1];
  bc[2] = r % bg.nb[2];
  r /= bg.nb[2];
  bc[3] = r % bg.nb[3];
  bc[0] = r / bg.nb[3];
}
__device__ inline int blk_index(const BlkGeom& bg, const int bc[4]) {
  return ((bc[0] * bg.nb[3] + bc[3]) * bg.nb[2] + bc[2]) * bg.nb[1] + bc[1];
}
// site of local index l in block blk; lc = local coordinates
__device__ inline int blk_site(const BlkGeom& bg, const Geom& g, int blk, int l, int lc[4], int c[4]) {
  int bc[4];
  blk_coords(bg, blk, bc);
  int r = l;
  lc[1] = r % bg.b[1]; r /= bg.b[1];
  lc[2] = r % bg.b[2]; r /= bg.b[2];
  lc[3] = r % bg.b[3];
  lc[0] = r / bg.b[3];
  for (int mu = 0; mu < 4; mu++) c[mu] = bc[mu] * bg.b[mu] + lc[mu];
  return ((c[0] * g.L[3] + c[3]) * g.L[2] + c[2]) * g.L[1] + c[1];
}
__device__ inline double2 dwarp_sum2(double2 v) {
#pragma unroll
  for (int o = 16; o > 0; o >>= 1) {
    v.x += __shfl_xor_sync(0xffffffffu, v.x, o);
    v.y += __shfl_xor_sync(0xffffffffu, v.y, o);
  }
  return v;
}
// block-wide complex sum, result broadcast to all threads (fixed order)
__device__ inline double2 cta_sum2(double2 v, double2* sh) {
  v = dwarp_sum2(v);
  const int w = threadIdx.x >> 5, l = threadIdx.x & 31, nw = (blockDim.x + 31) >> 5;
  __syncthreads();
  if (l == 0) sh[w] = v;
  __syncthreads();
  double2 t = make_double2(0, 0);
  for (int i = 0; i < nw; i++) {
    t.x += sh[i].x;
    t.y += sh[i].y;
  }
  return t;
}

// ---------------------------------------------------------------------------
// Block Gram-Schmidt (modified, in the order k = 0, 1, ...), one CTA per block
// ---------------------------------------------------------------------------
__global__ void k_dfl_gs(char* __restrict__ phi, Geom g, BlkGeom bg, int ns) {
  __shared__ double2 sh[32];
  const int blk = blockIdx.x, l = threadIdx.x;
  int lc[4], c[4];
  const int s = blk_site(bg, g, blk, l, lc, c);
  const size_t fb = FieldsF::spinor_bytes * (size_t)g.V;
  for (int k = 0; k < ns; k++) {
    Spinor<float> v = FieldsF::load_spinor(phi + k * fb, g.V, s);
    for (int j = 0; j < k; j++) {
      Spinor<float> u = FieldsF::load_spinor(phi + j * fb, g.V, s);
      float dr = 0, di = 0;
#pragma unroll
      for (int q = 0; q < 12; q++) {
        dr += u.c[q].re * v.c[q].re + u.c[q].im * v.c[q].im;
        di += u.c[q].re * v.c[q].im - u.c[q].im * v.c[q].re;
      }
      double2 d = cta_sum2(make_double2(dr, di), sh);
      Cplx<float> df = cmk((float)d.x, (float)d.y);
#pragma unroll
      for (int q = 0; q < 12; q++) v.c[q] = v.c[q] - df * u.c[q];
    }
    float n2 = 0;
#pragma unroll
    for (int q = 0; q < 12; q++) n2 += v.c[q].re * v.c[q].re + v.c[q].im * v.c[q].im;
    double2 n = cta_sum2(make_double2(n2, 0), sh);
    float inv = n.x > 0 ? (float)(1.0 / sqrt(n.x)) : 0.f;
#pragma unroll
    for (int q = 0; q < 12; q++) v.c[q] = inv * v.c[q];
    FieldsF::store_spinor(phi + k * fb, g.V, s, v);
  }
}

// ---------------------------------------------------------------------------
// Parts of D phi_l split by block: Y[0] = D_block phi_l (site-diagonal term and
// hops inside the block), Y[1+mu] = the hops across the two mu faces of the
// block (the +mu and -mu faces are disjoint sets of sites when b_mu >= 2).
// One thread per (site, l).
// ---------------------------------------------------------------------------
template <int MU>
__device__ inline void ypart_dir(Spinor<float>& yint, Spinor<float>& yface, const char* in, const void* gauge,
                                 const Geom& g, const BlkGeom& bg, int s, const int c[4], const int lc[4],
                                 float mk) {
  {
    int sf = site_fwd(g, s, c, MU);
    float sign = (MU == 0 && c[0] == g.L[0] - 1) ? (float)g.bc_t * mk : mk;
    HalfSpinor<float> h = project<MU, -1>(FieldsF::load_spinor(in, g.V, sf));
    h = su3_mul(FieldsF::load_link(gauge, g.V, MU, s), h);
    if (lc[MU] < bg.b[MU] - 1) accum_recon<MU, -1>(yint, h, sign);
    else accum_recon<MU, -1>(yface, h, sign);
  }
  {
    int sb = site_bwd(g, s, c, MU);
    float sign = (MU == 0 && c[0] == 0) ? (float)g.bc_t * mk : mk;
    HalfSpinor<float> h = project<MU, +1>(FieldsF::load_spinor(in, g.V, sb));
    h = su3_dag_mul(FieldsF::load_link(gauge, g.V, MU, sb), h);
    if (lc[MU] > 0) accum_recon<MU, +1>(yint, h, sign);
    else accum_recon<MU, +1>(yface, h, sign);
  }
}

__global__ void __launch_bounds__(128) k_dfl_ypart(const char* __restrict__ phi, char* __restrict__ Y,
                                                   const void* __restrict__ gauge, const void* __restrict__ clover,
                                                   Geom g, BlkGeom bg, float kappa, int ns) {
  const int l = blockIdx.y;
  const int s = blockIdx.x * blockDim.x + threadIdx.x;
  if (s >= g.V) return;
  const size_t fb = FieldsF::spinor_bytes * (size_t)g.V;
  const char* in = phi + l * fb;
  int c[4], lc[4];
  site_coords(g, s, c);
  for (int mu = 0; mu < 4; mu++) lc[mu] = c[mu] % bg.b[mu];
  Spinor<float> yint = clover_apply<FieldsF>(clover, g.V, s, FieldsF::load_spinor(in, g.V, s));
  Spinor<float> yf[4];
#pragma unroll
  for (int m = 0; m < 4; m++)
#pragma unroll
    for (int q = 0; q < 12; q++) yf[m].c[q] = cmk(0.f, 0.f);
  ypart_dir<0>(yint, yf[0], in, gauge, g, bg, s, c, lc, -kappa);
  ypart_dir<1>(yint, yf[1], in, gauge, g, bg, s, c, lc, -kappa);
  ypart_dir<2>(yint, yf[2], in, gauge, g, bg, s, c, lc, -kappa);
  ypart_dir<3>(yint, yf[3], in, gauge, g, bg, s, c, lc, -kappa);
  FieldsF::store_spinor(Y + (0 * (size_t)ns + l) * fb, g.V, s, yint);
#pragma unroll
  for (int m = 0; m < 4; m++) FieldsF::store_spinor(Y + ((1 + m) * (size_t)ns + l) * fb, g.V, s, yf[m]);
}

// ---------------------------------------------------------------------------
// Per-block projection c[r][b][k] = sum_{y in b, comp} conj(Phi_k(y)) rho_r(y)
// of the unmasked right-hand sides on the deflation fields.  (The little Dirac
// operator itself is built on the tensor cores, dfl_tc.cu.)
//
// One CTA per block.  Chunks of PTS sites of both operands are staged entry-major
// (Pt[e][k], Rt[e][r], e = component * PTS + site; rows two words longer than the
// tiles, so that consecutive sites fall into different banks).  A thread owns a tile of
// 4 fields x 4 right-hand sides on one of the slices of the entries: four 128-bit
// shared-memory reads for 16 complex products (one output per thread took two
// reads a product, which bound the kernel).  The slices are summed in a fixed order
// at the end.
// ---------------------------------------------------------------------------
constexpr int PTS = 16;
constexpr int GEMM_TPB = 256;
constexpr int TK = 4, TR = 4;

struct ProjectShape {
  int tiles_k, tiles_r, slices, ldp, ldr;
  size_t smem;
};
ProjectShape project_shape(int ns, int nrhs) {
  ProjectShape s;
  s.tiles_k = (ns + TK - 1) / TK;
  s.tiles_r = (nrhs + TR - 1) / TR;
  s.slices = GEMM_TPB / (s.tiles_k * s.tiles_r);   // ns <= 32, nrhs <= 24: at most 64 tiles
  s.ldp = s.tiles_k * TK + 2;
  s.ldr = s.tiles_r * TR + 2;
  const size_t stage = (size_t)12 * PTS * (s.ldp + s.ldr);
  const size_t red = (size_t)s.slices * s.tiles_k * s.tiles_r * TK * TR;
  s.smem = sizeof(float2) * (stage > red ? stage : red);
  return s;
}

// acc += conj(x) y in (re, im) lanes; miy = -i y
__device__ __forceinline__ void cmac_conj2(float2& acc, float2 x, float2 y, float2 miy) {
  acc = pfma(pbc(x.x), y, acc);
  acc = pfma(pbc(x.y), miy, acc);
}

__global__ void __launch_bounds__(GEMM_TPB) k_dfl_project(const char* __restrict__ phi, const char* __restrict__ rho,
                                                           float2* __restrict__ cout, Geom g, BlkGeom bg, int ns,
                                                           int nrhs, ProjectShape sh, const int* mask) {
  extern __shared__ __align__(16) unsigned char smem_raw[];
  float2* Pt = (float2*)smem_raw;                          // [12 PTS][ldp]
  float2* Rt = Pt + (size_t)12 * PTS * sh.ldp;             // [12 PTS][ldr]
  const int blk = blockIdx.x;
  const size_t fb = FieldsF::spinor_bytes * (size_t)g.V;
  const int kp = sh.tiles_k * TK, rp = sh.tiles_r * TR;    // padded rows (zeros beyond ns and nrhs)
  const int ntile = sh.tiles_k * sh.tiles_r;
  const int tile = threadIdx.x % ntile, slice = threadIdx.x / ntile;
  const int k0 = (tile / sh.tiles_r) * TK, r0 = (tile % sh.tiles_r) * TR;
  float2 acc[TK][TR];
#pragma unroll
  for (int i = 0; i < TK; i++)
#pragma unroll
    for (int j = 0; j < TR; j++) acc[i][j] = p2(0.f, 0.f);
  __shared__ int site[PTS];
  for (int t0 = 0; t0 < bg.vb; t0 += PTS) {
    __syncthreads();
    if (threadIdx.x < PTS) {
      int lc[4], c[4];
      site[threadIdx.x] = blk_site(bg, g, blk, t0 + threadIdx.x, lc, c);
    }
    __syncthreads();
    for (int task = threadIdx.x; task < (kp + rp) * PTS; task += blockDim.x) {
      const int i = task % PTS, f = task / PTS;
      const int s = site[i];
      const bool isphi = f < kp;
      const int r = f - kp;
      const bool on = isphi ? f < ns : (r < nrhs && (!mask || mask[r]));
      const float4* src = (const float4*)(isphi ? phi + (size_t)f * fb : rho + (size_t)r * fb);
      float2* dst = isphi ? Pt + f : Rt + r;
      const int ld = isphi ? sh.ldp : sh.ldr;
#pragma unroll
      for (int q = 0; q < 6; q++) {
        const float4 v = on ? __ldg(src + (size_t)q * g.V + s) : make_float4(0.f, 0.f, 0.f, 0.f);
        dst[(2 * q * PTS + i) * ld] = make_float2(v.x, v.y);
        dst[((2 * q + 1) * PTS + i) * ld] = make_float2(v.z, v.w);
      }
    }
    __syncthreads();
    if (slice < sh.slices)
      for (int e = slice; e < 12 * PTS; e += sh.slices) {
        const float4* xp = (const float4*)(Pt + e * sh.ldp + k0);
        const float4* yp = (const float4*)(Rt + e * sh.ldr + r0);
        const float4 x0 = xp[0], x1 = xp[1], y0 = yp[0], y1 = yp[1];
        const float2 x[TK] = {p2(x0.x, x0.y), p2(x0.z, x0.w), p2(x1.x, x1.y), p2(x1.z, x1.w)};
        const float2 y[TR] = {p2(y0.x, y0.y), p2(y0.z, y0.w), p2(y1.x, y1.y), p2(y1.z, y1.w)};
#pragma unroll
        for (int j = 0; j < TR; j++) {
          const float2 miy = p2(y[j].y, -y[j].x);
#pragma unroll
          for (int i = 0; i < TK; i++) cmac_conj2(acc[i][j], x[i], y[j], miy);
        }
      }
  }
  __syncthreads();
  float2* red = (float2*)smem_raw;   // [slice][r][k] over the padded rows
  if (slice < sh.slices)
#pragma unroll
    for (int i = 0; i < TK; i++)
#pragma unroll
      for (int j = 0; j < TR; j++)
        red[((size_t)slice * rp + r0 + j) * kp + k0 + i] = acc[i][j];
  __syncthreads();
  for (int o = threadIdx.x; o < ns * nrhs; o += blockDim.x) {
    const int r = o / ns, k = o - r * ns;
    float2 t = make_float2(0.f, 0.f);
    for (int q = 0; q < sh.slices; q++) {
      const float2 v = red[((size_t)q * rp + r) * kp + k];
      t.x += v.x;
      t.y += v.y;
    }
    cout[((size_t)r * bg.nblk + blk) * ns + k] = t;
  }
}

// Prolongation x_r(y) = sum_k e[r][b(y)][k] phi_k(y).  Each of a block's three CTAs
// takes PRW of the six words of its sites; the block's coefficients in shared memory;
// a thread takes a word (two components) of up to 12 right-hand sides at a time, so
// phi is read once per 12.  (16^3x32, 12 RHS, N_s 20: with two-lane arithmetic here and
// in the projection, and three CTAs per block instead of one, which left the second of
// two waves two thirds empty, 1.77 -> 1.61 ms of deflation per outer iteration.
// Fields kept in block order: 1.58, not worth a second layout.)
constexpr int PRG = 12, PRW = 2;
__global__ void __launch_bounds__(256, 2) k_dfl_prolong(const char* __restrict__ phi, const float2* __restrict__ e,
                                                        char* __restrict__ x, Geom g, BlkGeom bg, int ns, int nrhs,
                                                        const int* mask) {
  extern __shared__ __align__(16) unsigned char smem_raw[];
  float2* cf = (float2*)smem_raw;   // [k][nrhs rounded up to PRG], zeros beyond nrhs
  const int blk = blockIdx.x / (6 / PRW), ld = (nrhs + PRG - 1) / PRG * PRG;
  const int q0 = blockIdx.x % (6 / PRW) * PRW;
  for (int o = threadIdx.x; o < ns * ld; o += blockDim.x) {
    const int r = o / ns, k = o - r * ns;
    cf[k * ld + r] = r < nrhs ? e[((size_t)r * bg.nblk + blk) * ns + k] : make_float2(0.f, 0.f);
  }
  __syncthreads();
  const size_t fb = FieldsF::spinor_bytes * (size_t)g.V;
  for (int l = threadIdx.x; l < bg.vb; l += blockDim.x) {
    int lc[4], c[4];
    const int s = blk_site(bg, g, blk, l, lc, c);
    for (int r0 = 0; r0 < nrhs; r0 += PRG)
#pragma unroll 1
      for (int q = q0; q < q0 + PRW; q++) {
        float2 a0[PRG], a1[PRG];
#pragma unroll
        for (int i = 0; i < PRG; i++) a0[i] = a1[i] = p2(0.f, 0.f);
#pragma unroll 4
        for (int k = 0; k < ns; k++) {
          const float4 v = __ldg((const float4*)(phi + k * fb) + (size_t)q * g.V + s);
          const float2 v0 = p2(v.x, v.y), v1 = p2(v.z, v.w), iv0 = p2(-v.y, v.x), iv1 = p2(-v.w, v.z);
          const float4* w = (const float4*)(cf + k * ld + r0);
#pragma unroll
          for (int i = 0; i < PRG; i += 2) {
            const float4 u = w[i >> 1];
            a0[i] = pfma(pbc(u.y), iv0, pfma(pbc(u.x), v0, a0[i]));
            a1[i] = pfma(pbc(u.y), iv1, pfma(pbc(u.x), v1, a1[i]));
            a0[i + 1] = pfma(pbc(u.w), iv0, pfma(pbc(u.z), v0, a0[i + 1]));
            a1[i + 1] = pfma(pbc(u.w), iv1, pfma(pbc(u.z), v1, a1[i + 1]));
          }
        }
#pragma unroll
        for (int i = 0; i < PRG; i++)
          if (r0 + i < nrhs && (!mask || mask[r0 + i]))
            ((float4*)(x + (size_t)(r0 + i) * fb))[(size_t)q * g.V + s] =
                make_float4(a0[i].x, a0[i].y, a1[i].x, a1[i].y);
      }
  }
}

// ---------------------------------------------------------------------------
// Diagonal-block inverses by Gauss-Jordan elimination with partial pivoting
// in FP64 (one 32-thread CTA per block); stored in FP64.
// ---------------------------------------------------------------------------
__global__ void k_dfl_block_inverse(const double2* __restrict__ A, double2* __restrict__ Ainv, int ns, int* singular) {
  extern __shared__ __align__(16) unsigned char smem_raw[];
  double2* M = (double2*)smem_raw;   // [ns][2 ns]
  __shared__ int piv;
  __shared__ double2 fcol[32];       // column col of M before the elimination step
  const int blk = blockIdx.x, w = 2 * ns;
  const double2* a = A + (size_t)blk * 9 * ns * ns;   // part 0
  for (int idx = threadIdx.x; idx < ns * w; idx += blockDim.x) {
    int i = idx / w, j = idx - i * w;
    double2 v = make_double2(0, 0);
    if (j < ns) v = make_double2(a[i * ns + j].x, a[i * ns + j].y);
    else if (j - ns == i) v = make_double2(1, 0);
    M[idx] = v;
  }
  __syncthreads();
  for (int col = 0; col < ns; col++) {
    if (threadIdx.x == 0) {
      int best = col;
      double bv = -1;
      for (int i = col; i < ns; i++) {
        double m = M[i * w + col].x * M[i * w + col].x + M[i * w + col].y * M[i * w + col].y;
        if (m > bv) { bv = m; best = i; }
      }
      piv = best;
      if (bv <= 0) atomicExch(singular, 1);
    }
    __syncthreads();
    const int p = piv;
    if (p != col)
      for (int j = threadIdx.x; j < w; j += blockDim.x) {
        double2 t = M[col * w + j];
        M[col * w + j] = M[p * w + j];
        M[p * w + j] = t;
      }
    __syncthreads();
    double2 d = M[col * w + col];
    double dn = d.x * d.x + d.y * d.y;
    double2 inv = dn > 0 ? make_double2(d.x / dn, -d.y / dn) : make_double2(0, 0);
    __syncthreads();
    for (int j = threadIdx.x; j < w; j += blockDim.x) {
      double2 v = M[col * w + j];
      M[col * w + j] = make_double2(v.x * inv.x - v.y * inv.y, v.x * inv.y + v.y * inv.x);
    }
    for (int i = threadIdx.x; i < ns; i += blockDim.x) fcol[i] = M[i * w + col];
    __syncthreads();
    for (int idx = threadIdx.x; idx < ns * w; idx += blockDim.x) {
      int i = idx / w, j = idx - i * w;
      if (i == col) continue;
      double2 f = fcol[i];
      double2 v = M[col * w + j];
      M[idx].x -= f.x * v.x - f.y * v.y;
      M[idx].y -= f.x * v.y + f.y * v.x;
    }
    __syncthreads();
  }
  for (int idx = threadIdx.x; idx < ns * ns; idx += blockDim.x) {
    int i = idx / ns, j = idx - i * ns;
    double2 v = M[i * w + ns + j];
    Ainv[(size_t)blk * ns * ns + idx] = v;
  }
}

// ---------------------------------------------------------------------------
// Little operator and little vector algebra.  x, y: float2 [nrhs][nblk][ns].
// A and the diagonal-block inverses are stored in FP64; the little solve
// applies FP32 copies of them (an approximate inverse inside the flexible
// preconditioner, whose FP32 vectors bound its accuracy anyway: FP64
// arithmetic runs at 1/64 of the FP32 rate on this GPU).  The FP64 form
// serves the exact products A x of the test entry point.
// ---------------------------------------------------------------------------
__device__ inline void little_mac(double& ar, double& ai, double2 a, float2 v) {
  ar = fma(a.x, (double)v.x, ar);
  ar = fma(-a.y, (double)v.y, ar);
  ai = fma(a.x, (double)v.y, ai);
  ai = fma(a.y, (double)v.x, ai);
}
__device__ inline void little_mac(float& ar, float& ai, float2 a, float2 v) {
  ar = fmaf(a.x, v.x, ar);
  ar = fmaf(-a.y, v.y, ar);
  ai = fmaf(a.x, v.y, ai);
  ai = fmaf(a.y, v.x, ai);
}

// the blocks the nine parts of A couple a block to
__device__ inline void little_neighbours(const BlkGeom& bg, int blk, int nbr[9]) {
  int bc[4];
  blk_coords(bg, blk, bc);
  nbr[0] = blk;
#pragma unroll
  for (int mu = 0; mu < 4; mu++) {
    int cc[4] = {bc[0], bc[1], bc[2], bc[3]};
    cc[mu] = bc[mu] + 1 == bg.nb[mu] ? 0 : bc[mu] + 1;
    nbr[1 + 2 * mu] = blk_index(bg, cc);
    cc[mu] = bc[mu] == 0 ? bg.nb[mu] - 1 : bc[mu] - 1;
    nbr[2 + 2 * mu] = blk_index(bg, cc);
  }
}

// y = A x with the FP64 matrix (the test entry point).  One CTA per block, thread
// (k, rr) = row k for the RHS rr, rr + rb, ...: the rb threads of a row read the same
// matrix row (L1 broadcast), the ns threads of an RHS the same neighbour vector.
__global__ void k_little_apply(const double2* __restrict__ M, const float2* __restrict__ x, float2* __restrict__ y,
                               BlkGeom bg, int ns, int nrhs) {
  const int blk = blockIdx.x;
  const int k = threadIdx.x % ns, rr = threadIdx.x / ns;
  const int rb = blockDim.x / ns;
  if (rr >= rb) return;
  int nbr[9];
  little_neighbours(bg, blk, nbr);
  for (int r = rr; r < nrhs; r += rb) {
    double ar = 0, ai = 0;
    for (int p = 0; p < 9; p++) {
      const double2* row = M + (((size_t)blk * 9 + p) * ns + k) * ns;
      const float2* xv = x + ((size_t)r * bg.nblk + nbr[p]) * ns;
      for (int l = 0; l < ns; l++) little_mac(ar, ai, __ldg(row + l), __ldg(xv + l));
    }
    y[((size_t)r * bg.nblk + blk) * ns + k] = make_float2((float)ar, (float)ai);
  }
}

// FP32 copy of na / (ns ns) matrices, transposed
__global__ void k_little_transpose(const double2* __restrict__ in, float2* __restrict__ out, int ns, size_t na) {
  for (size_t i = blockIdx.x * (size_t)blockDim.x + threadIdx.x; i < na; i += (size_t)gridDim.x * blockDim.x) {
    const size_t m = i / ns, b = m / ns;
    const int l = (int)(m - b * ns), k = (int)(i - m * ns);
    const double2 v = in[(b * ns + k) * ns + l];
    out[i] = make_float2((float)v.x, (float)v.y);
  }
}

// FP32 copy of an FP64 complex array
__global__ void k_to_float2(const double2* __restrict__ in, float2* __restrict__ out, size_t n) {
  for (size_t i = blockIdx.x * (size_t)blockDim.x + threadIdx.x; i < n; i += (size_t)gridDim.x * blockDim.x)
    out[i] = make_float2((float)in[i].x, (float)in[i].y);
}

// ---------------------------------------------------------------------------
// The little GCR step in five launches (twelve before: product with the diagonal
// inverses, product with A, dots, their sums, orthogonalisation, norm, its sum,
// scaling, overlap, its sum, update).  The vectors of a 16^3x32 lattice are 1 MB
// for 12 RHS, so a launch takes microseconds and their number counts.  Sums over
// threads are FP64 in a fixed order; a CTA of the summing kernels is one warp (an FP64
// addition of a warp takes the SM 16 cycles: the shuffle sums of 256 threads were
// most of the time of the dots).  Masked right-hand sides have a zero residual and
// stay zero.  A deflated 16^3x32 solve, 12 RHS, N_s 20, 24 steps: all deflation
// kernels of an outer iteration 3.5 -> 1.75 ms; with each launch overlapping the end of
// the one before it 1.41 -> 1.24.
// ---------------------------------------------------------------------------
constexpr int LTPB = 256;
constexpr int LITTLE_G = 608;    // CTAs of the kernels that leave partial sums
constexpr int LITTLE_RHS = 24;   // right-hand sides of one little solve

// hi + lo += v, without rounding but of lo
__device__ __forceinline__ void two_sum(float& hi, float& lo, float v) {
  const float t = hi + v, b = t - hi;
  lo += (hi - (t - b)) + (v - b);
  hi = t;
}

// The dots of q's block (qs) with the nj vectors' (at qb, `stride` apart, their right-hand
// sides rstride) added to the running sums.  At most ten products are summed in FP32 (in two
// chains, which round less than the one of 8 to 10 that the dots had in a launch of their
// own); what is summed over a block's chunks and a CTA's blocks, N_s products of each, keeps
// the exact error of every addition beside it (Knuth's TwoSum).  A thread takes a chunk, so
// that the loads of a block are one round; its sum goes to the first thread of its dot,
// whose running sum waits in shared memory (in registers it would spill).
__device__ __forceinline__ void little_dots(const float2* qb, size_t stride, size_t rstride, const float2* qs, float4* dot,
                                         int ns, int n, int nj) {
  const int lch = ns <= 10 ? 0 : ns <= 20 ? 1 : 2;               // 2^lch chunks
  const int len = (((ns + (1 << lch) - 1) >> lch) + 1) & ~1;     // of len products
  for (int t = threadIdx.x; t < (((nj * n) << lch) + 31 & ~31); t += LTPB) {   // (whole warps)
    const int o = t >> lch, ch = t & ((1 << lch) - 1);
    float2 sum[2] = {make_float2(0.f, 0.f), make_float2(0.f, 0.f)};
    if (o < nj * n) {
      const int j = o / n, r = o - j * n;
      const float2* qj = qb + j * stride + r * rstride;
      auto mac = [](float2& s, float2 u, float2 v) {
        s.x = fmaf(u.x, v.x, s.x);
        s.x = fmaf(u.y, v.y, s.x);
        s.y = fmaf(u.x, v.y, s.y);
        s.y = fmaf(-u.y, v.x, s.y);
      };
      const int k0 = ch * len, kn = min(len, ns - k0);
      float2 u[10];   // all loads before the first use
      if (ns % 2 == 0) {   // (then every little vector's block is 16-byte aligned)
#pragma unroll
        for (int k = 0; k < 10; k += 2) {
          const float4 w = k < kn ? __ldcg((const float4*)(qj + k0 + k)) : make_float4(0.f, 0.f, 0.f, 0.f);
          u[k] = p2(w.x, w.y);
          u[k + 1] = p2(w.z, w.w);
        }
      } else {
#pragma unroll
        for (int k = 0; k < 10; k++) u[k] = k < kn ? __ldcg(qj + k0 + k) : make_float2(0.f, 0.f);
      }
#pragma unroll
      for (int k = 0; k < 10; k++)
        if (k < kn) mac(sum[k & 1], u[k], qs[(k0 + k) * n + r]);
    }
    const float2 v = make_float2(sum[0].x + sum[1].x, sum[0].y + sum[1].y);
    const bool first = ch == 0 && o < nj * n;
    float4 d = first ? dot[o] : make_float4(0.f, 0.f, 0.f, 0.f);
    for (int c = 0; c < 1 << lch; c++) {
      two_sum(d.x, d.z, __shfl_sync(0xffffffffu, v.x, (t & 31) - ch + c));
      two_sum(d.y, d.w, __shfl_sync(0xffffffffu, v.y, (t & 31) - ch + c));
    }
    if (first) dot[o] = d;
  }
}

// q = A p on the CTA's blocks, and the CTA's partial sums of (q_j, q), j < nj, to
// part[(r nj + j) gridDim + cta].  At: the matrix with the row index of each of its
// nine parts fastest.  A thread takes row k of one of the nine parts for up to LQR right-hand
// sides: the matrix is read once, consecutive rows by consecutive threads, from
// global memory, and the neighbours' p are broadcast reads from shared memory, six
// 128-bit words for 12 products.  (One output per thread took two shared-memory words
// per product, 86,000 per block and step, and staged the matrix.)  Bound by the latency
// of its loads and the barriers between its phases (16^3x32, 12 RHS, N_s 12: issue 22 %,
// waits for barriers 9.0 and for loads 7.4 cycles per instruction): four CTAs of 64 registers per SM hold all 512 blocks of a 16^3x32
// lattice at once (three, in two waves, are no faster than the old form); the dots read
// 128-bit words, the orthogonalisation below keeps 24 loads in flight: deflation 1.61
// -> 1.41 ms per outer iteration (12 RHS, N_s 20, 24 steps).  The nine parts are summed in a
// fixed order.
constexpr int LQR = 12;
constexpr size_t little_q_smem(int ns, int n, int nj) {
  return sizeof(float2) * ((size_t)2 * 9 * ns * LQR + (size_t)(ns * n + 1) / 2 * 2) + sizeof(float4) * nj * n;
}
__global__ void __launch_bounds__(LTPB, 4) k_little_q(const float2* __restrict__ At, const float2* __restrict__ p,
                                                   float2* __restrict__ q, const float2* __restrict__ qbase,
                                                   size_t stride, int nj, double2* __restrict__ part, BlkGeom bg,
                                                   int ns, int n) {
  extern __shared__ __align__(16) unsigned char smem_raw[];
  float2* xs = (float2*)smem_raw;                 // [9 ns][LQR]
  float2* red = xs + (size_t)9 * ns * LQR;        // [9][LQR][ns]
  float2* qs = red + (size_t)9 * ns * LQR;        // [ns][n]
  float4* dot = (float4*)(qs + (size_t)(ns * n + 1) / 2 * 2);   // [nj][n] (sum re, im, their errors)
  launch_dependents();
  dependency_wait();
  for (int o = threadIdx.x; o < nj * n; o += LTPB) dot[o] = make_float4(0.f, 0.f, 0.f, 0.f);
  for (int blk = blockIdx.x; blk < bg.nblk; blk += gridDim.x) {
    for (int c0 = 0; c0 < n; c0 += LQR) {
      int nbr[9];   // (here: not in registers during the products below)
      little_neighbours(bg, blk, nbr);
      __syncthreads();
#pragma unroll
      for (int m = 0; m < 9; m++)
        for (int i = threadIdx.x; i < ns * LQR; i += LTPB) {
          const int r = i / ns, k = i - r * ns;
          xs[(m * ns + k) * LQR + r] =
              c0 + r < n ? __ldcg(p + ((size_t)(c0 + r) * bg.nblk + nbr[m]) * ns + k) : make_float2(0.f, 0.f);
        }
      __syncthreads();
      for (int t = threadIdx.x; t < 9 * ns; t += LTPB) {
        const int m = t / ns, k = t - m * ns;
        const float2* a = At + ((size_t)blk * 9 + m) * ns * ns + k;
        const float4* xv = (const float4*)(xs + (size_t)m * ns * LQR);
        float2 u[LQR];
#pragma unroll
        for (int r = 0; r < LQR; r++) u[r] = p2(0.f, 0.f);
        auto row = [&](int l, float2 w) {
          const float2 wi = p2(-w.y, w.y);
#pragma unroll
          for (int r = 0; r < LQR; r += 2) {
            const float4 x = xv[(l * LQR + r) >> 1];
            u[r] = pfma(wi, p2(x.y, x.x), pfma(pbc(w.x), p2(x.x, x.y), u[r]));
            u[r + 1] = pfma(wi, p2(x.w, x.z), pfma(pbc(w.x), p2(x.z, x.w), u[r + 1]));
          }
        };
        int l = 0;
        for (; l + 8 <= ns; l += 8) {   // 8 loads before the first use
          float2 w[8];   // (left to the compiler they are not: 10,400 -> 13,400 cycles, N_s 20)
#pragma unroll
          for (int i = 0; i < 8; i++) w[i] = __ldg(a + (l + i) * ns);
#pragma unroll
          for (int i = 0; i < 8; i++) row(l + i, w[i]);
        }
#pragma unroll 1
        for (; l < ns; l++) row(l, __ldg(a + l * ns));
#pragma unroll
        for (int r = 0; r < LQR; r++) red[(m * LQR + r) * ns + k] = u[r];
      }
      __syncthreads();
      for (int o = threadIdx.x; o < ns * LQR; o += LTPB) {
        const int r = o / ns, k = o - r * ns;
        if (c0 + r >= n) continue;
        float2 t = red[o];
#pragma unroll
        for (int m = 1; m < 9; m++) {
          const float2 w = red[m * LQR * ns + o];
          t.x += w.x;
          t.y += w.y;
        }
        qs[k * n + c0 + r] = t;
        q[((size_t)(c0 + r) * bg.nblk + blk) * ns + k] = t;
      }
    }
    if (nj == 0) continue;
    __syncthreads();
    little_dots(qbase + (size_t)blk * ns, stride, (size_t)bg.nblk * ns, qs, dot, ns, n, nj);
  }
  __syncthreads();
  for (int o = threadIdx.x; o < nj * n; o += LTPB) {
    const int j = o / n, r = o - j * n;
    const float4 t = dot[o];
    part[((size_t)r * nj + j) * gridDim.x + blockIdx.x] =
        make_double2((double)t.x + (double)t.z, (double)t.y + (double)t.w);
  }
}

// out[j][r] = sum over g of part[(r nj + j) G + g]: one warp per (j, r)
__global__ void k_little_sum(const double2* __restrict__ part, int nj, int G, double2* __restrict__ out, int n) {
  const int j = blockIdx.x, r = blockIdx.y;
  double2 t = make_double2(0, 0);
  launch_dependents();
  dependency_wait();
  for (int i = threadIdx.x; i < G; i += 32) {
    const double2 v = __ldcg(part + ((size_t)r * nj + j) * G + i);
    t.x += v.x;
    t.y += v.y;
  }
  t = dwarp_sum2(t);
  if (threadIdx.x == 0) out[(size_t)j * n + r] = t;
}

// q -= sum_j d_j q_j, p -= sum_j d_j p_j; CTA partial sums of |q|^2 (part[r][0])
// and (q, res) (part[r][1])
__global__ void __launch_bounds__(LTPB) k_little_orth(float2* __restrict__ qi, float2* __restrict__ pi,
                                                      const float2* __restrict__ qbase,
                                                      const float2* __restrict__ pbase, size_t stride, int nj,
                                                      const double2* __restrict__ d, const float2* __restrict__ res,
                                                      int N, int n, double2* __restrict__ part) {
  __shared__ float2 ds[64];
  __shared__ float sh[3][LTPB];
  const int r = blockIdx.y;
  launch_dependents();
  dependency_wait();
  if ((int)threadIdx.x < nj) {
    const double2 v = __ldcg(d + (size_t)threadIdx.x * n + r);
    ds[threadIdx.x] = make_float2((float)v.x, (float)v.y);
  }
  __syncthreads();
  float n2 = 0.f, cr = 0.f, ci = 0.f;
  for (int i = blockIdx.x * LTPB + threadIdx.x; i < N; i += gridDim.x * LTPB) {
    const size_t o = (size_t)r * N + i;
    float2 q = __ldcg(qi + o), p = __ldcg(pi + o);
#pragma unroll 12
    for (int j = 0; j < nj; j++) {
      const float2 w = ds[j], a = __ldcg(qbase + j * stride + o), b = __ldcg(pbase + j * stride + o);
      q.x -= w.x * a.x - w.y * a.y; q.y -= w.x * a.y + w.y * a.x;
      p.x -= w.x * b.x - w.y * b.y; p.y -= w.x * b.y + w.y * b.x;
    }
    qi[o] = q;
    pi[o] = p;
    const float2 v = __ldcg(res + o);
    n2 = fmaf(q.x, q.x, n2);
    n2 = fmaf(q.y, q.y, n2);
    cr = fmaf(q.x, v.x, cr);
    cr = fmaf(q.y, v.y, cr);
    ci = fmaf(q.x, v.y, ci);
    ci = fmaf(-q.y, v.x, ci);
  }
  sh[0][threadIdx.x] = n2;
  sh[1][threadIdx.x] = cr;
  sh[2][threadIdx.x] = ci;
  __syncthreads();
  const int w = threadIdx.x >> 5, l = threadIdx.x & 31;
  if (w < 3) {
    double t = 0;
#pragma unroll
    for (int i = 0; i < LTPB / 32; i++) t += (double)sh[w][32 * i + l];
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) t += __shfl_xor_sync(0xffffffffu, t, o);
    if (l == 0) {
      double* out = (double*)(part + (size_t)r * 2 * gridDim.x);
      if (w == 0) out[2 * blockIdx.x] = t;
      else out[2 * (gridDim.x + blockIdx.x) + w - 1] = t;
    }
  }
}

// from the partial sums of k_little_orth: f = 1/|q| and alpha = (q, res)/|q|^2 (the
// step along the normalised q is alpha |q|), per right-hand side {f, alpha |q|}
__global__ void k_little_scalars(const double2* __restrict__ part, int G, float4* __restrict__ out) {
  const int r = blockIdx.x;
  double2 a = make_double2(0, 0), c = make_double2(0, 0);
  launch_dependents();
  dependency_wait();
  for (int i = threadIdx.x; i < G; i += 32) {
    a.x += __ldcg(part + (size_t)r * 2 * G + i).x;
    const double2 v = __ldcg(part + ((size_t)r * 2 + 1) * G + i);
    c.x += v.x;
    c.y += v.y;
  }
  a = dwarp_sum2(a);
  c = dwarp_sum2(c);
  if (threadIdx.x == 0) {
    const double f = a.x > 0 ? 1.0 / sqrt(a.x) : 0.0;
    out[r] = make_float4((float)f, (float)(c.x * f), (float)(c.y * f), 0.f);
  }
}

// q, p normalised; x += alpha p, res -= alpha q (first: x = alpha p); pnext = the
// diagonal-block inverses times the new residual.  start: only that product.
__global__ void __launch_bounds__(LTPB) k_little_step(float2* __restrict__ x, float2* __restrict__ res,
                                                      float2* __restrict__ p, float2* __restrict__ q,
                                                      float2* __restrict__ pnext, const float2* __restrict__ Ainv,
                                                      const float4* __restrict__ sc, int first, int start, BlkGeom bg,
                                                      int ns, int n) {
  extern __shared__ __align__(16) unsigned char smem_raw[];
  float2* rs = (float2*)smem_raw;                 // [ns][n]
  float2* As = rs + (size_t)ns * n;               // [ns][ns]
  launch_dependents();
  for (int blk = blockIdx.x; blk < bg.nblk; blk += gridDim.x) {
    __syncthreads();
    if (pnext)
      for (int i = threadIdx.x; i < ns * ns; i += LTPB) As[i] = __ldg(Ainv + (size_t)blk * ns * ns + i);
    dependency_wait();   // (the inverses are constant)
    for (int i = threadIdx.x; i < ns * n; i += LTPB) {
      const int r = i / ns, k = i - r * ns;
      const size_t o = ((size_t)r * bg.nblk + blk) * ns + k;
      float2 v = __ldcg(res + o);
      if (!start) {
        const float4 c = __ldcg(sc + r);
        float2 pp = __ldcg(p + o), qq = __ldcg(q + o), xx = first ? make_float2(0.f, 0.f) : __ldcg(x + o);
        pp.x *= c.x; pp.y *= c.x;
        qq.x *= c.x; qq.y *= c.x;
        xx.x += c.y * pp.x - c.z * pp.y; xx.y += c.y * pp.y + c.z * pp.x;
        v.x -= c.y * qq.x - c.z * qq.y; v.y -= c.y * qq.y + c.z * qq.x;
        p[o] = pp;
        q[o] = qq;
        x[o] = xx;
        res[o] = v;
      }
      rs[k * n + r] = v;
    }
    if (!pnext) continue;
    __syncthreads();
    for (int i = threadIdx.x; i < ns * n; i += LTPB) {
      const int k = i / n, r = i - k * n;
      float ar = 0.f, ai = 0.f;
      for (int l = 0; l < ns; l++) little_mac(ar, ai, As[k * ns + l], rs[l * n + r]);
      pnext[((size_t)r * bg.nblk + blk) * ns + k] = make_float2(ar, ai);
    }
  }
}

}  // namespace

// ---------------------------------------------------------------------------
// Host side
// ---------------------------------------------------------------------------
struct DflState {
  int ns = 0, ready = 0;
  BlkGeom bg;
  DevBuf phi, A, Ainv, Af, Ainvf, Y, little, part, tmp, flags;
};

static DflState* dfl_of(qcd_ctx* c) {
  if (!c->dfl) c->dfl = new DflState();
  return (DflState*)c->dfl;
}

void dfl_free(qcd_ctx* c) {
  if (!c->dfl) return;
  DflState* d = (DflState*)c->dfl;
  devbuf_free(d->phi);
  devbuf_free(d->A);
  devbuf_free(d->Ainv);
  devbuf_free(d->Af);
  devbuf_free(d->Ainvf);
  devbuf_free(d->Y);
  devbuf_free(d->little);
  devbuf_free(d->part);
  devbuf_free(d->tmp);
  devbuf_free(d->flags);
  delete d;
  c->dfl = nullptr;
}

int dfl_ready(qcd_ctx* c) { return c->dfl && ((DflState*)c->dfl)->ready; }
int dfl_ns(qcd_ctx* c) { return c->dfl ? ((DflState*)c->dfl)->ns : 0; }
int dfl_nblk(qcd_ctx* c) { return c->dfl ? ((DflState*)c->dfl)->bg.nblk : 0; }
void* dfl_phi(qcd_ctx* c) { return c->dfl ? ((DflState*)c->dfl)->phi.p : nullptr; }
void* dfl_little(qcd_ctx* c) { return c->dfl ? ((DflState*)c->dfl)->A.p : nullptr; }

qcd_status solver_run(qcd_ctx* c, int n, const double* tol, qcd_rhs_stats* st);
qcd_status dfl_little_tc(qcd_ctx* c, const void* phi, const void* Y, double* A, const int b[4], int ns, int* err);

// Little operator (tensor cores, FP64 store) and diagonal-block inverses
// (FP64) from the current d->phi.
static qcd_status dfl_little_build(qcd_ctx* c) {
  DflState* d = dfl_of(c);
  const BlkGeom& bg = d->bg;
  const int ns = d->ns;
  const size_t fb = spinor_bytes(c, QCD_PREC_F32);
  QCD_TRY(devbuf_ensure(d->Y, 5 * fb * ns));
  QCD_TRY(devbuf_ensure(d->A, sizeof(double2) * (size_t)bg.nblk * 9 * ns * ns));
  QCD_TRY(devbuf_ensure(d->Ainv, sizeof(double2) * (size_t)bg.nblk * ns * ns));
  QCD_TRY(devbuf_ensure(d->flags, 2 * sizeof(int)));
  int* flags = (int*)d->flags.p;      // [0] singular diagonal block, [1] tensor-core wait timed out
  QCD_CUDA_OK(cudaMemsetAsync(flags, 0, 2 * sizeof(int), c->stream));
  {
    ProfScope ps(c, FAM_DFL, (double)c->g.V * ns * (96 + 5 * 96 + 192 + 288), (double)c->g.V * ns * 1824);
    dim3 grid((c->g.V + 127) / 128, ns);
    k_dfl_ypart<<<grid, 128, 0, c->stream>>>((const char*)d->phi.p, (char*)d->Y.p, c->gaugeF.p, c->cloverF.p, c->g, bg,
                                            (float)c->kappa, ns);
    QCD_CUDA_OK(cudaGetLastError());
  }
  QCD_TRY(dfl_little_tc(c, d->phi.p, d->Y.p, (double*)d->A.p, bg.b, ns, flags + 1));
  {
    ProfScope ps(c, FAM_DFL, 16.0 * bg.nblk * ns * ns * 2, 8.0 * bg.nblk * ns * ns * ns * 2);
    k_dfl_block_inverse<<<bg.nblk, 32, sizeof(double2) * ns * 2 * ns, c->stream>>>((const double2*)d->A.p,
                                                                                   (double2*)d->Ainv.p, ns, flags);
    QCD_CUDA_OK(cudaGetLastError());
    int h[2] = {0, 0};
    QCD_CUDA_OK(cudaMemcpyAsync(h, flags, sizeof(h), cudaMemcpyDeviceToHost, c->stream));
    QCD_CUDA_OK(cudaStreamSynchronize(c->stream));
    if (h[1]) {
      qcd_set_error("the tensor-core little Dirac build timed out waiting for its matrix multiplies");
      return QCD_ERR_TIMEOUT;
    }
    if (h[0]) {
      qcd_set_error("a diagonal block of the little Dirac operator is singular");
      return QCD_ERR_BREAKDOWN;
    }
  }
  {
    // FP32 copies for the little solve
    const size_t na = (size_t)bg.nblk * 9 * ns * ns, ni = (size_t)bg.nblk * ns * ns;
    QCD_TRY(devbuf_ensure(d->Af, sizeof(float2) * na));
    QCD_TRY(devbuf_ensure(d->Ainvf, sizeof(float2) * ni));
    ProfScope ps(c, FAM_DFL, 24.0 * (na + ni), 0.0, 2);
    k_little_transpose<<<1024, 256, 0, c->stream>>>((const double2*)d->A.p, (float2*)d->Af.p, ns, na);
    k_to_float2<<<1024, 256, 0, c->stream>>>((const double2*)d->Ainv.p, (float2*)d->Ainvf.p, ni);
    QCD_CUDA_OK(cudaGetLastError());
  }
  return QCD_OK;
}

// threads of a k_little_apply CTA: ns rows x rb RHS lanes, at most 256
static int little_threads(int ns, int n) {
  int rb = 256 / ns;
  if (rb > n) rb = n;
  if (rb < 1) rb = 1;
  return ns * rb;
}

// scratch of little_gcr in d->part: partial sums, dots, scalars
static size_t little_part_count(int n, int m) { return (size_t)n * (m + 2) * LITTLE_G; }
static size_t little_part_bytes(int n, int m) {
  if (n > LITTLE_RHS) n = LITTLE_RHS;
  return sizeof(double2) * (little_part_count(n, m) + (size_t)(m + 2) * n) + sizeof(float4) * n;
}

// little_gcr for at most LITTLE_RHS right-hand sides; vlen: distance of P's and Q's vectors
static qcd_status little_gcr_tile(qcd_ctx* c, DflState* d, float2* res, float2* xl, float2* P, float2* Q, size_t vlen,
                                  int n, int m) {
  const BlkGeom& bg = d->bg;
  const int ns = d->ns;
  const int N = bg.nblk * ns;
  double2* part = (double2*)d->part.p;
  double2* dots = part + little_part_count(n, m);
  float4* sc = (float4*)(dots + (size_t)(m + 2) * n);
  const int Gq = bg.nblk < LITTLE_G ? bg.nblk : LITTLE_G;
  // one element per thread of the orthogonalisation (its time is the latency of the
  // loads along j), at most LITTLE_G CTAs per RHS
  const int Go = (N + LTPB - 1) / LTPB < LITTLE_G ? (N + LTPB - 1) / LTPB : LITTLE_G;
  const size_t sm_s = sizeof(float2) * ((size_t)ns * n + (size_t)ns * ns);
  QCD_CUDA_OK(allow_smem(k_little_q, little_q_smem(MAX_NS, LITTLE_RHS, 64)));
  const float2* Ainv = (const float2*)d->Ainvf.p;
  const unsigned Gs = (unsigned)bg.nblk;
  const dim3 threads(LTPB);
  QCD_CUDA_OK(launch_after(c->stream, false, Gs, threads, sm_s, k_little_step, xl, res, nullptr, nullptr, P, Ainv, sc, 0,
                           1, bg, ns, n));
  for (int i = 0; i < m; i++) {
    float2* pi = P + vlen * i;
    float2* qi = Q + vlen * i;
    QCD_CUDA_OK(launch_after(c->stream, true, Gq, threads, little_q_smem(ns, n, i), k_little_q, (const float2*)d->Af.p, pi, qi, Q, vlen, i,
                             part, bg, ns, n));
    if (i > 0) QCD_CUDA_OK(launch_after(c->stream, true, dim3(i, n), 32, 0, k_little_sum, part, i, Gq, dots, n));
    QCD_CUDA_OK(launch_after(c->stream, true, dim3(Go, n), threads, 0, k_little_orth, qi, pi, Q, P, vlen, i, dots, res, N,
                             n, part));
    QCD_CUDA_OK(launch_after(c->stream, true, n, 32, 0, k_little_scalars, part, Go, sc));
    QCD_CUDA_OK(launch_after(c->stream, true, Gs, threads, sm_s, k_little_step, xl, res, pi, qi,
                             i + 1 < m ? pi + vlen : nullptr, Ainv, sc, i == 0, 0, bg, ns, n));
  }
  QCD_CUDA_OK(cudaGetLastError());
  return QCD_OK;
}

// m steps of block-Jacobi preconditioned GCR on the little vectors from x = 0:
// res holds the right-hand side on entry and the residual on exit, xl the
// approximate solution; P, Q: m (p, q) pairs of n little vectors each.  Every
// right-hand side is a problem of its own; they are taken LITTLE_RHS at a time.
static qcd_status little_gcr(qcd_ctx* c, DflState* d, float2* res, float2* xl, float2* P, float2* Q, int n, int m) {
  const size_t N = (size_t)d->bg.nblk * d->ns;
  for (int r0 = 0; r0 < n; r0 += LITTLE_RHS)
    QCD_TRY(little_gcr_tile(c, d, res + N * r0, xl + N * r0, P + N * r0, Q + N * r0, N * n,
                            n - r0 < LITTLE_RHS ? n - r0 : LITTLE_RHS, m));
  return QCD_OK;
}

static qcd_status dfl_gs(qcd_ctx* c) {
  DflState* d = dfl_of(c);
  const size_t fb = spinor_bytes(c, QCD_PREC_F32);
  ProfScope ps(c, FAM_DFL, 2.0 * fb * d->ns * d->ns / 2, 0.0);
  k_dfl_gs<<<d->bg.nblk, d->bg.vb, 0, c->stream>>>((char*)d->phi.p, c->g, d->bg, d->ns);
  QCD_CUDA_OK(cudaGetLastError());
  return QCD_OK;
}

// Build the subspace from the ns FP32 internal fields already in d->phi:
// block Gram-Schmidt; then n_inv rounds of inverse iteration, each followed
// by block Gram-Schmidt.  The approximate inverse of a round is M_SAP when
// gen_iters == 0; otherwise M_SAP for the first round and, once a little
// operator exists, gen_iters iterations of the deflated SAP-GCR solver (the
// subspace then improves the solver that refines it).
static qcd_status dfl_build(qcd_ctx* c, int n_inv, int gen_iters) {
  DflState* d = dfl_of(c);
  const int ns = d->ns;
  const size_t fb = spinor_bytes(c, QCD_PREC_F32);
  d->ready = 0;
  QCD_TRY(dfl_gs(c));
  for (int it = 0; it < n_inv; it++) {
    if (gen_iters > 0 && it > 0) {
      // solve D x = phi_l approximately with the deflated solver (fixed iteration count)
      const qcd_solver_params saved = c->params;
      c->params.max_outer = gen_iters;
      c->params.nkv = gen_iters < saved.nkv ? gen_iters : saved.nkv;
      c->params.restart_drop = 0.0;
      c->params.dfl = 1;
      c->params.precision = QCD_PREC_F32;
      const size_t bD = spinor_bytes(c, QCD_PREC_F64) * ns;
      qcd_status st = devbuf_ensure(c->wsD[0], bD);
      if (st == QCD_OK) st = devbuf_ensure(c->wsD[1], bD);
      if (st == QCD_OK) st = blas_convert(c, d->phi.p, QCD_PREC_F32, c->wsD[0].p, QCD_PREC_F64, ns, nullptr);
      if (st == QCD_OK && cudaMemsetAsync(c->wsD[1].p, 0, bD, c->stream) != cudaSuccess) st = QCD_ERR_CUDA;
      std::vector<double> tol(ns, 1e-14);
      std::vector<qcd_rhs_stats> rs(ns);
      if (st == QCD_OK) st = solver_run(c, ns, tol.data(), rs.data());
      c->params = saved;
      QCD_TRY(st);
      QCD_TRY(blas_convert(c, c->wsD[1].p, QCD_PREC_F64, d->phi.p, QCD_PREC_F32, ns, nullptr));
    } else {
      QCD_TRY(devbuf_ensure(d->tmp, 2 * fb * ns));
      char* rho = (char*)d->tmp.p;
      char* delta = rho + fb * ns;
      QCD_CUDA_OK(cudaMemcpyAsync(rho, d->phi.p, fb * ns, cudaMemcpyDeviceToDevice, c->stream));
      QCD_TRY(sap_apply(c, rho, d->phi.p, delta, QCD_PREC_F32, ns, nullptr, ns));
    }
    QCD_TRY(dfl_gs(c));
    if (gen_iters > 0 && it + 1 < n_inv) {
      QCD_TRY(dfl_little_build(c));
      d->ready = 1;
    }
  }
  QCD_TRY(dfl_little_build(c));
  d->ready = 1;
  return QCD_OK;
}

qcd_status dfl_setup(qcd_ctx* c, const double* init_dev, int ns, int n_inv) {
  DflState* d = dfl_of(c);
  d->ready = 0;
  d->ns = ns;
  d->bg = blk_geom(c);
  QCD_TRY(devbuf_ensure(d->phi, spinor_bytes(c, QCD_PREC_F32) * ns));
  QCD_TRY(layout_spinor_import(c, init_dev, d->phi.p, QCD_PREC_F32, ns));
  return dfl_build(c, n_inv, c->params.dfl_gen_iters);
}

// Low-mode part of the deflated preconditioner for n right-hand sides:
// x = Phi e with e = (little GCR, m steps) approx A^-1 Phi^+ rho.  rho and x
// are FP32 internal fields; masked RHS are skipped.
qcd_status dfl_low_mode(qcd_ctx* c, const void* rho, void* x, int n, const int* mask, int nactive, int m) {
  DflState* d = dfl_of(c);
  const BlkGeom& bg = d->bg;
  const int ns = d->ns;
  if (ns * n > 4 * GEMM_TPB) {
    qcd_set_error("deflation: ns x rhs tile = %d exceeds %d", ns * n, 4 * GEMM_TPB);
    return QCD_ERR_ARG;
  }
  const int N = bg.nblk * ns;                     // little vector length per rhs
  const size_t vlen = (size_t)N * n;              // float2 per little vector (all rhs)
  // little workspace: residual (the projection on entry), x, then m (p, q) pairs
  QCD_TRY(devbuf_ensure(d->little, sizeof(float2) * vlen * (2 + 2 * (size_t)m)));
  float2* res = (float2*)d->little.p;
  float2* xl = res + vlen;
  float2* P = xl + vlen;
  float2* Q = P + vlen * m;
  QCD_TRY(devbuf_ensure(d->part, little_part_bytes(n, m)));
  {
    ProfScope ps(c, FAM_DFL, (double)spinor_bytes(c, QCD_PREC_F32) * (ns + nactive), 8.0 * c->g.V * 12 * ns * nactive);
    for (int r0 = 0; r0 < n; r0 += LITTLE_RHS) {   // at most 64 tiles of outputs
      const int nr = n - r0 < LITTLE_RHS ? n - r0 : LITTLE_RHS;
      const ProjectShape sh = project_shape(ns, nr);
      QCD_CUDA_OK(allow_smem(k_dfl_project, project_shape(MAX_NS, LITTLE_RHS).smem));
      k_dfl_project<<<bg.nblk, GEMM_TPB, sh.smem, c->stream>>>(
          (const char*)d->phi.p, (const char*)rho + spinor_bytes(c, QCD_PREC_F32) * r0, res + (size_t)N * r0, c->g, bg,
          ns, nr, sh, mask ? mask + r0 : nullptr);
      QCD_CUDA_OK(cudaGetLastError());
    }
  }
  // little GCR with block-Jacobi preconditioning, x = 0 start, m steps
  {
    ProfScope ps(c, FAM_DFL, 8.0 * vlen * (6.0 + 3.0 * m) * m, 0.0, 5 * m);
    QCD_TRY(little_gcr(c, d, res, xl, P, Q, n, m));
  }
  {
    ProfScope ps(c, FAM_DFL, (double)spinor_bytes(c, QCD_PREC_F32) * (ns + nactive), 8.0 * c->g.V * 12 * ns * nactive);
    k_dfl_prolong<<<6 / PRW * bg.nblk, bg.vb < 256 ? bg.vb : 256,
                    sizeof(float2) * ns * ((n + PRG - 1) / PRG * PRG), c->stream>>>((const char*)d->phi.p, xl, (char*)x,
                                                                                    c->g, bg, ns, n, mask);
    QCD_CUDA_OK(cudaGetLastError());
  }
  return QCD_OK;
}

// Little-vector entry points for the tests: y = A x (apply = 0) or the
// m-step little solve x = approx A^-1 y (apply = 1); vectors host FP64 complex
// [n][nblk][ns].
qcd_status dfl_little_host(qcd_ctx* c, const double* in, double* out, int n, int mode, int m) {
  DflState* d = dfl_of(c);
  const int N = d->bg.nblk * d->ns;
  const size_t vlen = (size_t)N * n;
  std::vector<float2> h(vlen);
  for (size_t i = 0; i < vlen; i++) h[i] = make_float2((float)in[2 * i], (float)in[2 * i + 1]);
  QCD_TRY(devbuf_ensure(d->tmp, sizeof(float2) * vlen * 2));
  float2* x = (float2*)d->tmp.p;
  float2* y = x + vlen;
  QCD_CUDA_OK(cudaMemcpyAsync(x, h.data(), sizeof(float2) * vlen, cudaMemcpyHostToDevice, c->stream));
  if (mode == 0) {
    k_little_apply<<<d->bg.nblk, little_threads(d->ns, n), 0, c->stream>>>((const double2*)d->A.p, x, y, d->bg, d->ns, n);
  } else {
    // the solver on little vectors, without projection and prolongation
    QCD_TRY(devbuf_ensure(d->little, sizeof(float2) * vlen * (2 + 2 * (size_t)m)));
    QCD_TRY(devbuf_ensure(d->part, little_part_bytes(n, m)));
    float2* res = (float2*)d->little.p;
    float2* xl = res + vlen;
    float2* P = xl + vlen;
    float2* Q = P + vlen * m;
    QCD_CUDA_OK(cudaMemcpyAsync(res, x, sizeof(float2) * vlen, cudaMemcpyDeviceToDevice, c->stream));
    QCD_TRY(little_gcr(c, d, res, xl, P, Q, n, m));
    QCD_CUDA_OK(cudaMemcpyAsync(y, xl, sizeof(float2) * vlen, cudaMemcpyDeviceToDevice, c->stream));
  }
  QCD_CUDA_OK(cudaGetLastError());
  QCD_CUDA_OK(cudaMemcpyAsync(h.data(), y, sizeof(float2) * vlen, cudaMemcpyDeviceToHost, c->stream));
  QCD_CUDA_OK(cudaStreamSynchronize(c->stream));
  for (size_t i = 0; i < vlen; i++) {
    out[2 * i] = h[i].x;
    out[2 * i + 1] = h[i].y;
  }
  return QCD_OK;
}

// For the tests (not part of qcd.h): q = A p and the dots of q with nj vectors, as a little
// GCR step computes them; n <= 24 right-hand sides, nj <= 64.  Device memory: p, q
// [n][nblk][ns], qj [nj] such vectors, dots [nj][n].
extern "C" qcd_status qcd_test_little_dots(qcd_ctx* c, const float2* p, const float2* qj, int nj, int n, float2* q,
                                           double2* dots) {
  DflState* d = dfl_of(c);
  if (!d->ready || n < 1 || n > LITTLE_RHS || nj < 1 || nj > 64) return QCD_ERR_ARG;
  QCD_TRY(devbuf_ensure(d->part, little_part_bytes(n, nj)));
  double2* part = (double2*)d->part.p;
  const int ns = d->ns, Gq = d->bg.nblk < LITTLE_G ? d->bg.nblk : LITTLE_G;
  QCD_CUDA_OK(allow_smem(k_little_q, little_q_smem(MAX_NS, LITTLE_RHS, 64)));
  k_little_q<<<Gq, LTPB, little_q_smem(ns, n, nj), c->stream>>>((const float2*)d->Af.p, p, q, qj,
                                                                (size_t)d->bg.nblk * ns * n, nj, part, d->bg, ns, n);
  k_little_sum<<<dim3(nj, n), 32, 0, c->stream>>>(part, nj, Gq, dots, n);
  QCD_CUDA_OK(cudaGetLastError());
  QCD_CUDA_OK(cudaStreamSynchronize(c->stream));
  return QCD_OK;
}
