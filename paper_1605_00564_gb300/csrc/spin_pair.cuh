// FP32 spinor arithmetic on pairs of spins.
//
// sm_103a has two-lane FP32 instructions (fma.rn.f32x2): one issue slot for two
// fused multiply-adds.  The rate of the FP32 pipe is the same (measured 78.5
// against 77.1 TFLOP/s of scalar FFMA), but the issue slots that scalar
// multiply-adds took are free for the shared-memory loads and conversions of
// the stencil kernels, which were issue-bound.
//
// The two lanes are the two spins of one chirality, (0, 1) or (2, 3): an SU(3)
// entry multiplies both alike, the projections (1 -+ gamma_mu) and their
// reconstructions act on a pair by at most an exchange of its lanes and a sign
// per lane, and so does the clover term.  Exchanges, negations and broadcasts
// of an operand cost nothing (they are part of the instruction), so every
// multiply-add of the operator is a two-lane one with one right-hand side and
// one site per thread.
//
// A spinor is a PairSpinor: re[c][a], im[c][a] for chirality c and colour a.
// In shared memory it is six 16-byte records q = 3 c + a: (re0, re1, im0, im1).
#pragma once

#include "qcd_internal.cuh"

struct PairSpinor {
  float2 re[2][3], im[2][3];
};

__device__ __forceinline__ float2 p2(float a, float b) { return make_float2(a, b); }
__device__ __forceinline__ float2 pbc(float a) { return make_float2(a, a); }            // broadcast
__device__ __forceinline__ float2 psw(float2 a) { return make_float2(a.y, a.x); }       // exchange of the spins
__device__ __forceinline__ float2 pneg(float2 a) { return make_float2(-a.x, -a.y); }
__device__ __forceinline__ float2 pfma(float2 a, float2 b, float2 c) { return __ffma2_rn(a, b, c); }
__device__ __forceinline__ float2 pmul(float2 a, float2 b) { return __fmul2_rn(a, b); }

// h = up + SIGN e_mu dn for one colour (the (1 + SIGN gamma_mu) projection; the
// matrices e_mu are those of project<> in qcd_internal.cuh)
template <int MU, int SIGN>
__device__ __forceinline__ void pair_project(float2 ur, float2 ui, float2 dr, float2 di, float2& hr, float2& hi) {
  constexpr float S = (float)SIGN;
  if (MU == 0) { hr = pfma(dr, pbc(-S), ur); hi = pfma(di, pbc(-S), ui); }
  if (MU == 1) { hr = pfma(psw(di), pbc(S), ur); hi = pfma(psw(dr), pbc(-S), ui); }
  if (MU == 2) { hr = pfma(psw(dr), p2(-S, S), ur); hi = pfma(psw(di), p2(-S, S), ui); }
  if (MU == 3) { hr = pfma(di, p2(S, -S), ur); hi = pfma(dr, p2(-S, S), ui); }
}

// out += s (1 + SIGN gamma_mu)-reconstruction of h for one colour a
template <int MU, int SIGN>
__device__ __forceinline__ void pair_recon(PairSpinor& o, int a, float2 hr, float2 hi, float s) {
  o.re[0][a] = pfma(hr, pbc(s), o.re[0][a]);
  o.im[0][a] = pfma(hi, pbc(s), o.im[0][a]);
  const float t = SIGN < 0 ? -s : s;
  if (MU == 0) { o.re[1][a] = pfma(hr, pbc(-t), o.re[1][a]); o.im[1][a] = pfma(hi, pbc(-t), o.im[1][a]); }
  if (MU == 1) { o.re[1][a] = pfma(psw(hi), pbc(-t), o.re[1][a]); o.im[1][a] = pfma(psw(hr), pbc(t), o.im[1][a]); }
  if (MU == 2) { o.re[1][a] = pfma(psw(hr), p2(t, -t), o.re[1][a]); o.im[1][a] = pfma(psw(hi), p2(t, -t), o.im[1][a]); }
  if (MU == 3) { o.re[1][a] = pfma(hi, p2(-t, t), o.re[1][a]); o.im[1][a] = pfma(hr, p2(t, -t), o.im[1][a]); }
}

// (g, per colour) = U h with h the (1 + SIGN gamma_mu) projection of the
// neighbour's spinor (DAG: U^+ h); rec(q) returns its record q, link(k) entry
// k = 3 row + column of U as (re, im); row(a, re, im) receives colour a.
template <int MU, int SIGN, bool DAG, typename Rec, typename Link, typename Row>
__device__ __forceinline__ void pair_project_mul(Rec rec, Link link, Row row) {
  float2 hr[3], hi[3];
#pragma unroll
  for (int b = 0; b < 3; b++) {
    const float4 u = rec(b), d = rec(3 + b);
    pair_project<MU, SIGN>(p2(u.x, u.y), p2(u.z, u.w), p2(d.x, d.y), p2(d.z, d.w), hr[b], hi[b]);
  }
#pragma unroll
  for (int a = 0; a < 3; a++) {
    float2 gr, gi;
#pragma unroll
    for (int b = 0; b < 3; b++) {
      const float2 u = DAG ? link(3 * b + a) : link(3 * a + b);
      const float ui = DAG ? -u.y : u.y;
      if (b == 0) {
        gr = pmul(pbc(u.x), hr[b]);
        gi = pmul(pbc(u.x), hi[b]);
      } else {
        gr = pfma(pbc(u.x), hr[b], gr);
        gi = pfma(pbc(u.x), hi[b], gi);
      }
      gr = pfma(pbc(-ui), hi[b], gr);
      gi = pfma(pbc(ui), hr[b], gi);
    }
    row(a, gr, gi);
  }
}

// One hop: o += s (1 + SIGN gamma_mu) U psi (DAG: U^+ psi)
template <int MU, int SIGN, bool DAG, typename Rec, typename Link>
__device__ __forceinline__ void pair_hop(PairSpinor& o, Rec rec, Link link, float s) {
  pair_project_mul<MU, SIGN, DAG>(rec, link,
                                  [&](int a, float2 gr, float2 gi) { pair_recon<MU, SIGN>(o, a, gr, gi, s); });
}

// The full matrix of an FP32 link stored as its first two rows (three float4),
// the third the conjugate of their cross product
struct LinkRows {
  float2 m[9];
};
__device__ __forceinline__ LinkRows link_rows(float4 a, float4 b, float4 c) {
  LinkRows u;
  u.m[0] = p2(a.x, a.y); u.m[1] = p2(a.z, a.w); u.m[2] = p2(b.x, b.y);
  u.m[3] = p2(b.z, b.w); u.m[4] = p2(c.x, c.y); u.m[5] = p2(c.z, c.w);
#pragma unroll
  for (int k = 0; k < 3; k++) {
    const float2 p = u.m[(k + 1) % 3], q = u.m[3 + (k + 2) % 3], r = u.m[(k + 2) % 3], t = u.m[3 + (k + 1) % 3];
    u.m[6 + k] = p2((p.x * q.x - p.y * q.y) - (r.x * t.x - r.y * t.y),
                    -((p.x * q.y + p.y * q.x) - (r.x * t.y + r.y * t.x)));
  }
  return u;
}

// The packed Hermitian 6x6 block of one chirality, [[A0, E^+], [E, A1]] over
// (spin, colour), arranged for pairs: d the diagonals of (A0, A1); for the
// colour pairs m = (1,0), (2,0), (2,1) the entries l = (A0[a][b], A1[a][b]) and
// o = (conj E[a][b], E[b][a]); e the diagonal of E.
struct CloverPairs {
  float2 d[3], lr[3], li[3], e[3], orr[3], oi[3];
};

// o = block * v for chirality c
__device__ __forceinline__ void pair_clover_block(const CloverPairs& m, int c, const PairSpinor& v, PairSpinor& o) {
#pragma unroll
  for (int a = 0; a < 3; a++) {
    o.re[c][a] = pmul(m.d[a], v.re[c][a]);
    o.im[c][a] = pmul(m.d[a], v.im[c][a]);
    // E[a][a] between the spins: lane 0 takes its conjugate
    const float2 sr = psw(v.re[c][a]), si = psw(v.im[c][a]), ei = p2(-m.e[a].y, m.e[a].y);
    o.re[c][a] = pfma(pbc(m.e[a].x), sr, o.re[c][a]);
    o.re[c][a] = pfma(pneg(ei), si, o.re[c][a]);
    o.im[c][a] = pfma(pbc(m.e[a].x), si, o.im[c][a]);
    o.im[c][a] = pfma(ei, sr, o.im[c][a]);
  }
#pragma unroll
  for (int k = 0; k < 3; k++) {
    const int a = k == 0 ? 1 : 2, b = k == 2 ? 1 : 0;   // a > b
    // same spin: o_a += l v_b, o_b += conj(l) v_a
    o.re[c][a] = pfma(m.lr[k], v.re[c][b], o.re[c][a]);
    o.re[c][a] = pfma(pneg(m.li[k]), v.im[c][b], o.re[c][a]);
    o.im[c][a] = pfma(m.lr[k], v.im[c][b], o.im[c][a]);
    o.im[c][a] = pfma(m.li[k], v.re[c][b], o.im[c][a]);
    o.re[c][b] = pfma(m.lr[k], v.re[c][a], o.re[c][b]);
    o.re[c][b] = pfma(m.li[k], v.im[c][a], o.re[c][b]);
    o.im[c][b] = pfma(m.lr[k], v.im[c][a], o.im[c][b]);
    o.im[c][b] = pfma(pneg(m.li[k]), v.re[c][a], o.im[c][b]);
    // other spin: o_b += o v_a with the spins of v exchanged, and o_a += its
    // Hermitian counterpart (exchanged, imaginary part negated)
    o.re[c][b] = pfma(m.orr[k], psw(v.re[c][a]), o.re[c][b]);
    o.re[c][b] = pfma(pneg(m.oi[k]), psw(v.im[c][a]), o.re[c][b]);
    o.im[c][b] = pfma(m.orr[k], psw(v.im[c][a]), o.im[c][b]);
    o.im[c][b] = pfma(m.oi[k], psw(v.re[c][a]), o.im[c][b]);
    o.re[c][a] = pfma(psw(m.orr[k]), psw(v.re[c][b]), o.re[c][a]);
    o.re[c][a] = pfma(psw(m.oi[k]), psw(v.im[c][b]), o.re[c][a]);
    o.im[c][a] = pfma(psw(m.orr[k]), psw(v.im[c][b]), o.im[c][a]);
    o.im[c][a] = pfma(pneg(psw(m.oi[k])), psw(v.re[c][b]), o.im[c][a]);
  }
}

// Arrange 18 words w(j) = reals (2j, 2j + 1) of a packed block: words 0..2 are
// the diagonal, word 3 + i (i - 1) / 2 + j is entry (i, j).
template <typename W>
__device__ __forceinline__ CloverPairs clover_pairs(W w) {
  CloverPairs m;
  const float2 d0 = w(0), d1 = w(1), d2 = w(2);
  m.d[0] = p2(d0.x, d1.y);
  m.d[1] = p2(d0.y, d2.x);
  m.d[2] = p2(d1.x, d2.y);
  const int l0[3] = {3, 4, 5}, l1[3] = {12, 16, 17};          // A0 and A1 entries (1,0), (2,0), (2,1)
  const int eab[3] = {9, 13, 14}, eba[3] = {7, 8, 11};        // E[a][b], E[b][a] of the same pairs
  const int ed[3] = {6, 10, 15};                              // E[a][a]
#pragma unroll
  for (int k = 0; k < 3; k++) {
    const float2 x = w(l0[k]), y = w(l1[k]);
    m.lr[k] = p2(x.x, y.x);
    m.li[k] = p2(x.y, y.y);
    const float2 u = w(eab[k]), v = w(eba[k]);
    m.orr[k] = p2(u.x, v.x);
    m.oi[k] = p2(-u.y, v.y);
    m.e[k] = w(ed[k]);
  }
  return m;
}

// FP32 global layout (float4 [6][V], components 2k, 2k + 1) <-> pairs
__device__ __forceinline__ PairSpinor pair_from_words(const float4 (&w)[6]) {
  float re[12], im[12];
#pragma unroll
  for (int k = 0; k < 6; k++) {
    re[2 * k] = w[k].x; im[2 * k] = w[k].y; re[2 * k + 1] = w[k].z; im[2 * k + 1] = w[k].w;
  }
  PairSpinor o;
#pragma unroll
  for (int c = 0; c < 2; c++)
#pragma unroll
    for (int a = 0; a < 3; a++) {
      o.re[c][a] = p2(re[6 * c + a], re[6 * c + 3 + a]);
      o.im[c][a] = p2(im[6 * c + a], im[6 * c + 3 + a]);
    }
  return o;
}
__device__ __forceinline__ void load_words(const void* base, int V, int s, float4 (&w)[6]) {
  const float4* p = (const float4*)base;
#pragma unroll
  for (int k = 0; k < 6; k++) w[k] = __ldg(p + (size_t)k * V + s);
}
__device__ __forceinline__ PairSpinor pair_load(const void* base, int V, int s) {
  float4 w[6];
  load_words(base, V, s, w);
  return pair_from_words(w);
}
__device__ __forceinline__ void pair_store(void* base, int V, int s, const PairSpinor& o) {
  float4* p = (float4*)base;
  float re[12], im[12];
#pragma unroll
  for (int c = 0; c < 2; c++)
#pragma unroll
    for (int a = 0; a < 3; a++) {
      re[6 * c + a] = o.re[c][a].x; re[6 * c + 3 + a] = o.re[c][a].y;
      im[6 * c + a] = o.im[c][a].x; im[6 * c + 3 + a] = o.im[c][a].y;
    }
#pragma unroll
  for (int k = 0; k < 6; k++) p[(size_t)k * V + s] = make_float4(re[2 * k], im[2 * k], re[2 * k + 1], im[2 * k + 1]);
}

__device__ __forceinline__ void pair_add(PairSpinor& y, const PairSpinor& x) {
#pragma unroll
  for (int c = 0; c < 2; c++)
#pragma unroll
    for (int a = 0; a < 3; a++) {
      y.re[c][a] = __fadd2_rn(y.re[c][a], x.re[c][a]);
      y.im[c][a] = __fadd2_rn(y.im[c][a], x.im[c][a]);
    }
}

// record q = 3 c + a of a spinor held in registers
__device__ __forceinline__ float4 pair_rec(const PairSpinor& v, int q) {
  const int c = q / 3, a = q % 3;
  return make_float4(v.re[c][a].x, v.re[c][a].y, v.im[c][a].x, v.im[c][a].y);
}
