// Both operators in FP64 with four lanes of a warp sharing a site.
//
// The FP64 pipe takes 64 clocks of its scheduler for a warp's instruction, so
// one thread per site (about 900 FP64 instructions) needs 27 us for a lattice
// of any size, and several warps per scheduler to balance.  Four lanes a site
// cut that chain to about 220 and spread a small lattice over four times as
// many warps.  Lane q takes direction q of the hops (staggered Wilson: and the
// corners +-s_2q, +-s_(2q+1)); the lanes then add up so that each ends with
// its share of the result.  Everything that differs between the lanes is a
// selection or a sign flip (integer instructions), never a branch: a branch
// would run the FP64 pipe once per side.
//
// The share of lane q, `kOwn` real numbers: Wilson: spin q (3 complex
// numbers); staggered Wilson: real (q & 2 == 0) or imaginary parts, of
// components 0 and 2 (q even) or 1 (q odd; its second number is none).
#pragma once
#include "dslash.cuh"

namespace swc {

__device__ __forceinline__ double flip_if(bool neg, double v) {
  return __hiloint2double(__double2hiint(v) ^ (neg ? 0x80000000 : 0), __double2loint(v));
}
__device__ __forceinline__ cx<double> flip_if(bool neg, cx<double> v) { return {flip_if(neg, v.re), flip_if(neg, v.im)}; }
__device__ __forceinline__ cx<double> pick(bool a, cx<double> x, cx<double> y) { return {a ? x.re : y.re, a ? x.im : y.im}; }
// i v if `im`, else v
__device__ __forceinline__ cx<double> turn_if(bool im, cx<double> v) { return {im ? -v.im : v.re, im ? v.re : v.im}; }
// a + b (send, kept across lane ^ mask): what the partner sent is added to what this lane keeps
__device__ __forceinline__ double take(double keep, double send, int mask) {
  return keep + __shfl_xor_sync(0xffffffffu, send, mask);
}

// Wilson: the hops of direction mu = q; o: the 3 components of spin q of
// sum_mu [(r - c g_mu) U psi(x+mu) + (r + c g_mu) U^+ psi(x-mu)], c = -1 for the adjoint.
// With uf, ub the transported rows, the upper spins take S = uf + ub and the
// lower ones the phase of D = uf - ub = 2 uf - S: S continues uf's chain of
// FMAs, so the two sums cost one FMA where they cost two additions each.
template <bool R1, typename G, typename In>
__device__ __forceinline__ void wilson_quad(const Geom& g, int n, int q, const G& U, const In& in, double r, bool dag,
                                            cx<double> o[3]) {
  int x[4];
  coords(g, n, x);
  const int s = q == 0 ? g.stride[0] : q == 1 ? g.stride[1] : q == 2 ? g.stride[2] : g.stride[3];
  const int L = q == 0 ? g.L[0] : q == 1 ? g.L[1] : q == 2 ? g.L[2] : g.L[3];
  const int xq = q == 0 ? x[0] : q == 1 ? x[1] : q == 2 ? x[2] : x[3];
  const int nf = xq == L - 1 ? n - (L - 1) * s : n + s, nb = xq == 0 ? n + (L - 1) * s : n - s;
  const bool ff = q == 3 && g.apbc && xq == L - 1, fb = q == 3 && g.apbc && xq == 0;
  const bool im = q == 0 || q == 2;  // gamma_q's blocks are imaginary
  const bool sw = q < 2;             // and couple spins (0,3), (1,2); else (0,2), (1,3)
  cx<double> lo[4][3];               // contributions to the four spins
  const M3<double> Uf = U.link(n, q), Ub = U.link(nb, q);
  if constexpr (R1) {
    // rows of (1 - c' g_q) psi: a0 - c' k0 (i) b0, a1 - c' k1 (i) b1 with (b0, b1) = (3, 2) or (2, 3) and
    // (k0, k1) = (1, 1), (-1, 1), (1, -1), (1, 1)
    V3<double> h0, h1, u0, u1;
    auto project = [&](int y, bool neg) {  // c' = -1 if neg
      const Sp<double> p = ld_sp<In, double>(in, y);
#pragma unroll
      for (int i = 0; i < 3; ++i) {
        const cx<double> b0 = turn_if(im, pick(sw, p.s[3].c[i], p.s[2].c[i]));
        const cx<double> b1 = turn_if(im, pick(sw, p.s[2].c[i], p.s[3].c[i]));
        h0.c[i] = p.s[0].c[i] + flip_if(neg == (q == 1), b0);
        h1.c[i] = p.s[1].c[i] + flip_if(neg == (q == 2), b1);
      }
    };
    // flip_if's argument: a0 - c' k0 b0 has a minus for c' k0 = 1, that is for (neg, k0 = -1) equal
    project(nf, dag);
    u0 = mv(Uf, h0);
    u1 = mv(Uf, h1);
    // boundary signs ride on the vectors: backward relative to forward
    V3<double> s0, s1;
#pragma unroll
    for (int i = 0; i < 3; ++i) {
      u0.c[i] = flip_if(ff, u0.c[i]);
      u1.c[i] = flip_if(ff, u1.c[i]);
      s0.c[i] = u0.c[i];
      s1.c[i] = u1.c[i];
    }
    project(nb, !dag);
#pragma unroll
    for (int i = 0; i < 3; ++i) {
      h0.c[i] = flip_if(fb, h0.c[i]);
      h1.c[i] = flip_if(fb, h1.c[i]);
    }
    mdv_acc(s0, Ub, h0, 1.0);
    mdv_acc(s1, Ub, h1, 1.0);
    // lower spins: c k' (i) D with (D for spin 2, spin 3) = (D1, D0) or (D0, D1), the signs of
    // (2, 3): (+,+), (-,+), (+,-), (-,-) times c
#pragma unroll
    for (int i = 0; i < 3; ++i) {
      const cx<double> d0 = {fma(2.0, u0.c[i].re, -s0.c[i].re), fma(2.0, u0.c[i].im, -s0.c[i].im)};
      const cx<double> d1 = {fma(2.0, u1.c[i].re, -s1.c[i].re), fma(2.0, u1.c[i].im, -s1.c[i].im)};
      lo[0][i] = s0.c[i];
      lo[1][i] = s1.c[i];
      lo[2][i] = flip_if(dag != (q == 1 || q == 3), turn_if(im, pick(sw, d1, d0)));
      lo[3][i] = flip_if(dag != (q == 2 || q == 3), turn_if(im, pick(sw, d0, d1)));
    }
  } else {
    const Sp<double> pf = ld_sp<In, double>(in, nf), pb = ld_sp<In, double>(in, nb);
    cx<double> d[4][3];
#pragma unroll
    for (int k = 0; k < 4; ++k) {
      V3<double> u = mv(Uf, pf.s[k]), hb = pb.s[k], sm;
#pragma unroll
      for (int i = 0; i < 3; ++i) {
        u.c[i] = flip_if(ff, u.c[i]);
        sm.c[i] = u.c[i];
        hb.c[i] = flip_if(fb, hb.c[i]);
      }
      mdv_acc(sm, Ub, hb, 1.0);
#pragma unroll
      for (int i = 0; i < 3; ++i) {
        lo[k][i] = r * sm.c[i];
        d[k][i] = {fma(2.0, u.c[i].re, -sm.c[i].re), fma(2.0, u.c[i].im, -sm.c[i].im)};
      }
    }
    // - c g_q D: g_q D = (i)(k0 b0, k1 b1) in the upper spins, the adjoint block in the lower
#pragma unroll
    for (int i = 0; i < 3; ++i) {
      const cx<double> u0 = turn_if(im, pick(sw, d[3][i], d[2][i])), u1 = turn_if(im, pick(sw, d[2][i], d[3][i]));
      const cx<double> l2 = turn_if(im, pick(sw, d[1][i], d[0][i])), l3 = turn_if(im, pick(sw, d[0][i], d[1][i]));
      lo[0][i] = lo[0][i] + flip_if(dag == (q == 1), u0);
      lo[1][i] = lo[1][i] + flip_if(dag == (q == 2), u1);
      lo[2][i] = lo[2][i] + flip_if(dag != (q == 1 || q == 3), l2);
      lo[3][i] = lo[3][i] + flip_if(dag != (q == 2 || q == 3), l3);
    }
  }
  const bool hi = q & 2, odd = q & 1;
#pragma unroll
  for (int i = 0; i < 3; ++i) {
    cx<double> k[2];
#pragma unroll
    for (int j = 0; j < 2; ++j) {
      const cx<double> keep = pick(hi, lo[2 + j][i], lo[j][i]), send = pick(hi, lo[j][i], lo[2 + j][i]);
      k[j] = {take(keep.re, send.re, 2), take(keep.im, send.im, 2)};
    }
    const cx<double> keep = pick(odd, k[1], k[0]), send = pick(odd, k[0], k[1]);
    o[i] = {take(keep.re, send.re, 1), take(keep.im, send.im, 1)};
  }
}

// staggered Wilson: this lane's part (real: q & 2 == 0) of the three components of D psi without the site's own term
template <typename G, typename Wt, typename In>
__device__ __forceinline__ void sw_quad(const Geom& g, int n, int q, const G& U, const Wt& W, const In& in, double r,
                                        bool dag, double o[3]) {
  int x[4], df[4], db[4];
  coords(g, n, x);
  hop_deltas(g, n, x, df, db);
  const bool ff = bc_flip(g, x, +1), fb = bc_flip(g, x, -1);
  const int dfq = q == 0 ? df[0] : q == 1 ? df[1] : q == 2 ? df[2] : df[3];
  const int dbq = q == 0 ? db[0] : q == 1 ? db[1] : q == 2 ? db[2] : db[3];
  const int par = (q > 0 ? x[0] : 0) + (q > 1 ? x[1] : 0) + (q > 2 ? x[2] : 0);
  auto ldf = [&](int y, bool neg) {
    V3<double> v = ld3<In, double>(in, y);
#pragma unroll
    for (int i = 0; i < 3; ++i) v.c[i] = flip_if(neg, v.c[i]);
    return v;
  };
  V3<double> d = zero3<double>(), h = zero3<double>();
  const bool eta = par & 1;
  mv_acc(d, U.link(n, q), ldf(n + dfq, (q == 3 && ff) != eta));
  mdv_acc(d, U.link(n + dbq, q), ldf(n + dbq, (q == 3 && fb) == eta), 1.0);
#pragma unroll
  for (int j = 0; j < 2; ++j) {
    int of, ob;
    corner_offsets(2 * q + j, df, db, of, ob);
    mv_acc(h, W.mat(n, 2 * q + j), ldf(n + of, ff));
    mdv_acc(h, W.mat(n + ob, 2 * q + j), ldf(n + ob, fb), 1.0);
  }
  const double hs = (eps_eta5_neg(x) ? r : -r) * 0.0625, ss = dag ? -0.5 : 0.5;
  const bool imag = q & 2;
#pragma unroll
  for (int i = 0; i < 3; ++i) {
    const double re = fma(ss, d.c[i].re, hs * h.c[i].re), im = fma(ss, d.c[i].im, hs * h.c[i].im);
    o[i] = take(imag ? im : re, imag ? re : im, 2);
    o[i] += __shfl_xor_sync(0xffffffffu, o[i], 1);
  }
}

}  // namespace swc
