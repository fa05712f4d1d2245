// mg_me64l.cuh -- the FP64 helicity sum of 3 to 5 gluons in a basis of linear gluon polarisations.
//
// The amplitude is linear in each gluon's polarisation vector, and the two helicity vectors are a unitary combination of
// the two real transverse vectors e_theta, e_phi: summed over both, |M|^2 is the same.  With real polarisations every
// gluon current is real (the vertices and propagators are), which makes the three-gluon vertex 30 FP64 instructions
// instead of 80, the four-gluon vertex 13 (products of currents tabulated) instead of 102, and a quark current times a gluon current 8 instead of 16;
// and flipping both top helicities conjugates the amplitude, so top helicity -1 with both antitop helicities is enough.
// So where every helicity is good (always, from 3 gluons on, at the default threshold) and only the sum is asked for,
// mg_me64.cuh's scheme runs in this basis: 2^K polarisation combinations x 2 antitop helicities, as many as there are
// helicities there.  With J real, psi . (gamma.J) v = (psi gamma^mu v) . J costs 8, so the quark line's terms become
//     A = (u g v).J(1..K) + (u g chi_K).J(1..K-1) + sum over prefixes of i = 1 .. K-3 gluons of
//         [ (psi_i g v).J(i+1..K) + (psi_i g chi_K).J(i+1..K-1) ] + psi_{K-2} . Z(s_{K-1}, s_K)
// with the bilinears tabulated, except (psi_2 g chi_K) of 5 gluons, whose 480 bilinears per event would cost more than
// they save (there psi_2 . (gamma.J) chi_K).  The record's polarisation vectors are e / sqrt 2, which the final factor
// 2^K undoes; the other factor 2 is the flip.
//
// Measured against the helicity basis: gg->ttg 9.47 vs 12.05 ms per 524,288 events, gg->ttgg 1.87 vs 2.64 ms per 10,007,
// gg->ttggg 21.5 vs 31.7 ms per 8,192; with the all-gluon currents formed only in their contraction with the quark
// current (ViewL::full) and the products of currents tabulated for the four-gluon vertices 8.98, 1.63 and 17.8 ms.
#pragma once

#include "mg_me64.cuh"

namespace mg {
namespace m64 {

// doubles of one combination's own items (LOCAL)
template <int K> struct LocL;
template <> struct LocL<3> { static constexpr int n = 331; };
template <> struct LocL<4> { static constexpr int n = 1100; };
template <> struct LocL<5> { static constexpr int n = 3600; };

__device__ __forceinline__ double rdot(const double* a, const double* b) {
  return fma(-a[3], b[3], fma(-a[2], b[2], fma(-a[1], b[1], a[0] * b[0])));
}
__device__ __forceinline__ cx<double> qdot(const cx<double>* q, const double* j) {   // complex . real
  cx<double> r = {q[0].r * j[0], q[0].i * j[0]};
#pragma unroll
  for (int m = 1; m < 4; ++m) {
    r.r = fma(-q[m].r, j[m], r.r);
    r.i = fma(-q[m].i, j[m], r.i);
  }
  return r;
}

// v3_acc on real currents
__device__ __forceinline__ void v3r_acc(double* acc, const double* JL, const double* JR, const double* PL, const double* PR,
                                        bool neg) {
  double jj = rdot(JL, JR);
  if (neg) jj = -jj;
  const double two = neg ? -2.0 : 2.0, cl = two * rdot(JL, PR), cr = two * rdot(JR, PL);
#pragma unroll
  for (int m = 0; m < 4; ++m) acc[m] = fma(-cr, JL[m], fma(cl, JR[m], fma(PL[m] - PR[m], jj, acc[m])));
}

// gamma.J of a real current: a = J0 + J3, b = J0 - J3, and J1 -+ i J2
struct RSlash { double a, b, x, y; };
__device__ __forceinline__ RSlash rslash(const double* J, bool neg) {
  RSlash g = {J[0] + J[3], J[0] - J[3], J[1], J[2]};
  if (neg) g = {-g.a, -g.b, -g.x, -g.y};
  return g;
}
__device__ __forceinline__ void cmacp(cx<double>& c, cx<double> s, double x, double y) {   // c += s (x + i y)
  c.r = fma(s.r, x, c.r); c.r = fma(-s.i, y, c.r);
  c.i = fma(s.i, x, c.i); c.i = fma(s.r, y, c.i);
}
// acc += s g (row spinor) and o += g v (column spinor), as row_slash_acc and col_slash_acc
__device__ __forceinline__ void row_rslash_acc(cx<double>* acc, const cx<double>* s, const RSlash& g) {
  v2::cmacr(acc[0], g.a, s[2]); cmacp(acc[0], s[3], g.x, g.y);
  cmacp(acc[1], s[2], g.x, -g.y); v2::cmacr(acc[1], g.b, s[3]);
  v2::cmacr(acc[2], g.b, s[0]); cmacp(acc[2], s[1], -g.x, -g.y);
  v2::cmacr(acc[3], g.a, s[1]); cmacp(acc[3], s[0], -g.x, g.y);
}
__device__ __forceinline__ void col_rslash_acc(cx<double>* o, const RSlash& g, const cx<double>* v) {
  v2::cmacr(o[0], g.b, v[2]); cmacp(o[0], v[3], -g.x, g.y);
  v2::cmacr(o[1], g.a, v[3]); cmacp(o[1], v[2], -g.x, -g.y);
  v2::cmacr(o[2], g.a, v[0]); cmacp(o[2], v[1], g.x, -g.y);
  cmacp(o[3], v[0], g.x, g.y); v2::cmacr(o[3], g.b, v[1]);
}

// The items of one event for the polarisations gc (bit g: e_phi instead of e_theta), stored as View's.
template <int K, bool LOCAL>
struct ViewL {
  using L = v2::EvLayout<K>;
  static constexpr int ST = LOCAL ? 1 : kPage;
  const double* in;
  double* buf;
  const Tables* tab;
  const Tab64* t;
  const Tab64::OffL* o;
  int gc;
  double gs;

  __device__ __forceinline__ int h(int mask) const { return LOCAL ? 0 : pext_bits(gc, mask); }
  __device__ __forceinline__ double rec(int item) const { return __ldg(in + item * kPage); }
  __device__ __forceinline__ void ld(int off, cx<double>* v) const {
    const double* p = buf + static_cast<int64_t>(off) * ST;
#pragma unroll
    for (int m = 0; m < 4; ++m) v[m] = {p[(2 * m) * ST], p[(2 * m + 1) * ST]};
  }
  __device__ __forceinline__ void st(int off, const cx<double>* v) const {
    double* p = buf + static_cast<int64_t>(off) * ST;
#pragma unroll
    for (int m = 0; m < 4; ++m) {
      p[(2 * m) * ST] = v[m].r;
      p[(2 * m + 1) * ST] = v[m].i;
    }
  }
  __device__ __forceinline__ int offJ(int s) const { return o->J[s] + h(tab->seq_mask[s]) * 4; }
  __device__ __forceinline__ void J(int s, double* v) const {
    const double* p = buf + static_cast<int64_t>(offJ(s)) * ST;
#pragma unroll
    for (int m = 0; m < 4; ++m) v[m] = p[m * ST];
  }
  __device__ __forceinline__ void stJ(int s, const double* v) const {
    double* p = buf + static_cast<int64_t>(offJ(s)) * ST;
#pragma unroll
    for (int m = 0; m < 4; ++m) p[m * ST] = v[m];
  }
  __device__ __forceinline__ void top(int item, cx<double>* v) const {
#pragma unroll
    for (int q = 0; q < 4; ++q) v[q] = {rec(item + 2 * q), rec(item + 2 * q + 1)};
  }
  __device__ __forceinline__ void qc(int S, double* q) const {
#pragma unroll
    for (int i = 0; i < 5; ++i) q[i] = rec(L::QC + 5 * S + i);
  }
  __device__ __forceinline__ void mom(int s, double* P) const {
#pragma unroll
    for (int m = 0; m < 4; ++m) P[m] = rec(L::PT + 4 * tab->seq_mask[s] + m);
  }
  __device__ __forceinline__ void gluon(int g, double* J) const {   // e_theta or e_phi (no z component), / sqrt 2
    const int phi = (gc >> g) & 1;
    J[0] = 0.0;
    J[1] = rec(L::EPS + 5 * g + (phi ? 3 : 0));
    J[2] = rec(L::EPS + 5 * g + (phi ? 4 : 1));
    J[3] = phi ? 0.0 : rec(L::EPS + 5 * g + 2);
  }
  __device__ __forceinline__ int offPsi(int m, int p) const {
    return o->psi[m][p] + h(tab->prefix_mask[p * kFact[K - m]][m]) * 8;
  }
  __device__ __forceinline__ int offQv(int m, int p, int b) const {
    return o->qv[m][p] + (h(tab->prefix_mask[p * kFact[K - m]][m]) * 2 + b) * 8;
  }
  __device__ __forceinline__ int offChi(int g, int b) const { return o->chi[g] + (h(1 << g) * 2 + b) * 8; }
  __device__ __forceinline__ int offQg(int g, int b) const { return o->qg[g] + (h(1 << g) * 2 + b) * 8; }
  __device__ __forceinline__ int offZ(int g, int g2, int b) const {
    return o->z[g * kMaxGluons + g2] + (h(1 << g | 1 << g2) * 2 + b) * 8;
  }
  __device__ __forceinline__ int offY(int s, int g, int b) const {
    return o->y[s][g] + (h(tab->seq_mask[s] | 1 << g) * 2 + b) * 8;
  }
  __device__ __forceinline__ int offQQ(int g, int g2, int b) const {
    return o->qq[g * kMaxGluons + g2] + (h(1 << g | 1 << g2) * 2 + b) * 8;
  }
  __device__ __forceinline__ int offFull(int f) const { return o->full[f] + h((1 << K) - 1) * 4; }

  __device__ __forceinline__ double dot(int r, int s) const {   // g J_r . J_s
    return buf[static_cast<int64_t>(o->dot[r][s] + h(tab->seq_mask[r] | tab->seq_mask[s])) * ST];
  }
  __device__ __forceinline__ cx<double> d(int s, int b) const {
    const double* p = buf + static_cast<int64_t>(o->d[s] + h(tab->seq_mask[s]) * 4 + 2 * b) * ST;
    return {p[0], p[ST]};
  }
  __device__ __forceinline__ void st_d(int s, int b, cx<double> x) const {
    double* p = buf + static_cast<int64_t>(o->d[s] + h(tab->seq_mask[s]) * 4 + 2 * b) * ST;
    p[0] = x.r;
    p[ST] = x.i;
  }
  __device__ __forceinline__ int offU(int s, int b) const { return o->u[s] + (h(tab->seq_mask[s]) * 2 + b) * 8; }

  // current of a canonical split list; the four-gluon vertices from the tabulated products: 13 instructions each
  __device__ __forceinline__ void vertices(double* acc, int n3, const int16_t (*v3)[2], int n4, const int16_t (*v4)[3]) const {
    for (int k = 0; k < n3; ++k) {
      const int16_t rl = v3[k][0], rr = v3[k][1];
      double JL[4], JR[4], PL[4], PR[4];
      J(v2::rslot(rl), JL);
      J(v2::rslot(rr), JR);
      mom(v2::rslot(rl), PL);
      mom(v2::rslot(rr), PR);
      v3r_acc(acc, JL, JR, PL, PR, v2::rneg(rl) != v2::rneg(rr));
    }
    for (int k = 0; k < n4; ++k) {
      const int a = v2::rslot(v4[k][0]), b = v2::rslot(v4[k][1]), c = v2::rslot(v4[k][2]);
      const bool neg = v2::rneg(v4[k][0]) ^ v2::rneg(v4[k][1]) ^ v2::rneg(v4[k][2]);
      double JA[4], JB[4], JC[4];
      J(a, JA);
      J(b, JB);
      J(c, JC);
      double ab = dot(a, b), bc = dot(b, c), ac = -2.0 * dot(a, c);
      if (neg) { ab = -ab; bc = -bc; ac = -ac; }
#pragma unroll
      for (int m = 0; m < 4; ++m) acc[m] = fma(ac, JB[m], fma(bc, JA[m], fma(ab, JC[m], acc[m])));
    }
  }
  // all gluons on one current contracted with ubar gamma^mu v, without the propagator.  A three-gluon vertex of a
  // split (L, R) is the shorter side's U times the longer side's current, antisymmetric in L and R; a four-gluon vertex
  // combines tabulated products: 16 and 13 instructions for both antitop helicities, where the vector form takes 30
  // and 13 and the contraction 16 more per current.
  __device__ __forceinline__ void full(int f, cx<double>* x) const {
    x[0] = x[1] = {0.0, 0.0};
    for (int k = 0; k < tab->full_nv3[f]; ++k) {
      const int16_t rl = tab->full_v3[f][k][0], rr = tab->full_v3[f][k][1];
      const int l = v2::rslot(rl), r = v2::rslot(rr);
      const bool left = tab->seq_len[l] <= tab->seq_len[r];
      const bool neg = (v2::rneg(rl) != v2::rneg(rr)) != !left;
      double Jl[4];
      J(left ? r : l, Jl);
      if (neg)
#pragma unroll
        for (int m = 0; m < 4; ++m) Jl[m] = -Jl[m];
#pragma unroll
      for (int b = 0; b < 2; ++b) {
        cx<double> U[4];
        ld(offU(left ? l : r, b), U);
        x[b].r = fma(U[0].r, Jl[0], x[b].r);
        x[b].i = fma(U[0].i, Jl[0], x[b].i);
#pragma unroll
        for (int m = 1; m < 4; ++m) {
          x[b].r = fma(-U[m].r, Jl[m], x[b].r);
          x[b].i = fma(-U[m].i, Jl[m], x[b].i);
        }
      }
    }
    for (int k = 0; k < tab->full_nv4[f]; ++k) {
      const int16_t* v = tab->full_v4[f][k];
      const int a = v2::rslot(v[0]), b = v2::rslot(v[1]), c = v2::rslot(v[2]);
      double ab = dot(a, b), bc = dot(b, c), ac = -2.0 * dot(a, c);
      if (v2::rneg(v[0]) ^ v2::rneg(v[1]) ^ v2::rneg(v[2])) { ab = -ab; bc = -bc; ac = -ac; }
#pragma unroll
      for (int q = 0; q < 2; ++q) {
        v2::cmacr(x[q], ab, d(c, q));
        v2::cmacr(x[q], bc, d(a, q));
        v2::cmacr(x[q], ac, d(b, q));
      }
    }
  }
};

// psi_M of prefix p, and its bilinears with v where an amplitude uses them (M <= K - 3)
template <int K, bool LOCAL, int M>
__device__ __forceinline__ void task_psi_l(const ViewL<K, LOCAL>& V, int p) {
  using L = v2::EvLayout<K>;
  const int c0 = p * kFact[K - M];
  cx<double> acc[4] = {};
#pragma unroll
  for (int j = 0; j < M; ++j) {
    const int16_t r = V.tab->sub[c0][j][M];
    double Jr[4];
    if constexpr (M == 1) V.gluon(v2::rslot(r), Jr);
    else V.J(v2::rslot(r), Jr);
    cx<double> s[4];
    if (j == 0) V.top(L::UB, s);
    else V.ld(V.offPsi(j, c0 / kFact[K - j]), s);
    row_rslash_acc(acc, s, rslash(Jr, v2::rneg(r)));
  }
  double q[5];
  V.qc(V.tab->prefix_mask[c0][M], q);
  cx<double> out[4];
  v2::row_prop(acc, q, out);
  V.st(V.offPsi(M, p), out);
  if constexpr (M <= K - 3) {
#pragma unroll
    for (int b = 0; b < 2; ++b) {
      cx<double> v[4], Jq[4];
      V.top(L::VV + 8 * b, v);
      v2::quark_current(out, v, Jq);
      V.st(V.offQv(M, p, b), Jq);
    }
  }
}

template <int K, bool LOCAL>
__device__ __forceinline__ void run_task_l(const ViewL<K, LOCAL>& V, uint32_t task) {
  using L = v2::EvLayout<K>;
  const int type = task & 15, a_ = (task >> 4) & 1023, b_ = (task >> 14) & 63;
  switch (type) {
    case Tab64::kJ1: {
      double J[4];
      V.gluon(a_, J);
      V.stJ(a_, J);
      break;
    }
    case Tab64::kJq0: {
#pragma unroll
      for (int b = 0; b < 2; ++b) {
        cx<double> u[4], v[4], Jq[4];
        V.top(L::UB, u);
        V.top(L::VV + 8 * b, v);
        v2::quark_current(u, v, Jq);
        V.st(V.o->q0 + b * 8, Jq);
      }
      break;
    }
    case Tab64::kChi: {   // chi(g), and ubar gamma^mu chi(g)
      double J[4];
      V.gluon(a_, J);
      const RSlash g = rslash(J, false);
      double q[5];
      V.qc(((1 << K) - 1) ^ (1 << a_), q);
#pragma unroll
      for (int b = 0; b < 2; ++b) {
        cx<double> v[4], X[4] = {}, chi[4], u[4], Jq[4];
        V.top(L::VV + 8 * b, v);
        col_rslash_acc(X, g, v);
        col_prop(X, q, chi);
        V.st(V.offChi(a_, b), chi);
        V.top(L::UB, u);
        v2::quark_current(u, chi, Jq);
        V.st(V.offQg(a_, b), Jq);
      }
      break;
    }
    case Tab64::kPsi:
      if (b_ == 1) task_psi_l<K, LOCAL, 1>(V, a_);
      if constexpr (K >= 4) if (b_ == 2) task_psi_l<K, LOCAL, 2>(V, a_);
      if constexpr (K >= 5) if (b_ == 3) task_psi_l<K, LOCAL, 3>(V, a_);
      break;
    case Tab64::kSeq: {
      double acc[4] = {};
      V.vertices(acc, V.tab->seq_nv3[a_], V.tab->seq_v3[a_], V.tab->seq_nv4[a_], V.tab->seq_v4[a_]);
      const double f = V.rec(L::GP + V.tab->seq_mask[a_]);
#pragma unroll
      for (int m = 0; m < 4; ++m) acc[m] *= f;
      V.stJ(a_, acc);
      if (K == 5 && V.tab->seq_len[a_] == 3)
#pragma unroll
        for (int b = 0; b < 2; ++b) {
          cx<double> Jq[4];
          V.ld(V.o->q0 + b * 8, Jq);
          V.st_d(a_, b, qdot(Jq, acc));
        }
      break;
    }
    case Tab64::kZ: {   // Z(g, h) and Z(h, g) of a canonical pair: J(h, g) = -J(g, h)
      const int m = V.tab->seq_mask[a_], g = __ffs(m) - 1, g2 = __ffs(m & (m - 1)) - 1;
      double J[4], Jg[4], Jh[4];
      V.J(a_, J);
      V.J(g, Jg);
      V.J(g2, Jh);
      const RSlash sj = rslash(J, false), sg = rslash(Jg, false), sh = rslash(Jh, false);
#pragma unroll
      for (int b = 0; b < 2; ++b) {
        cx<double> v[4], X[4] = {}, z[4], c[4];
        V.top(L::VV + 8 * b, v);
        col_rslash_acc(X, sj, v);
#pragma unroll
        for (int i = 0; i < 4; ++i) z[i] = v2::cneg(X[i]);
        V.ld(V.offChi(g2, b), c);
        col_rslash_acc(X, sg, c);
        V.st(V.offZ(g, g2, b), X);
        V.ld(V.offChi(g, b), c);
        col_rslash_acc(z, sh, c);
        V.st(V.offZ(g2, g, b), z);
      }
      break;
    }
    case Tab64::kFull: {
      cx<double> x[2];
      V.full(a_, x);
      const double f = V.rec(L::GP + (1 << K) - 1);
      double* p = V.buf + static_cast<int64_t>(V.offFull(a_)) * ViewL<K, LOCAL>::ST;
#pragma unroll
      for (int b = 0; b < 2; ++b) {
        p[(2 * b) * ViewL<K, LOCAL>::ST] = f * x[b].r;
        p[(2 * b + 1) * ViewL<K, LOCAL>::ST] = f * x[b].i;
      }
      break;
    }
    case Tab64::kU: {
      // D = Jq.J and U = 2 [(Jq.P) J + (J.P') Jq - (Jq.J) P] for Jq = ubar gamma^mu v, P the current's momentum and P'
      // the other gluons': U.R = Jq . V3(J, R) for a conserved current R of the other gluons (P'.R = 0), Jq being
      // conserved too (Jq.(P + P') = 0)
      double J[4], P[4], PR[4];
      V.J(a_, J);
      V.mom(a_, P);
      const int rest = ((1 << K) - 1) ^ V.tab->seq_mask[a_];
#pragma unroll
      for (int m = 0; m < 4; ++m) PR[m] = V.rec(L::PT + 4 * rest + m);
      const double jp = 2.0 * rdot(J, PR);
#pragma unroll
      for (int m = 0; m < 4; ++m) P[m] *= 2.0;
#pragma unroll
      for (int b = 0; b < 2; ++b) {
        cx<double> Jq[4], U[4];
        V.ld(V.o->q0 + b * 8, Jq);
        const cx<double> qp = qdot(Jq, P), qj = qdot(Jq, J);
        V.st_d(a_, b, qj);
#pragma unroll
        for (int m = 0; m < 4; ++m) {
          U[m] = v2::cscale(J[m], qp);
          v2::cmacr(U[m], jp, Jq[m]);
          v2::cmacr(U[m], -P[m], qj);
        }
        V.st(V.offU(a_, b), U);
      }
      break;
    }
    case Tab64::kDot: {   // g J.J' of two sequences
      double A[4], B[4];
      V.J(a_, A);
      V.J(b_, B);
      V.buf[static_cast<int64_t>(V.o->dot[a_][b_] + V.h(V.tab->seq_mask[a_] | V.tab->seq_mask[b_])) * ViewL<K, LOCAL>::ST] =
          V.gs * rdot(A, B);
      break;
    }
    case Tab64::kY: {   // (gamma.J_s) chi(g), 5 gluons
      double J[4];
      V.J(a_, J);
      const RSlash s = rslash(J, false);
#pragma unroll
      for (int b = 0; b < 2; ++b) {
        cx<double> c[4], Y[4] = {};
        V.ld(V.offChi(b_, b), c);
        col_rslash_acc(Y, s, c);
        V.st(V.offY(a_, b_, b), Y);
      }
      break;
    }
    default: {   // kQQ: psi_1(g) gamma^mu chi(h), 4 and 5 gluons
#pragma unroll
      for (int b = 0; b < 2; ++b) {
        cx<double> s[4], c[4], Jq[4];
        V.ld(V.offPsi(1, a_), s);
        V.ld(V.offChi(b_, b), c);
        v2::quark_current(s, c, Jq);
        V.st(V.offQQ(a_, b_, b), Jq);
      }
      break;
    }
  }
}

// The amplitudes of one (event, polarisation combination, antitop helicity b).
template <int K, bool LOCAL>
__device__ __forceinline__ void row64_l(const ViewL<K, LOCAL>& V, int b, cx<double>* A) {
  constexpr int NCOL = v2::Sizes<K>::ncol, NFULL = v2::Sizes<K>::nfull;
  constexpr bool kNegK = (K & 1) == 0, kNegK1 = !kNegK;
  const Tab64* t = V.t;
  for (int f = 0; f < NFULL; ++f) {
    const double* p = V.buf + static_cast<int64_t>(V.offFull(f) + 2 * b) * ViewL<K, LOCAL>::ST;
    const cx<double> x = {p[0], p[ViewL<K, LOCAL>::ST]};
    A[t->full_c[f]] = x;
    A[t->full_cr[f]] = kNegK ? v2::cneg(x) : x;
  }
  auto add = [&](int c, cx<double> x, bool neg) {
    A[c].r = neg ? A[c].r - x.r : A[c].r + x.r;
    A[c].i = neg ? A[c].i - x.i : A[c].i + x.i;
  };
  constexpr int NLAST = NCOL / 2 / K;
  for (int g = 0; g < K; ++g) {
    cx<double> Q[4];
    V.ld(V.offQg(g, b), Q);
    for (int i = g * NLAST; i < (g + 1) * NLAST; ++i) {
      double J[4];
      V.J(t->t1[i][0], J);
      const cx<double> x = qdot(Q, J);
      add(t->t1[i][1], x, false);
      add(t->t1[i][2], x, kNegK1);
    }
  }
  if constexpr (K == 5) {
    for (int g = 0; g < K; ++g) {
      cx<double> Q[4];
      V.ld(V.offQv(1, g, b), Q);
      for (int i = g * NLAST; i < (g + 1) * NLAST; ++i) {
        double J[4];
        V.J(t->t2[i][0], J);
        const cx<double> x = qdot(Q, J);
        add(t->t2[i][1], x, false);
        add(t->t2[i][2], x, true);
      }
    }
    for (int q = 0; q < K * (K - 1); ++q) {
      cx<double> Q[4];
      V.ld(V.offQQ(t->t3q[q][0], t->t3q[q][1], b), Q);
#pragma unroll
      for (int i = 0; i < 3; ++i) {
        double J[4];
        V.J(t->t3[3 * q + i][0], J);
        const cx<double> x = qdot(Q, J);
        add(t->t3[3 * q + i][1], x, false);
        add(t->t3[3 * q + i][2], x, false);
      }
    }
  }
  for (int p = 0; p < NCOL / 6; ++p) {   // six orderings with a common prefix, as in slot64
    cx<double> acc[6] = {};
    if constexpr (K >= 4) {
      cx<double> Q[4];
      V.ld(V.offQv(K - 3, p, b), Q);
      constexpr int c3[3] = {0, 1, 2}, r3[3] = {5, 3, 4};
#pragma unroll
      for (int i = 0; i < 3; ++i) {
        double J[4];
        V.J(t->g3[p][i], J);
        acc[c3[i]] = acc[r3[i]] = qdot(Q, J);
      }
      constexpr int cy[3] = {0, 1, 3}, ry[3] = {2, 4, 5};
      cx<double> s[4];
      if constexpr (K == 5) V.ld(V.offPsi(K - 3, p), s);
#pragma unroll
      for (int i = 0; i < 3; ++i) {
        cx<double> v = {};
        if constexpr (K == 5) {
          cx<double> Y[4];
          V.ld(V.offY(t->gy[p][i][0], t->gy[p][i][1], b), Y);
          v2::sdot_acc(v, s, Y, false);
        } else {
          double J[4];
          V.ld(V.offQQ(p, t->gy[p][i][1], b), s);   // (4 gluons: prefix p is gluon p)
          V.J(t->gy[p][i][0], J);
          v = qdot(s, J);
        }
        acc[cy[i]].r += v.r; acc[cy[i]].i += v.i;
        acc[ry[i]].r -= v.r; acc[ry[i]].i -= v.i;
      }
    }
#pragma unroll
    for (int i = 0; i < 3; ++i) {
      cx<double> s[4];
      V.ld(V.offPsi(K - 2, 3 * p + i), s);
#pragma unroll
      for (int q = 0; q < 2; ++q) {
        const int z = t->gz[p][2 * i + q];
        cx<double> Z[4];
        V.ld(V.offZ(z / kMaxGluons, z % kMaxGluons, b), Z);
        v2::sdot_acc(acc[2 * i + q], s, Z, false);
      }
    }
#pragma unroll
    for (int c = 0; c < 6; ++c) add(6 * p + c, acc[c], false);
  }
}

// amplitude of (event, row, ordering) in a buffer of all of them, interleaved by page
template <int K>
__host__ __device__ constexpr int amp_doubles() { return (2 << K) * v2::Sizes<K>::ncol * 2; }
template <int K>
__device__ __forceinline__ double* amp_at(double* amp, int64_t e, int row, int c) {
  return amp + (e / kPage) * static_cast<int64_t>(amp_doubles<K>()) * kPage + (row * v2::Sizes<K>::ncol + c) * 2 * kPage + e % kPage;
}

// A warp takes one top helicity pair of one combination (the all-gluon currents, which the pairs share, are items
// of the last pass): a thread doing all four pairs made 4 times longer warps, of which gg->ttgg's 10,007 events are
// 4.1 per sub-partition, so the busiest had 5; measured in the helicity basis 2.81 vs 3.19 ms there, gg->ttggg + TC colour 7.60 vs 8.60 ms
// per 2,049 events, gg->ttg 12.05 vs 12.13 ms per 524,288.
//
// One thread of a block (32 events x 4 warps) on event tile `tile`, block `blk` < 2^(K-1) of the tile.
// amp (AMP): the amplitudes of row 4 blk + w = 2 * polarisations + antitop helicity for warp w.  Else the colour sums:
// *lin != 0: of the same row, into out[row * stride + e]; *lin = 0: of helicities, with the shared items warp w on the
// top helicity pair w of combination hslots[blk]; without them (LOCAL) on the four pairs of combination
// hslots[4 blk + w], whose items it builds once.
template <int K, bool AMP, bool LOCAL>
__device__ __forceinline__ void thread64(const double* __restrict__ rec, int64_t nevt, int64_t tile, int blk,
                                         const Tables* __restrict__ tab, const Tab64* __restrict__ t64,
                                         const int* __restrict__ hslots, const int* __restrict__ nslot,
                                         const int* __restrict__ lin, const uint32_t* __restrict__ mask,
                                         const double* __restrict__ ctri, const MeConst& cst, double* __restrict__ out,
                                         int64_t stride, const double* __restrict__ share) {
  constexpr int NCOL = v2::Sizes<K>::ncol;
  const int64_t e = tile * kPage + threadIdx.x % kPage;
  const int warp = threadIdx.x / kPage;
  if (e >= nevt) return;
  const double* in = rec + (e / kPage) * v2::EvLayout<K>::NITEM * kPage + (e % kPage);
  double own[!LOCAL ? 1 : AMP || Loc<K>::n < LocL<K>::n ? LocL<K>::n : Loc<K>::n];
  double* buf = own;
  if constexpr (!LOCAL)
    buf = const_cast<double*>(share) + (e / kPage) * static_cast<int64_t>(t64->stride) * kPage + (e % kPage);
  if (AMP || *lin) {
    const int row = 4 * blk + warp;
    const ViewL<K, LOCAL> V = {in, buf, tab, t64, LOCAL ? &t64->locl : &t64->shl, row >> 1, cst.gs};
    if constexpr (LOCAL)
      for (int i = 0; i < t64->nltaskl; ++i) run_task_l<K, true>(V, t64->ltaskl[i]);
    cx<double> A[NCOL];
    row64_l<K, LOCAL>(V, row & 1, A);
    if constexpr (AMP) {
      double* p = amp_at<K>(out, e, row, 0);
      for (int c = 0; c < NCOL; ++c) {
        p[2 * c * kPage] = A[c].r;
        p[(2 * c + 1) * kPage] = A[c].i;
      }
    } else {
      out[row * stride + e] = colour_sum64<K>(A, t64, ctri) * cst.colour_scale;
    }
    return;
  }
  if constexpr (!AMP) {
    const int slot = LOCAL ? 4 * blk + warp : blk;
    if (slot >= *nslot) return;
    const View<K, LOCAL> V = {in, buf, tab, t64, LOCAL ? &t64->loc : &t64->sh, hslots[slot], cst.gs};
    if constexpr (LOCAL) {
      for (int i = 0; i < t64->nltask; ++i) run_task<K, true>(V, t64->ltask[i]);
      for (int ab = 0; ab < 4; ++ab) slot64<K, true>(V, e, slot, ab, mask, ctri, cst, out, stride);
    } else {
      slot64<K, false>(V, e, slot, warp, mask, ctri, cst, out, stride);
    }
  }
}

// From the linear polarisations' amplitudes of one (event, ordering, antitop helicity b) to the helicities': per gluon
// M(+) = -M(theta) + i s M(phi), M(-) = M(theta) + i s M(phi), s = +1 outgoing (ext_gluon).  a[x]: bit g of x = phi in,
// helicity +1 out; top helicity -1 throughout.
template <int K>
__device__ __forceinline__ void to_helicities(cx<double>* a) {
#pragma unroll
  for (int g = 0; g < K; ++g)
#pragma unroll
    for (int x = 0; x < (1 << K); ++x)
      if (!((x >> g) & 1)) {
        const cx<double> t = a[x], f = a[x | 1 << g];
        const cx<double> p = g < 2 ? cx<double>{f.i, -f.r} : cx<double>{-f.i, f.r};   // i s M(phi)
        a[x] = {t.r + p.r, t.i + p.i};
        a[x | 1 << g] = {p.r - t.r, p.i - t.i};
      }
}

// helicity index of gluon helicities x (bit g: +1), top helicity -1, antitop helicity b
template <int K>
__device__ __forceinline__ int hel_of_row(int x, int b) {
  constexpr int npar = K + 2;
  int h = b << (npar - 4);
#pragma unroll
  for (int g = 0; g < K; ++g)
    if ((x >> g) & 1) h |= 1 << (npar - 1 - (g < 2 ? g : g + 2));
  return h;
}

}  // namespace m64
}  // namespace mg
