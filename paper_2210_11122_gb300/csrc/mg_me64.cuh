// mg_me64.cuh -- the FP64 matrix elements of 3 to 5 gluons: colour-ordered amplitudes with the quark line cut
// in front of its last two gluons, one thread per (event, gluon-helicity combination).
//
// GB300 issues one FP64 instruction per warp and SM sub-partition every 64 cycles, so the FP64 instruction count is
// the cost and everything else (loads, integer work, local memory) hides behind it.  Two things keep it low:
//   * everything that depends on fewer than all gluons is computed once per helicity assignment of those gluons and
//     read by every combination that shares it (k_pass64, a few launches of independent tasks per event, into a
//     page-interleaved buffer);
//   * the amplitude of an ordering sigma of K gluons is not built by carrying the quark line up to the antitop but
//     by cutting it.  With the row spinors psi_m (top and the first m gluons, propagator included), the column
//     spinors chi(g) = S (gamma.J_g) v (antitop and the last gluon, propagator included) and the gluon currents J,
//         A = psi_{K-2} . Z(s_{K-1}, s_K) + sum_{i < K-2} psi_i . [ X(i+1..K) + (gamma.J(i+1..K-1)) chi(s_K) ],
//         Z(g, h) = (gamma.J_g) chi(h) + (gamma.J_gh) v,   X(i+1..K) = (gamma.J(i+1..K)) v:
//     every term is one spinor or vector product (16 FP64 instructions per helicity), the factors are shared, and a
//     term whose current holds two or more consecutive gluons serves two orderings (reflection, up to a sign).  No
//     prefix of K-1 gluons is formed, which was most of the quark line's cost (5 gluons: 256 instead of 704
//     instructions per ordering and combination).
// A flipped combination's |M|^2 equals the combination's (hel_weight), so gluon K-1 has helicity -1 throughout and
// an item's helicity index leaves its bit out.
//
// The helicity basis of this file is the path of partial helicity masks; with every helicity good the same scheme runs
// over linear polarisations (mg_me64l.cuh).  Measured in this basis against carrying the prefixes of up to K-1 gluons, both
// on half of the combinations: gg->ttg 12.13 vs 14.48 ms per 524,288 events, amplitudes of gg->ttggg 8.60 vs 12.37 ms
// per 2,049; with 20 of 32 / 50 of 64 / 112 of 128 helicities good now 0.17 / 1.14 / 15.5 ms per 4,099 events of
// gg->ttg / ttgg / ttggg (0.28 / 2.95 / 57.3 before).
//
// The combination may also build its own items in local memory (LOCAL, no buffer): the same functions, so the same
// bits, at about three times the FP64 work and, with 5 gluons, 50 KB of local memory per thread.
#pragma once

#include "mg_me_algebra.cuh"

namespace mg {
namespace m64 {

using v2::cx;

__device__ constexpr int kFact[6] = {1, 1, 2, 6, 24, 120};

// doubles of one combination's own items (LOCAL)
template <int K> struct Loc;
template <> struct Loc<3> { static constexpr int n = 392; };
template <> struct Loc<4> { static constexpr int n = 1328; };
template <> struct Loc<5> { static constexpr int n = 5832; };

// (Qslash + m) f on a column spinor, coefficients as row_prop's
__device__ __forceinline__ void col_prop(const cx<double>* s, const double* q, cx<double>* o) {
  const double qa = q[0], qb = q[1], qm = q[4];
  const cx<double> qp = {q[2], q[3]}, qn = {q[2], -q[3]};
  o[0] = v2::cscale(qb, s[2]); v2::cmsub(o[0], qn, s[3]); v2::cmacr(o[0], qm, s[0]);
  o[1] = v2::cscale(qa, s[3]); v2::cmsub(o[1], qp, s[2]); v2::cmacr(o[1], qm, s[1]);
  o[2] = v2::cscale(qa, s[0]); v2::cmac(o[2], qn, s[1]); v2::cmacr(o[2], qm, s[2]);
  o[3] = v2::cscale(qb, s[1]); v2::cmac(o[3], qp, s[0]); v2::cmacr(o[3], qm, s[3]);
}

// o += (gamma.J) v from the current's gamma.J entries
__device__ __forceinline__ void col_slash_acc(cx<double>* o, const v2::Slash<double>& g, const cx<double>* v) {
  v2::cmac(o[0], g.b, v[2]); v2::cmsub(o[0], g.jm, v[3]);
  v2::cmac(o[1], g.a, v[3]); v2::cmsub(o[1], g.jp, v[2]);
  v2::cmac(o[2], g.a, v[0]); v2::cmac(o[2], g.jm, v[1]);
  v2::cmac(o[3], g.jp, v[0]); v2::cmac(o[3], g.b, v[1]);
}

// The items of one event for the helicities gc: in the shared buffer (double d of event e at
// (e / 32) * stride * 32 + d * 32 + e % 32, so a warp's access is one 256-byte line) or in the thread's own array.
template <int K, bool LOCAL>
struct View {
  using L = v2::EvLayout<K>;
  static constexpr int ST = LOCAL ? 1 : kPage;
  const double* in;   // the event's record
  double* buf;
  const Tables* tab;
  const Tab64* t;
  const Tab64::Off* o;
  int gc;
  double gs;

  __device__ __forceinline__ int h(int mask) const { return LOCAL ? 0 : pext_bits(gc, mask & ((1 << (K - 1)) - 1)); }
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
  __device__ __forceinline__ void top(int item, cx<double>* v) const {   // L::UB or L::VV + 8 * helicity
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
  __device__ __forceinline__ void gluon(int g, cx<double>* J) const {   // the external current itself
    double pol[5];
#pragma unroll
    for (int i = 0; i < 5; ++i) pol[i] = rec(L::EPS + 5 * g + i);
    v2::ext_gluon(pol, (gc >> g) & 1 ? 1 : -1, g >= 2, J);
  }
  __device__ __forceinline__ int offJ(int s) const { return o->J[s] + h(tab->seq_mask[s]) * 8; }
  __device__ __forceinline__ int offX(int s, int b) const { return o->X[s] + (h(tab->seq_mask[s]) * 2 + b) * 8; }
  __device__ __forceinline__ int offPsi(int m, int p, int a) const {
    return o->psi[m][p] + (h(tab->prefix_mask[p * kFact[K - m]][m]) * 2 + a) * 8;
  }
  __device__ __forceinline__ int offChi(int g, int b) const { return o->chi[g] + (h(1 << g) * 2 + b) * 8; }
  __device__ __forceinline__ int offQg(int g, int ab) const { return o->qg[g] + (h(1 << g) * 4 + ab) * 8; }
  __device__ __forceinline__ int offZ(int g, int g2, int b) const {
    return o->z[g * kMaxGluons + g2] + (h(1 << g | 1 << g2) * 2 + b) * 8;
  }
  __device__ __forceinline__ int offY(int s, int g, int b) const {
    return o->y[s][g] + (h(tab->seq_mask[s] | 1 << g) * 2 + b) * 8;
  }
  __device__ __forceinline__ int offQQ(int g, int g2, int ab) const {
    return o->qq[g * kMaxGluons + g2] + (h(1 << g | 1 << g2) * 4 + ab) * 8;
  }
  __device__ __forceinline__ int offFull(int f) const { return o->full[f] + h((1 << K) - 1) * 8; }
  __device__ __forceinline__ void J(int s, cx<double>* v) const { ld(offJ(s), v); }

  // current of a canonical split list: three- and four-gluon vertices summed
  __device__ __forceinline__ void vertices(cx<double>* acc, int n3, const int16_t (*v3)[2], int n4,
                                           const int16_t (*v4)[3]) const {
    for (int k = 0; k < n3; ++k) {
      const int16_t rl = v3[k][0], rr = v3[k][1];
      cx<double> JL[4], JR[4];
      double PL[4], PR[4];
      J(v2::rslot(rl), JL);
      J(v2::rslot(rr), JR);
      mom(v2::rslot(rl), PL);
      mom(v2::rslot(rr), PR);
      v2::v3_acc(acc, JL, JR, PL, PR, v2::rneg(rl) != v2::rneg(rr));
    }
    for (int k = 0; k < n4; ++k) {
      const int16_t ra = v4[k][0], rb = v4[k][1], rc = v4[k][2];
      cx<double> JA[4], JB[4], JC[4];
      J(v2::rslot(ra), JA);
      J(v2::rslot(rb), JB);
      J(v2::rslot(rc), JC);
      v2::v4_acc(acc, JA, JB, JC, gs, v2::rneg(ra) ^ v2::rneg(rb) ^ v2::rneg(rc));
    }
  }
};

// psi_M of prefix p for both top helicities (each current's gamma.J entries shared by the two)
template <int K, bool LOCAL, int M>
__device__ __forceinline__ void task_psi(const View<K, LOCAL>& V, int p) {
  using L = v2::EvLayout<K>;
  const int c0 = p * kFact[K - M];
  v2::Slash<double> g[M];
#pragma unroll
  for (int j = 0; j < M; ++j) {
    const int16_t r = V.tab->sub[c0][j][M];
    cx<double> Jr[4];
    if constexpr (M == 1) V.gluon(v2::rslot(r), Jr);
    else V.J(v2::rslot(r), Jr);
    g[j] = v2::slash_of(Jr, v2::rneg(r));
  }
  double q[5];
  V.qc(V.tab->prefix_mask[c0][M], q);
#pragma unroll
  for (int a = 0; a < 2; ++a) {
    cx<double> acc[4] = {};
#pragma unroll
    for (int j = 0; j < M; ++j) {
      cx<double> s[4];
      if (j == 0) V.top(L::UB + 8 * a, s);
      else V.ld(V.offPsi(j, c0 / kFact[K - j], a), s);
      v2::row_slash_acc(acc, s, g[j]);
    }
    cx<double> out[4];
    v2::row_prop(acc, q, out);
    V.st(V.offPsi(M, p, a), out);
  }
}

// One task of the passes: an item (or a few that share work) for the view's helicities.
template <int K, bool LOCAL>
__device__ __forceinline__ void run_task(const View<K, LOCAL>& V, uint32_t task) {
  using L = v2::EvLayout<K>;
  const int type = task & 15, a_ = (task >> 4) & 1023, b_ = (task >> 14) & 63;
  switch (type) {
    case Tab64::kJ1: {
      cx<double> J[4];
      V.gluon(a_, J);
      V.st(V.offJ(a_), J);
      break;
    }
    case Tab64::kJq0: {   // ubar gamma^mu v of the four top helicity pairs
#pragma unroll
      for (int ab = 0; ab < 4; ++ab) {
        cx<double> u[4], v[4], Jq[4];
        V.top(L::UB + 8 * (ab >> 1), u);
        V.top(L::VV + 8 * (ab & 1), v);
        v2::quark_current(u, v, Jq);
        V.st(V.o->q0 + ab * 8, Jq);
      }
      break;
    }
    case Tab64::kChi: {   // chi(g), and ubar gamma^mu chi(g)
      cx<double> J[4];
      V.gluon(a_, J);
      double q[5];
      V.qc(((1 << K) - 1) ^ (1 << a_), q);
#pragma unroll
      for (int b = 0; b < 2; ++b) {
        cx<double> v[4], X[4], chi[4];
        V.top(L::VV + 8 * b, v);
        v2::gamma_col(J, v, X);
        col_prop(X, q, chi);
        V.st(V.offChi(a_, b), chi);
#pragma unroll
        for (int a = 0; a < 2; ++a) {
          cx<double> u[4], Jq[4];
          V.top(L::UB + 8 * a, u);
          v2::quark_current(u, chi, Jq);
          V.st(V.offQg(a_, 2 * a + b), Jq);
        }
      }
      break;
    }
    case Tab64::kPsi:
      if (b_ == 1) task_psi<K, LOCAL, 1>(V, a_);
      if constexpr (K >= 4) if (b_ == 2) task_psi<K, LOCAL, 2>(V, a_);
      if constexpr (K >= 5) if (b_ == 3) task_psi<K, LOCAL, 3>(V, a_);
      break;
    case Tab64::kSeq: {   // J of a sequence of two or more gluons; X for those of three or more
      cx<double> acc[4] = {}, J[4];
      V.vertices(acc, V.tab->seq_nv3[a_], V.tab->seq_v3[a_], V.tab->seq_nv4[a_], V.tab->seq_v4[a_]);
      const double f = V.rec(L::GP + V.tab->seq_mask[a_]);
#pragma unroll
      for (int m = 0; m < 4; ++m) J[m] = v2::cscale(f, acc[m]);
      V.st(V.offJ(a_), J);
      if (V.o->X[a_] >= 0) {
#pragma unroll
        for (int b = 0; b < 2; ++b) {
          cx<double> v[4], X[4];
          V.top(L::VV + 8 * b, v);
          v2::gamma_col(J, v, X);
          V.st(V.offX(a_, b), X);
        }
      }
      break;
    }
    case Tab64::kZ: {   // Z(g, h) and Z(h, g) of a canonical pair: J(h, g) = -J(g, h)
      const int m = V.tab->seq_mask[a_], g = __ffs(m) - 1, g2 = __ffs(m & (m - 1)) - 1;
      cx<double> J[4];
      V.J(a_, J);
      cx<double> Jg[4], Jh[4];
      V.J(g, Jg);
      V.J(g2, Jh);
      const v2::Slash<double> sg = v2::slash_of(Jg, false), sh = v2::slash_of(Jh, false);
#pragma unroll
      for (int b = 0; b < 2; ++b) {
        cx<double> v[4], X[4], c[4];
        V.top(L::VV + 8 * b, v);
        v2::gamma_col(J, v, X);
        cx<double> z[4];
#pragma unroll
        for (int i = 0; i < 4; ++i) z[i] = v2::cneg(X[i]);
        V.ld(V.offChi(g2, b), c);
        col_slash_acc(X, sg, c);
        V.st(V.offZ(g, g2, b), X);
        V.ld(V.offChi(g, b), c);
        col_slash_acc(z, sh, c);
        V.st(V.offZ(g2, g, b), z);
      }
      break;
    }
    case Tab64::kFull: {   // all gluons on one current, contracted with the four quark currents: 4 complex numbers
      cx<double> acc[4] = {}, x[4];
      V.vertices(acc, V.tab->full_nv3[a_], V.tab->full_v3[a_], V.tab->full_nv4[a_], V.tab->full_v4[a_]);
      const double f = V.rec(L::GP + (1 << K) - 1);
      cx<double> JF[4];
#pragma unroll
      for (int m = 0; m < 4; ++m) JF[m] = v2::cscale(f, acc[m]);
#pragma unroll
      for (int ab = 0; ab < 4; ++ab) {
        cx<double> Jq[4];
        V.ld(V.o->q0 + ab * 8, Jq);
        x[ab] = v2::mdot(Jq, JF);
      }
      V.st(V.offFull(a_), x);
      break;
    }
    case Tab64::kY: {   // (gamma.J_s) chi(g)
      cx<double> J[4];
      V.J(a_, J);
#pragma unroll
      for (int b = 0; b < 2; ++b) {
        cx<double> c[4], Y[4];
        V.ld(V.offChi(b_, b), c);
        v2::gamma_col(J, c, Y);
        V.st(V.offY(a_, b_, b), Y);
      }
      break;
    }
    default: {   // kQQ: psi_1(g) gamma^mu chi(h), four top helicity pairs
#pragma unroll
      for (int ab = 0; ab < 4; ++ab) {
        cx<double> s[4], c[4], Jq[4];
        V.ld(V.offPsi(1, a_, ab >> 1), s);
        V.ld(V.offChi(b_, ab & 1), c);
        v2::quark_current(s, c, Jq);
        V.st(V.offQQ(a_, b_, ab), Jq);
      }
      break;
    }
  }
}

// sums and differences of the 2^N complex numbers a[0 .. 2^N) over each bit of their index
template <int N>
__device__ __forceinline__ void signed_sums(cx<double>* a) {
#pragma unroll
  for (int bit = 1; bit < (1 << N); bit <<= 1)
#pragma unroll
    for (int m = 0; m < (1 << N); ++m)
      if (!(m & bit)) {
        const cx<double> x = a[m], y = a[m | bit];
        a[m] = {x.r + y.r, x.i + y.i};
        a[m | bit] = {x.r - y.r, x.i - y.i};
      }
}

// Colour sum of the jamps A (overwritten) of one helicity.  4 and 5 gluons: in the basis of Tab64::blk, whose blocks of
// at most 4 / 16 replace the full triangle of 24 / 120: 280 instead of 648 and 2,872 instead of 14,760 FP64
// instructions, most of the slot kernel's work with 5 gluons before.  Measured in the helicity basis: gg->ttggg FP64
// 31.7 vs 41.9 ms per 8,192 events, gg->ttgg 2.64 vs 2.81 ms per 10,007.  With 3 gluons the blocks save nothing.
template <int K>
__device__ __forceinline__ double colour_sum64(cx<double>* A, const Tab64* __restrict__ t, const double* __restrict__ ctri) {
  if constexpr (K < 4) {
    return v2::colour_sum<v2::Sizes<K>::ncol, double>(A, ctri);
  } else {
    for (int o = 0; o < t->n8; ++o) {
      cx<double> a[8];
#pragma unroll
      for (int m = 0; m < 8; ++m) a[m] = A[t->orb8[o][m]];
      signed_sums<3>(a);
#pragma unroll
      for (int m = 0; m < 8; ++m) A[t->orb8[o][m]] = a[m];
    }
    for (int o = 0; o < t->n4; ++o) {
      cx<double> a[4];
#pragma unroll
      for (int m = 0; m < 4; ++m) a[m] = A[t->orb4[o][m]];
      signed_sums<2>(a);
#pragma unroll
      for (int m = 0; m < 4; ++m) A[t->orb4[o][m]] = a[m];
    }
    double sum = 0.0;
    int idx = 0;
    for (int b = 0; b < t->nblk; ++b) {
      const int n = t->blk_n[b];
      for (int i = 0; i < n; ++i) {
        double wr = 0.0, wi = 0.0;
        for (int j = i; j < n; ++j, ++idx) {
          const double c = __ldg(t->blk_c + idx);
          const cx<double> v = A[t->blk[b][j]];
          wr = fma(c, v.r, wr);
          wi = fma(c, v.i, wi);
        }
        const cx<double> v = A[t->blk[b][i]];
        sum = fma(v.r, wr, sum);
        sum = fma(v.i, wi, sum);
      }
    }
    return sum;
  }
}

// The colour sum of one (event, combination, top helicity pair ab = 2 top + antitop) into row slot * 4 + ab:
// out[row * stride + e], 0 for weight 0.
template <int K, bool LOCAL>
__device__ __forceinline__ void slot64(const View<K, LOCAL>& V, int64_t e, int slot, int ab,
                                       const uint32_t* __restrict__ mask, const double* __restrict__ ctri,
                                       const MeConst& cst, double* __restrict__ out, int64_t stride) {
  constexpr int npar = K + 2, NCOL = v2::Sizes<K>::ncol, NFULL = v2::Sizes<K>::nfull;
  constexpr bool kNegK = (K & 1) == 0, kNegK1 = !kNegK;   // reflection signs of K and K-1 gluons: negative?
  const Tab64* t = V.t;
  const int a = ab >> 1, b = ab & 1, row = slot * 4 + ab;
  int hb = (a << (npar - 3)) | (b << (npar - 4));
#pragma unroll
  for (int g = 0; g < K; ++g)
    if ((V.gc >> g) & 1) hb |= 1 << (npar - 1 - (g < 2 ? g : g + 2));
  const int w = hel_weight(mask, hb, npar, cst.conj);
  if (!w) {
    out[row * stride + e] = 0.0;
    return;
  }
  cx<double> A[NCOL];
  for (int f = 0; f < NFULL; ++f) {   // all gluons on one current
    const double* p = V.buf + static_cast<int64_t>(V.offFull(f) + 2 * ab) * View<K, LOCAL>::ST;
    const cx<double> x = {p[0], p[View<K, LOCAL>::ST]};
    A[t->full_c[f]] = x;
    A[t->full_cr[f]] = kNegK ? v2::cneg(x) : x;
  }
  auto add = [&](int c, cx<double> x, bool neg) {
    A[c].r = neg ? A[c].r - x.r : A[c].r + x.r;
    A[c].i = neg ? A[c].i - x.i : A[c].i + x.i;
  };
  // the first K-1 gluons on one current, the last on chi
  constexpr int NLAST = NCOL / 2 / K;
  for (int g = 0; g < K; ++g) {
    cx<double> Jq[4];
    V.ld(V.offQg(g, ab), Jq);
    for (int i = g * NLAST; i < (g + 1) * NLAST; ++i) {
      cx<double> J[4];
      V.J(t->t1[i][0], J);
      const cx<double> x = v2::mdot(Jq, J);
      add(t->t1[i][1], x, false);
      add(t->t1[i][2], x, kNegK1);
    }
  }
  if constexpr (K == 5) {
    // one gluon on the top, the other four on one current
    for (int g = 0; g < K; ++g) {
      cx<double> s[4];
      V.ld(V.offPsi(1, g, a), s);
      for (int i = g * NLAST; i < (g + 1) * NLAST; ++i) {
        cx<double> X[4], x = {};
        V.ld(V.offX(t->t2[i][0], b), X);
        v2::sdot_acc(x, s, X, false);
        add(t->t2[i][1], x, false);
        add(t->t2[i][2], x, true);
      }
    }
    // or three of them and the last on chi
    for (int q = 0; q < K * (K - 1); ++q) {
      cx<double> Jq[4];
      V.ld(V.offQQ(t->t3q[q][0], t->t3q[q][1], ab), Jq);
#pragma unroll
      for (int i = 0; i < 3; ++i) {
        cx<double> J[4];
        V.J(t->t3[3 * q + i][0], J);
        const cx<double> x = v2::mdot(Jq, J);
        add(t->t3[3 * q + i][1], x, false);
        add(t->t3[3 * q + i][2], x, false);
      }
    }
  }
  // the orderings of the last three gluons after a common prefix: six consecutive orderings, x < y < z in
  // lexicographic order (xyz xzy yxz yzx zxy zyx), added up in registers
  for (int p = 0; p < NCOL / 6; ++p) {
    cx<double> acc[6] = {};
    if constexpr (K >= 4) {
      cx<double> s[4];
      V.ld(V.offPsi(K - 3, p, a), s);
      constexpr int c3[3] = {0, 1, 2}, r3[3] = {5, 3, 4};   // J(xyz) = J(zyx), ...
#pragma unroll
      for (int i = 0; i < 3; ++i) {
        cx<double> X[4];
        V.ld(V.offX(t->g3[p][i], b), X);
        v2::sdot_acc(acc[c3[i]], s, X, false);
        acc[r3[i]] = acc[c3[i]];
      }
      constexpr int cy[3] = {0, 1, 3}, ry[3] = {2, 4, 5};   // (xy)z, (xz)y, (yz)x: J(yx) = -J(xy)
#pragma unroll
      for (int i = 0; i < 3; ++i) {
        cx<double> Y[4], v = {};
        V.ld(V.offY(t->gy[p][i][0], t->gy[p][i][1], b), Y);
        v2::sdot_acc(v, s, Y, false);
        acc[cy[i]].r += v.r; acc[cy[i]].i += v.i;
        acc[ry[i]].r -= v.r; acc[ry[i]].i -= v.i;
      }
    }
#pragma unroll
    for (int i = 0; i < 3; ++i) {
      cx<double> s[4];
      V.ld(V.offPsi(K - 2, 3 * p + i, a), s);
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

  out[row * stride + e] = colour_sum64<K>(A, t, ctri) * cst.colour_scale;
}

}  // namespace m64
}  // namespace mg
