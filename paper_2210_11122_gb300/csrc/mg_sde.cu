// mg_sde.cu -- single-diagram-enhancement channel weights (the MadEvent phase-space channels the paper's
// Sec. 2 lists among the engine's features).
//
// For channel d, a Feynman diagram built from three-point vertices only, the weight of an event is
//     w_d = sum_h |A_d(h)|^2 / sum_d' sum_h |A_d'(h)|^2       (good helicities h),
// A_d the amplitude of the diagram alone, colour factor stripped: gluon trees attached along the quark
// line from the top to the antitop, Feynman-gauge three-gluon vertices in full (single diagrams carry
// no current conservation, so the simplified vertex of the recursion does not apply), quark and gluon
// propagators.  The recursion of the matrix-element kernels sums diagrams into shared currents and never
// forms one diagram alone, so this is a separate, table-driven FP64 kernel:
//   * host: every binary gluon tree over every gluon subset (3 / 9 / 37 / 225 for 2..5 gluons, children
//     before parents) and a depth-first walk over the ordered lists of trees that partition the gluons
//     (a "push" attaches a tree and propagates the spinor, a "leaf" closes a diagram with the antitop):
//     3 / 15 / 105 / 945 channels;
//   * device: one thread per (event, gluon-helicity combination; one of each flipped pair) builds every tree current once (the
//     gluon helicities fixed) and walks the list for each top helicity, the spinor prefixes on a stack,
//     adding |A_d|^2 of each good helicity into per-channel sums; a second kernel adds the combinations
//     and normalises per event.
// Where every helicity is good the weights run over linear gluon polarisations instead (the sum over a gluon's two
// polarisations is the same in either basis, for single diagrams too, and mg_me64l.cuh's arguments hold: real currents, one
// top helicity), and what depends on fewer than all gluons is computed once per polarisation of those gluons: tree
// currents, spinors after a list of trees (up to K-2 gluons), and their products with the antitop side, by a few passes
// (k_sde_pass); then one thread per (event, channel) adds |A_d|^2 over the polarisations (k_sde_leaf):
//   * the last gluon alone on the antitop: (psi_p gamma.J_n) . chi(g) over the prefix p, tree n in front of it;
//   * a pair: psi . (gamma.J) v; three or more: (psi gamma^mu v) . J; all gluons on one tree: the three-gluon vertex
//     of its children contracted with the quark current, from Jq.J of the children.
// gg -> t tbar g, 65,536 events: 1.05 ms, with one thread per helicity combination 2.27; gg -> t tbar g g, 16,384: 2.4 ms
// (14.8 with every helicity evaluated); gg -> t tbar g g g, 2,048: 4.9 ms (42.1).
// Every vertex carries one power of g (the quark propagators and gluon propagators of the per-event
// record carry it), so g^(n_g+1) and the propagator signs are common to all channels and cancel in w_d.
#include <cuda_runtime.h>

#include <cmath>
#include <cstring>
#include <functional>
#include <mutex>
#include <string>
#include <vector>

#include "mg_alloc.h"
#include "mg_ctx.h"
#include "mg_internal.h"
#include "mg_kernels.h"
#include "mg_me64l.cuh"
#include "mg_me_algebra.cuh"

namespace mg {
namespace sde {

constexpr int kMaxNode = 225, kMaxOp = 1655, kMaxCh = 945;

struct Tab {
  int K, nnode, nop, nch;
  int16_t node_l[kMaxNode], node_r[kMaxNode];   // children (internal nodes); node_l = -1 - g for leaf g
  uint8_t node_mask[kMaxNode];
  int16_t op_node[kMaxOp], op_ch[kMaxOp];       // op_ch >= 0: closes channel op_ch; -1: attaches and propagates
  uint8_t op_depth[kMaxOp], op_mask[kMaxOp];    // trees before this one; gluons attached including this tree
};

template <int K> struct Sz;
template <> struct Sz<2> { static constexpr int nnode = 3, nop = 5, nch = 3; };
template <> struct Sz<3> { static constexpr int nnode = 9, nop = 27, nch = 15; };
template <> struct Sz<4> { static constexpr int nnode = 37, nop = 187, nch = 105; };
template <> struct Sz<5> { static constexpr int nnode = 225, nop = 1655, nch = 945; };

// Linear polarisations: items (offsets in doubles per event; one entry per polarisation of the item's gluons), the tasks of
// the passes and the channels.
struct TabL {
  enum Task { kLeafJ, kQ0, kChi, kNode, kPre, kQ };
  enum Chan { kOne, kPair, kMany, kAll };
  static constexpr int kMaxPre = 190, kMaxTask = 3400, kMaxPass = 4;
  int stride, npass, pass0[kMaxPass + 1], npre;
  int J[kMaxNode], D[kMaxNode], X[kMaxNode];   // tree current (4); Jq.J, two antitop helicities (4); (gamma.J) v, pairs (16)
  int chi[5], q0;                               // column spinor before the last gluon (16); ubar gamma^mu v (16)
  int psi[kMaxPre], q[kMaxPre];                 // row spinor after a list of trees (8); psi gamma^mu v (16), -1: none
  int16_t pre_parent[kMaxPre], pre_node[kMaxPre];   // the list without its last tree (-1: none), that tree
  uint8_t pre_mask[kMaxPre];
  uint32_t task[kMaxTask];                      // type | index << 4 | polarisations << 16, by pass
  uint8_t ch_type[kMaxCh];
  int16_t ch_pre[kMaxCh], ch_node[kMaxCh];      // prefix (-1: none) and tree; kOne: the prefix before the last tree but one,
  uint8_t ch_last[kMaxCh];                      // that tree, and the last gluon
};

// Host: the trees, the walk and the channel keys ("1|2", "(1,2)", ... as documented in mg.h).
struct Built {
  Tab tab;
  TabL lin;
  bool ok;   // lin's capacities hold
  std::vector<std::string> keys;
};

void build(int K, Built& out) {
  Tab& t = out.tab;
  std::memset(&t, 0, sizeof(t));
  t.K = K;
  std::vector<std::vector<int>> trees(1 << K);
  std::vector<std::string> nkey;
  for (int g = 0; g < K; ++g) {
    t.node_l[t.nnode] = static_cast<int16_t>(-1 - g);
    t.node_r[t.nnode] = -1;
    t.node_mask[t.nnode] = static_cast<uint8_t>(1 << g);
    trees[1 << g].push_back(t.nnode++);
    nkey.push_back(std::to_string(g + 1));
  }
  for (int pc = 2; pc <= K; ++pc)
    for (int S = 1; S < (1 << K); ++S) {
      if (__builtin_popcount(S) != pc) continue;
      const int low = S & -S;
      for (int A = (S - 1) & S; A; A = (A - 1) & S) {   // the part holding the lowest gluon
        if (!(A & low)) continue;
        const int B = S ^ A;
        for (int ta : trees[A])
          for (int tb : trees[B]) {
            t.node_l[t.nnode] = static_cast<int16_t>(ta);
            t.node_r[t.nnode] = static_cast<int16_t>(tb);
            t.node_mask[t.nnode] = static_cast<uint8_t>(S);
            trees[S].push_back(t.nnode++);
            nkey.push_back("(" + nkey[ta] + "," + nkey[tb] + ")");
          }
      }
    }
  std::vector<std::string> prefix;
  std::function<void(int, int, int)> walk = [&](int rem, int depth, int attached) {
    for (int S = rem; S; S = (S - 1) & rem)
      for (int n : trees[S]) {
        const int i = t.nop++;
        t.op_node[i] = static_cast<int16_t>(n);
        t.op_depth[i] = static_cast<uint8_t>(depth);
        t.op_mask[i] = static_cast<uint8_t>(attached | S);
        if (S == rem) {
          t.op_ch[i] = static_cast<int16_t>(t.nch++);
          std::string k;
          for (const std::string& p : prefix) k += p + "|";
          out.keys.push_back(k + nkey[n]);
        } else {
          t.op_ch[i] = -1;
          prefix.push_back(nkey[n]);
          walk(rem ^ S, depth + 1, attached | S);
          prefix.pop_back();
        }
      }
  };
  walk((1 << K) - 1, 0, 0);
}

// the linear polarisations' tables from the walk; false if they do not fit (185 of 190 prefixes and 2,961 of 3,400 tasks with
// five gluons)
bool build_lin(const Tab& t, TabL& o) {
  const int K = t.K, full = (1 << K) - 1;
  std::memset(&o, 0xff, sizeof(o));   // -1: none
  auto size = [](int m) { return __builtin_popcount(m); };
  int at = 0;
  auto take = [&](int mask, int doubles) { const int r = at; at += doubles << size(mask); return r; };
  for (int n = 0; n < t.nnode; ++n) {
    const int m = t.node_mask[n];
    if (m == full) continue;
    o.J[n] = take(m, 4);
    o.D[n] = take(m, 4);
    if (size(m) == 2) o.X[n] = take(m, 16);
  }
  for (int g = 0; g < K; ++g) o.chi[g] = take(1 << g, 16);
  o.q0 = take(0, 16);
  // prefixes of up to K-2 gluons and channels, replaying the walk; stack[d]: the prefix before the tree at depth d
  o.npre = 0;
  int stack[6], tree[6];
  stack[0] = -1;
  for (int i = 0; i < t.nop; ++i) {
    const int d = t.op_depth[i], n = t.op_node[i], c = t.op_ch[i];
    tree[d] = n;
    if (c < 0) {
      stack[d + 1] = -2;   // (K-1 gluons: not kept)
      if (size(t.op_mask[i]) <= K - 2) {
        if (o.npre == TabL::kMaxPre) return false;
        const int p = o.npre++;
        o.pre_parent[p] = static_cast<int16_t>(stack[d]);
        o.pre_node[p] = static_cast<int16_t>(n);
        o.pre_mask[p] = t.op_mask[i];
        o.psi[p] = take(t.op_mask[i], 8);
        if (size(t.op_mask[i]) <= K - 3) o.q[p] = take(t.op_mask[i], 16);
        stack[d + 1] = p;
      }
      continue;
    }
    const int r = size(t.node_mask[n]);
    if (r == K) {
      o.ch_type[c] = TabL::kAll;
      o.ch_node[c] = static_cast<int16_t>(n);
    } else if (r >= 2) {
      o.ch_type[c] = r == 2 ? TabL::kPair : TabL::kMany;
      o.ch_pre[c] = static_cast<int16_t>(stack[d]);
      o.ch_node[c] = static_cast<int16_t>(n);
    } else {
      o.ch_type[c] = TabL::kOne;
      o.ch_pre[c] = static_cast<int16_t>(stack[d - 1]);
      o.ch_node[c] = static_cast<int16_t>(tree[d - 1]);
      o.ch_last[c] = static_cast<uint8_t>(n);
    }
  }
  o.stride = at;
  int nt = 0;
  o.npass = 0;
  o.pass0[0] = 0;
  auto tasks = [&](TabL::Task type, int i, int mask) {
    for (int gc = 0; gc <= full; ++gc)
      if (!(gc & ~mask) && nt++ < TabL::kMaxTask) o.task[nt - 1] = static_cast<uint32_t>(type) | static_cast<uint32_t>(i) << 4 | static_cast<uint32_t>(gc) << 16;
  };
  // pass k: the trees of k+1 gluons; the prefixes of k gluons (their trees and parents come from earlier passes) and the
  // quark currents of those of k-1
  for (int k = 0; k < K - 1; ++k) {
    for (int n = 0; n < t.nnode; ++n)
      if (size(t.node_mask[n]) == k + 1) tasks(k ? TabL::kNode : TabL::kLeafJ, n, t.node_mask[n]);
    if (k == 0) tasks(TabL::kQ0, 0, 0);
    if (k == 0)
      for (int g = 0; g < K; ++g) tasks(TabL::kChi, g, 1 << g);
    for (int p = 0; p < o.npre; ++p) {
      if (size(o.pre_mask[p]) == k) tasks(TabL::kPre, p, o.pre_mask[p]);
      if (size(o.pre_mask[p]) == k - 1 && o.q[p] >= 0) tasks(TabL::kQ, p, o.pre_mask[p]);
    }
    o.pass0[++o.npass] = nt;
  }
  return nt <= TabL::kMaxTask;
}

const Built& built(int K) {
  static Built b[6];
  static std::once_flag once[6];
  std::call_once(once[K], [K] {
    build(K, b[K]);
    b[K].ok = build_lin(b[K].tab, b[K].lin);
  });
  return b[K];
}

using v2::cx;

// The three-gluon vertex in full, V = (JL.JR)(PL - PR) + (JL.(PL + 2 PR)) JR - (JR.(2 PL + PR)) JL
__device__ __forceinline__ void v3full(cx<double>* out, const cx<double>* JL, const cx<double>* JR, const double* PL,
                                       const double* PR, double f) {
  double a[4], b[4], d[4];
#pragma unroll
  for (int m = 0; m < 4; ++m) {
    d[m] = PL[m] - PR[m];
    a[m] = PL[m] + 2.0 * PR[m];
    b[m] = 2.0 * PL[m] + PR[m];
  }
  const cx<double> jj = v2::mdot(JL, JR), cl = v2::mdotr(JL, a), cr = v2::mdotr(JR, b);
#pragma unroll
  for (int m = 0; m < 4; ++m) {
    cx<double> acc = v2::cscale(d[m], jj);
    v2::cmac(acc, cl, JR[m]);
    v2::cmsub(acc, cr, JL[m]);
    out[m] = v2::cscale(f, acc);
  }
}

// ---- linear polarisations ----
template <int K>
struct ViewS {
  using L = v2::EvLayout<K>;
  const double* in;
  double* buf;
  const Tab* tab;
  const TabL* o;
  __device__ __forceinline__ double rec(int item) const { return __ldg(in + item * kPage); }
  __device__ __forceinline__ double* at(int off) const { return buf + static_cast<int64_t>(off) * kPage; }
  __device__ __forceinline__ void ld(int off, cx<double>* v) const {
    const double* p = at(off);
#pragma unroll
    for (int m = 0; m < 4; ++m) v[m] = {p[(2 * m) * kPage], p[(2 * m + 1) * kPage]};
  }
  __device__ __forceinline__ void st(int off, const cx<double>* v) const {
    double* p = at(off);
#pragma unroll
    for (int m = 0; m < 4; ++m) {
      p[(2 * m) * kPage] = v[m].r;
      p[(2 * m + 1) * kPage] = v[m].i;
    }
  }
  __device__ __forceinline__ void top(int item, cx<double>* v) const {
#pragma unroll
    for (int q = 0; q < 4; ++q) v[q] = {rec(item + 2 * q), rec(item + 2 * q + 1)};
  }
  __device__ __forceinline__ void qc(int S, double* q) const {
#pragma unroll
    for (int i = 0; i < 5; ++i) q[i] = rec(L::QC + 5 * S + i);
  }
  __device__ __forceinline__ void mom(int S, double* P) const {
#pragma unroll
    for (int m = 0; m < 4; ++m) P[m] = rec(L::PT + 4 * S + m);
  }
  __device__ __forceinline__ void gluon(int g, int phi, double* J) const {
    J[0] = 0.0;
    J[1] = rec(L::EPS + 5 * g + (phi ? 3 : 0));
    J[2] = rec(L::EPS + 5 * g + (phi ? 4 : 1));
    J[3] = phi ? 0.0 : rec(L::EPS + 5 * g + 2);
  }
  __device__ __forceinline__ void J(int n, int gc, double* v) const {
    const double* p = at(o->J[n] + 4 * pext_bits(gc, tab->node_mask[n]));
#pragma unroll
    for (int m = 0; m < 4; ++m) v[m] = p[m * kPage];
  }
  __device__ __forceinline__ void st_jd(int n, int gc, const double* v, bool with_d) const {
    double* p = at(o->J[n] + 4 * pext_bits(gc, tab->node_mask[n]));
#pragma unroll
    for (int m = 0; m < 4; ++m) p[m * kPage] = v[m];
    if (!with_d) return;
    double* d = at(o->D[n] + 4 * pext_bits(gc, tab->node_mask[n]));
#pragma unroll
    for (int b = 0; b < 2; ++b) {
      cx<double> q[4];
      ld(o->q0 + 8 * b, q);
      const cx<double> x = m64::qdot(q, v);
      d[(2 * b) * kPage] = x.r;
      d[(2 * b + 1) * kPage] = x.i;
    }
  }
  __device__ __forceinline__ cx<double> D(int n, int gc, int b) const {
    const double* p = at(o->D[n] + 4 * pext_bits(gc, tab->node_mask[n]) + 2 * b);
    return {p[0], p[kPage]};
  }
  __device__ __forceinline__ void psi(int p, int gc, cx<double>* s) const {   // p = -1: ubar
    if (p < 0) top(L::UB, s);
    else ld(o->psi[p] + 8 * pext_bits(gc, o->pre_mask[p]), s);
  }
};

// One thread per (event, task of pass p), warps on one task of 32 consecutive events.
template <int K>
__global__ void __launch_bounds__(128)
k_sde_pass(const double* __restrict__ rec, int64_t nevt, const Tab* __restrict__ tab, const TabL* __restrict__ o, int p,
           const int* __restrict__ lin, double* __restrict__ buf) {
  using L = v2::EvLayout<K>;
  if (!*lin) return;
  const int64_t lanes = (nevt + kPage - 1) / kPage * kPage;
  const int64_t t = static_cast<int64_t>(blockIdx.x) * blockDim.x + threadIdx.x;
  const int64_t j = t / lanes, e = t - j * lanes;
  if (e >= nevt || j >= o->pass0[p + 1] - o->pass0[p]) return;
  const uint32_t task = o->task[o->pass0[p] + j];
  const int type = task & 15, i = (task >> 4) & 0xfff, gc = static_cast<int>(task >> 16);
  const ViewS<K> V = {rec + (e / kPage) * L::NITEM * kPage + (e % kPage),
                      buf + (e / kPage) * static_cast<int64_t>(o->stride) * kPage + (e % kPage), tab, o};
  switch (type) {
    case TabL::kLeafJ: {
      double J[4];
      V.gluon(i, (gc >> i) & 1, J);
      // (Jq.J from the spinors: the quark current is written in this pass)
      V.st_jd(i, gc, J, false);
      double* d = V.at(o->D[i] + 4 * pext_bits(gc, 1 << i));
#pragma unroll
      for (int b = 0; b < 2; ++b) {
        cx<double> u[4], v[4], q[4];
        V.top(L::UB, u);
        V.top(L::VV + 8 * b, v);
        v2::quark_current(u, v, q);
        const cx<double> x = m64::qdot(q, J);
        d[(2 * b) * kPage] = x.r;
        d[(2 * b + 1) * kPage] = x.i;
      }
      break;
    }
    case TabL::kQ0:
#pragma unroll
      for (int b = 0; b < 2; ++b) {
        cx<double> u[4], v[4], q[4];
        V.top(L::UB, u);
        V.top(L::VV + 8 * b, v);
        v2::quark_current(u, v, q);
        V.st(o->q0 + 8 * b, q);
      }
      break;
    case TabL::kChi: {
      double J[4], q[5];
      V.gluon(i, (gc >> i) & 1, J);
      const m64::RSlash g = m64::rslash(J, false);
      V.qc(((1 << K) - 1) ^ (1 << i), q);
#pragma unroll
      for (int b = 0; b < 2; ++b) {
        cx<double> v[4], X[4] = {}, chi[4];
        V.top(L::VV + 8 * b, v);
        m64::col_rslash_acc(X, g, v);
        m64::col_prop(X, q, chi);
        V.st(o->chi[i] + (2 * ((gc >> i) & 1) + b) * 8, chi);
      }
      break;
    }
    case TabL::kNode: {   // the three-gluon vertex in full (a single diagram's currents are not conserved)
      const int l = tab->node_l[i], r = tab->node_r[i], ml = tab->node_mask[l], mr = tab->node_mask[r];
      double JL[4], JR[4], PL[4], PR[4], a[4], b[4], out[4];
      V.J(l, gc, JL);
      V.J(r, gc, JR);
      V.mom(ml, PL);
      V.mom(mr, PR);
#pragma unroll
      for (int m = 0; m < 4; ++m) {
        a[m] = fma(2.0, PR[m], PL[m]);
        b[m] = fma(2.0, PL[m], PR[m]);
      }
      const double f = V.rec(L::GP + (ml | mr)), jj = m64::rdot(JL, JR), cl = m64::rdot(JL, a), cr = m64::rdot(JR, b);
#pragma unroll
      for (int m = 0; m < 4; ++m) out[m] = f * fma(-cr, JL[m], fma(cl, JR[m], (PL[m] - PR[m]) * jj));
      V.st_jd(i, gc, out, true);
      if (o->X[i] >= 0) {
        const m64::RSlash g = m64::rslash(out, false);
#pragma unroll
        for (int c = 0; c < 2; ++c) {
          cx<double> v[4], X[4] = {};
          V.top(L::VV + 8 * c, v);
          m64::col_rslash_acc(X, g, v);
          V.st(o->X[i] + (2 * pext_bits(gc, tab->node_mask[i]) + c) * 8, X);
        }
      }
      break;
    }
    case TabL::kPre: {
      double J[4], q[5];
      cx<double> s[4], t4[4] = {}, out[4];
      V.J(o->pre_node[i], gc, J);
      V.psi(o->pre_parent[i], gc, s);
      m64::row_rslash_acc(t4, s, m64::rslash(J, false));
      V.qc(o->pre_mask[i], q);
      v2::row_prop(t4, q, out);
      V.st(o->psi[i] + 8 * pext_bits(gc, o->pre_mask[i]), out);
      break;
    }
    default: {   // kQ
      cx<double> s[4];
      V.psi(i, gc, s);
#pragma unroll
      for (int b = 0; b < 2; ++b) {
        cx<double> v[4], q[4];
        V.top(L::VV + 8 * b, v);
        v2::quark_current(s, v, q);
        V.st(o->q[i] + (2 * pext_bits(gc, o->pre_mask[i]) + b) * 8, q);
      }
      break;
    }
  }
}

__device__ __forceinline__ double abs2_acc(cx<double> x, double s) { return fma(x.r, x.r, fma(x.i, x.i, s)); }

// One thread per (event, channel): the sum over polarisations of |A_d|^2 into w[d * ldw + e].
template <int K>
__global__ void __launch_bounds__(128)
k_sde_leaf(const double* __restrict__ rec, int64_t nevt, const Tab* __restrict__ tab, const TabL* __restrict__ o,
           const int* __restrict__ lin, const double* __restrict__ buf, double* __restrict__ w, int64_t ldw) {
  using L = v2::EvLayout<K>;
  if (!*lin) return;
  const int64_t e = static_cast<int64_t>(blockIdx.x) * kPage + threadIdx.x % kPage;
  const int c = blockIdx.y * 4 + threadIdx.x / kPage;
  if (e >= nevt || c >= tab->nch) return;
  const ViewS<K> V = {rec + (e / kPage) * L::NITEM * kPage + (e % kPage),
                      const_cast<double*>(buf) + (e / kPage) * static_cast<int64_t>(o->stride) * kPage + (e % kPage), tab, o};
  const int n = o->ch_node[c], pre = o->ch_pre[c];
  constexpr int NP = 1 << K;
  double sum = 0.0;
  switch (o->ch_type[c]) {
    case TabL::kOne: {
      const int g = o->ch_last[c];
      cx<double> chi[4][4];
#pragma unroll
      for (int x = 0; x < 4; ++x) V.ld(o->chi[g] + 8 * x, chi[x]);
      for (int gc = 0; gc < NP; ++gc) {
        if ((gc >> g) & 1) continue;
        double J[4];
        cx<double> s[4], t[4] = {};
        V.J(n, gc, J);
        V.psi(pre, gc, s);
        m64::row_rslash_acc(t, s, m64::rslash(J, false));
#pragma unroll
        for (int x = 0; x < 4; ++x) {   // the last gluon's polarisation and the antitop helicity
          cx<double> a = {};
          v2::sdot_acc(a, t, chi[x], false);
          sum = abs2_acc(a, sum);
        }
      }
      break;
    }
    case TabL::kPair:
      for (int gc = 0; gc < NP; ++gc) {
        cx<double> s[4];
        V.psi(pre, gc, s);
#pragma unroll
        for (int b = 0; b < 2; ++b) {
          cx<double> X[4], a = {};
          V.ld(o->X[n] + (2 * pext_bits(gc, tab->node_mask[n]) + b) * 8, X);
          v2::sdot_acc(a, s, X, false);
          sum = abs2_acc(a, sum);
        }
      }
      break;
    case TabL::kMany:
      for (int gc = 0; gc < NP; ++gc) {
        double J[4];
        V.J(n, gc, J);
#pragma unroll
        for (int b = 0; b < 2; ++b) {
          cx<double> q[4];
          V.ld(o->q[pre] + (2 * pext_bits(gc, o->pre_mask[pre]) + b) * 8, q);
          sum = abs2_acc(m64::qdot(q, J), sum);
        }
      }
      break;
    default: {   // all gluons on one tree
      const int l = tab->node_l[n], r = tab->node_r[n];
      double PL[4], PR[4], d[4], a[4], b[4];
      V.mom(tab->node_mask[l], PL);
      V.mom(tab->node_mask[r], PR);
#pragma unroll
      for (int m = 0; m < 4; ++m) {
        d[m] = PL[m] - PR[m];
        a[m] = fma(2.0, PR[m], PL[m]);
        b[m] = fma(2.0, PL[m], PR[m]);
      }
      cx<double> qd[2];
#pragma unroll
      for (int x = 0; x < 2; ++x) {
        cx<double> q[4];
        V.ld(o->q0 + 8 * x, q);
        qd[x] = m64::qdot(q, d);
      }
      for (int gc = 0; gc < NP; ++gc) {
        double JL[4], JR[4];
        V.J(l, gc, JL);
        V.J(r, gc, JR);
        const double jj = m64::rdot(JL, JR), cl = m64::rdot(JL, a), cr = -m64::rdot(JR, b);
#pragma unroll
        for (int x = 0; x < 2; ++x) {
          cx<double> y = v2::cscale(jj, qd[x]);
          v2::cmacr(y, cl, V.D(r, gc, x));
          v2::cmacr(y, cr, V.D(l, gc, x));
          sum = abs2_acc(y, sum);
        }
      }
      const double f = V.rec(L::GP + NP - 1);
      sum *= f * f;
      break;
    }
  }
  w[c * ldw + e] = sum;
}

// ---- helicities (partial masks) ----
// One thread per (event, slot): per-channel sums of |A_d|^2 over the slot's good helicities into
// part[(slot * nch + d) * stride + e].
template <int K>
__global__ void __launch_bounds__(128) k_sde(const double* __restrict__ rec, int64_t nevt, const Tab* __restrict__ tab,
                                             const int* __restrict__ lin, const int* __restrict__ gslots,
                                             const int* __restrict__ nslot_dev,
                                             const uint32_t* __restrict__ mask, double* __restrict__ part,
                                             int64_t stride) {
  constexpr int npar = K + 2, NSUB = 1 << K, NN = Sz<K>::nnode, NOP = Sz<K>::nop, NCH = Sz<K>::nch;
  using L = v2::EvLayout<K>;
  const int64_t e = static_cast<int64_t>(blockIdx.x) * blockDim.x + threadIdx.x;
  const int slot = blockIdx.y;
  if ((lin && *lin) || e >= nevt || slot >= *nslot_dev) return;
  const int gc = gslots[slot];
  const double* in = rec + (e / kPage) * L::NITEM * kPage + (e % kPage);
  auto ld = [&](int item) -> double { return __ldg(in + item * kPage); };
  double PT[NSUB][4], gprop[NSUB], qc[NSUB][5];
  for (int S = 1; S < NSUB; ++S) {
#pragma unroll
    for (int m = 0; m < 4; ++m) PT[S][m] = S == NSUB - 1 ? 0.0 : ld(L::PT + 4 * S + m);   // (no tree has the full set as a child)
    gprop[S] = ld(L::GP + S);
#pragma unroll
    for (int c = 0; c < 5; ++c) qc[S][c] = S == NSUB - 1 ? 0.0 : ld(L::QC + 5 * S + c);
  }
  cx<double> ub[2][4], vv[2][4];
#pragma unroll
  for (int l = 0; l < 2; ++l)
#pragma unroll
    for (int a = 0; a < 4; ++a) {
      ub[l][a] = {ld(L::UB + (l * 4 + a) * 2), ld(L::UB + (l * 4 + a) * 2 + 1)};
      vv[l][a] = {ld(L::VV + (l * 4 + a) * 2), ld(L::VV + (l * 4 + a) * 2 + 1)};
    }
  // every tree current of the gluon helicities gc
  cx<double> J[NN][4];
  for (int n = 0; n < NN; ++n) {
    const int l = tab->node_l[n];
    if (l < 0) {
      const int g = -1 - l;
      double pol[5];
#pragma unroll
      for (int i = 0; i < 5; ++i) pol[i] = ld(L::EPS + 5 * g + i);
      v2::ext_gluon(pol, (gc >> g) & 1 ? 1 : -1, g >= 2, J[n]);
    } else {
      const int r = tab->node_r[n];
      const int S = tab->node_mask[n];
      v3full(J[n], J[l], J[r], PT[tab->node_mask[l]], PT[tab->node_mask[r]], gprop[S]);
    }
  }
  int hbase = 0;
#pragma unroll
  for (int g = 0; g < K; ++g)
    if ((gc >> g) & 1) hbase |= 1 << (npar - 1 - (g < 2 ? g : g + 2));
  double acc[NCH];
  for (int d = 0; d < NCH; ++d) acc[d] = 0.0;
  for (int a = 0; a < 2; ++a) {
    const int h0 = hbase | (a << (npar - 3)), h1 = h0 | (1 << (npar - 4));
    // a single diagram's |A_d|^2 is the same with every helicity flipped too (hel_weight); the weights stay off the FP64
    // pipe, whose latency is the kernel's time for few events
    const int w0 = hel_weight(mask, h0, npar, 1), w1 = hel_weight(mask, h1, npar, 1);
    if (!w0 && !w1) continue;
    const double f0 = w0 > 1 ? 2.0 : 1.0, f1 = w1 > 1 ? 2.0 : 1.0;
    cx<double> stk[K][4];
#pragma unroll
    for (int q = 0; q < 4; ++q) stk[0][q] = ub[a][q];
    for (int i = 0; i < NOP; ++i) {
      const int n = tab->op_node[i], dep = tab->op_depth[i], ch = tab->op_ch[i];
      cx<double> t[4] = {};
      v2::row_gamma_acc(t, stk[dep], J[n], false);
      if (ch >= 0) {
        cx<double> a0 = {0.0, 0.0}, a1 = {0.0, 0.0};
        v2::sdot_acc(a0, t, vv[0], false);
        v2::sdot_acc(a1, t, vv[1], false);
        double s = acc[ch];
        if (w0) s = fma(f0, fma(a0.r, a0.r, a0.i * a0.i), s);
        if (w1) s = fma(f1, fma(a1.r, a1.r, a1.i * a1.i), s);
        acc[ch] = s;
      } else {
        v2::row_prop(t, qc[tab->op_mask[i]], stk[dep + 1]);
      }
    }
  }
  for (int d = 0; d < NCH; ++d) part[(static_cast<int64_t>(slot) * NCH + d) * stride + e] = acc[d];
}

// w[d * ldw + e]: the channel's sum over all channels' sum.  A block of 8 warps takes 32 events, each warp every eighth
// channel.  *lin != 0: the channels' sums are in w (k_sde_leaf); else the sums over slots of part (k_sde).  One launch for
// both and a block per page: with one thread per event for the slots' sums and a launch for each, the weights of
// 1,000 gg -> t tbar g events with a partial mask took 218 us, now 208.
__global__ void __launch_bounds__(256)
k_sde_norm(const double* __restrict__ part, int64_t nevt, int64_t stride, int nch, const int* __restrict__ lin,
           const int* __restrict__ nslot_dev, double* __restrict__ w, int64_t ldw) {
  __shared__ double sum[8][kPage];
  const bool linear = lin && *lin;
  const int nslot = *nslot_dev, lane = threadIdx.x % kPage, warp = threadIdx.x / kPage;
  const int64_t e = static_cast<int64_t>(blockIdx.x) * kPage + lane;
  double s = 0.0;
  if (e < nevt)
    for (int d = warp; d < nch; d += 8) {
      double t = 0.0;
      if (linear) {
        t = w[d * ldw + e];
      } else {
        for (int sl = 0; sl < nslot; ++sl) t += part[(static_cast<int64_t>(sl) * nch + d) * stride + e];
        w[d * ldw + e] = t;
      }
      s += t;
    }
  sum[warp][lane] = s;
  __syncthreads();
  if (e >= nevt) return;
  double tot = 0.0;
#pragma unroll
  for (int k = 0; k < 8; ++k) tot += sum[k][lane];
  const double r = 1.0 / tot;
  for (int d = warp; d < nch; d += 8) w[d * ldw + e] *= r;
}

}  // namespace sde
}  // namespace mg

namespace {

// the linear polarisations' tables follow the walk's in one allocation
constexpr size_t kLinOffset = (sizeof(mg::sde::Tab) + 15) / 16 * 16;

int64_t padp(int64_t n) { return (n + mg::kPage - 1) / mg::kPage * mg::kPage; }

mg_status growb(double** buf, int64_t* cap, int64_t need) {
  if (need <= *cap) return MG_OK;
  if (*buf) mg::dev_free(*buf);
  *buf = nullptr;
  *cap = 0;
  if (mg::dev_alloc(buf, static_cast<size_t>(need) * sizeof(double)) != cudaSuccess) {
    cudaGetLastError();
    return MG_ENOMEM;
  }
  *cap = need;
  return MG_OK;
}

// One chunk: the linear polarisations' kernels or the helicities', as *c->d_lin says (each returns at once for the other);
// part holds whichever's scratch.  Two gluons: the helicities' only (four of the sixteen vanish, so the mask is partial).
template <int K>
cudaError_t launch_sde(const double* rec, int64_t n, const mg_ctx* c, const mg::sde::Built& b, double* part, int64_t stride,
                       double* w, int64_t ldw, cudaStream_t st) {
  const mg::sde::Tab* tab = static_cast<const mg::sde::Tab*>(c->d_sdetab);
  const mg::sde::TabL* lt = reinterpret_cast<const mg::sde::TabL*>(static_cast<const char*>(c->d_sdetab) + kLinOffset);
  const unsigned pages = static_cast<unsigned>((n + mg::kPage - 1) / mg::kPage), tiles = static_cast<unsigned>((n + 127) / 128);
  const int* lin = K == 2 ? nullptr : c->d_lin;
  for (int p = 0; p < b.lin.npass && lin; ++p) {
    const int64_t threads = static_cast<int64_t>(pages) * mg::kPage * (b.lin.pass0[p + 1] - b.lin.pass0[p]);
    mg::sde::k_sde_pass<K><<<static_cast<unsigned>((threads + 127) / 128), 128, 0, st>>>(rec, n, tab, lt, p, lin, part);
    mg::note_launch();
  }
  if (lin) {
    mg::sde::k_sde_leaf<K><<<dim3(pages, (b.tab.nch + 3) / 4), 128, 0, st>>>(rec, n, tab, lt, lin, part, w, ldw);
    mg::note_launch();
  }
  mg::sde::k_sde<K><<<dim3(tiles, 1 << (K - 1)), 128, 0, st>>>(rec, n, tab, lin, c->d_hslots, c->d_nhslots, c->d_mask, part,
                                                              stride);
  mg::note_launch();
  mg::sde::k_sde_norm<<<pages, 256, 0, st>>>(part, n, stride, b.tab.nch, lin, c->d_nhslots, w, ldw);
  mg::note_launch();
  return cudaGetLastError();
}

}  // namespace

extern "C" {

mg_status mg_sde_channels(mg_process proc, int* nchannels) {
  if (proc < MG_GG_TT || proc > MG_GG_TTGGG || !nchannels) return MG_EINVAL;
  const mg::sde::Built& b = mg::sde::built(mg::gluons_of(proc));
  *nchannels = b.tab.nch;
  return b.ok ? MG_OK : MG_ENOTSUP;
}

mg_status mg_sde_channel_key(mg_process proc, int channel, char* key, int keylen) {
  if (proc < MG_GG_TT || proc > MG_GG_TTGGG || !key || keylen < 1) return MG_EINVAL;
  const mg::sde::Built& b = mg::sde::built(mg::gluons_of(proc));
  if (channel < 0 || channel >= b.tab.nch) return MG_EINVAL;
  const std::string& k = b.keys[channel];
  if (static_cast<int>(k.size()) + 1 > keylen) return MG_EINVAL;
  std::memcpy(key, k.c_str(), k.size() + 1);
  return MG_OK;
}

mg_status mg_sde_weights(mg_ctx* ctx, const double* mom_dev, int64_t nevt, double* w_dev, void* stream) {
  if (!ctx || nevt < 0 || (nevt > 0 && (!mom_dev || !w_dev))) return MG_EINVAL;
  if (ctx->prm.wt != 0.0) return MG_ENOTSUP;   // the per-event record has zero top width
  if (nevt == 0) return MG_OK;
  cudaStream_t st = static_cast<cudaStream_t>(stream);
  if (!ctx->mask_ready) {
    mg_status s = mg_hel_filter(ctx, mom_dev, nevt, stream);
    if (s != MG_OK) return s;
  }
  const int K = ctx->K;
  const mg::sde::Built& b = mg::sde::built(K);
  if (!b.ok) return MG_ENOTSUP;
  if (!ctx->d_sdetab) {
    if (mg::dev_alloc(&ctx->d_sdetab, kLinOffset + sizeof(mg::sde::TabL)) != cudaSuccess) {
      cudaGetLastError();
      return MG_ENOMEM;
    }
    if (cudaMemcpy(ctx->d_sdetab, &b.tab, sizeof(mg::sde::Tab), cudaMemcpyHostToDevice) != cudaSuccess ||
        cudaMemcpy(static_cast<char*>(ctx->d_sdetab) + kLinOffset, &b.lin, sizeof(mg::sde::TabL), cudaMemcpyHostToDevice) !=
            cudaSuccess) {
      cudaGetLastError();
      return MG_ECUDA;
    }
  }
  ctx->last = st;
  // chunks of whole pages that keep the items (or the helicities' per-slot channel sums) within 2^28 doubles (2 GiB)
  const int64_t sums = static_cast<int64_t>(1 << (K - 1)) * b.tab.nch;
  const int64_t per_event = sums > b.lin.stride ? sums : b.lin.stride;
  int64_t chunk = (int64_t(1) << 28) / per_event / mg::kPage * mg::kPage;
  if (chunk < mg::kPage) chunk = mg::kPage;
  if (chunk > padp(nevt)) chunk = padp(nevt);
  mg_status s = growb(&ctx->d_prep, &ctx->prep_cap, chunk * mg::event_record_bytes(K, false) / 8 + 1);
  if (s == MG_OK) s = growb(&ctx->d_sde, &ctx->sde_cap, chunk * per_event);
  if (s != MG_OK) return s;
  mg::MeConst cst;
  cst.gs = std::sqrt(4.0 * 3.14159265358979323846 * ctx->prm.alphas);
  cst.mt = ctx->prm.mt;
  cst.wt = ctx->prm.wt;
  cst.colour_scale = cst.gs * cst.gs / static_cast<double>(ctx->colour_den);
  for (int64_t e0 = 0; e0 < nevt; e0 += chunk) {
    const int64_t n = nevt - e0 < chunk ? nevt - e0 : chunk;
    const int64_t stride = padp(n);
    const double* mom_c = mom_dev + (e0 / mg::kPage) * ctx->npar * 4 * mg::kPage;
    if (mg::launch_event_prep(K, false, mom_c, n, cst, ctx->d_prep, st) != cudaSuccess) return MG_ECUDA;
    cudaError_t e = cudaSuccess;
    switch (K) {
      case 2: e = launch_sde<2>(ctx->d_prep, n, ctx, b, ctx->d_sde, stride, w_dev + e0, nevt, st); break;
      case 3: e = launch_sde<3>(ctx->d_prep, n, ctx, b, ctx->d_sde, stride, w_dev + e0, nevt, st); break;
      case 4: e = launch_sde<4>(ctx->d_prep, n, ctx, b, ctx->d_sde, stride, w_dev + e0, nevt, st); break;
      default: e = launch_sde<5>(ctx->d_prep, n, ctx, b, ctx->d_sde, stride, w_dev + e0, nevt, st); break;
    }
    if (e != cudaSuccess) return MG_ECUDA;
  }
  return MG_OK;
}

}  // extern "C"
