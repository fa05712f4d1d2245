// mg_tables64.cpp -- tables of the FP64 matrix elements of 3 to 5 gluons (mg_me64.cuh, mg_me64l.cuh; host side): the items
// shared between helicity or polarisation combinations and the tasks that compute them, the terms of the colour-ordered
// amplitudes, and the symmetry-adapted basis of the colour sum.
#include <algorithm>
#include <cstring>
#include <map>
#include <mutex>
#include <numeric>
#include <utility>
#include <vector>

#include "mg_internal.h"

namespace mg {

void build_tab64(int K, const Tables& t, const std::vector<int64_t>& num, Tab64& o) {
  std::memset(&o, 0, sizeof(o));
  o.K = K;
  const int top = 1 << (K - 1);
  auto nh = [&](int mask) { return 1 << __builtin_popcount(mask & (top - 1)); };
  auto fact = [](int n) { return factorial(n); };
  // ---- offsets: per helicity assignment (shared buffer) and for one assignment (a combination's own items) ----
  for (int own = 0; own < 2; ++own) {
    Tab64::Off& f = own ? o.loc : o.sh;
    int at = 0;
    auto take = [&](int mask, int entries) { const int r = at; at += 8 * entries * (own ? 1 : nh(mask)); return r; };
    std::memset(&f, 0xff, sizeof(f));   // -1: none
    for (int s = 0; s < t.nseq; ++s) {
      f.J[s] = take(t.seq_mask[s], 1);
      if (t.seq_len[s] >= 3) f.X[s] = take(t.seq_mask[s], 2);
    }
    for (int m = 1; m <= K - 2; ++m)
      for (int p = 0; p < t.ncol / fact(K - m); ++p) f.psi[m][p] = take(t.prefix_mask[p * fact(K - m)][m], 2);
    for (int g = 0; g < K; ++g) {
      f.chi[g] = take(1 << g, 2);
      f.qg[g] = take(1 << g, 4);
    }
    f.q0 = take(0, 4);
    for (int g = 0; g < K; ++g)
      for (int h = 0; h < K; ++h) {
        if (g == h) continue;
        f.z[g * kMaxGluons + h] = take(1 << g | 1 << h, 2);
        if (K == 5) f.qq[g * kMaxGluons + h] = take(1 << g | 1 << h, 4);
      }
    for (int i = 0; i < t.nfull; ++i) f.full[i] = take((1 << K) - 1, 1);
    if (K >= 4)
      for (int s = 0; s < t.nseq; ++s)
        for (int g = 0; g < K; ++g)
          if (t.seq_len[s] == 2 && !((t.seq_mask[s] >> g) & 1)) f.y[s][g] = take(t.seq_mask[s] | 1 << g, 2);
    (own ? o.nloc : o.stride) = at;
  }
  // ---- linear polarisations ----
  auto has_u = [&](int s) { return t.seq_len[s] <= (K == 3 ? 1 : 2); };
  auto has_dot = [&](int r, int s) { return !(t.seq_mask[r] & t.seq_mask[s]) && t.seq_len[r] + t.seq_len[s] <= K - 1; };
  for (int own = 0; own < 2; ++own) {
    Tab64::OffL& f = own ? o.locl : o.shl;
    int at = 0;
    auto take = [&](int mask, int doubles) {
      const int r = at;
      at += doubles * (own ? 1 : 1 << __builtin_popcount(mask));
      return r;
    };
    std::memset(&f, 0xff, sizeof(f));
    for (int s = 0; s < t.nseq; ++s) f.J[s] = take(t.seq_mask[s], 4);
    for (int m = 1; m <= K - 2; ++m)
      for (int p = 0; p < t.ncol / fact(K - m); ++p) {
        const int mask = t.prefix_mask[p * fact(K - m)][m];
        f.psi[m][p] = take(mask, 8);
        if (m <= K - 3) f.qv[m][p] = take(mask, 16);
      }
    for (int g = 0; g < K; ++g) {
      f.chi[g] = take(1 << g, 16);
      f.qg[g] = take(1 << g, 16);
    }
    f.q0 = take(0, 16);
    for (int g = 0; g < K; ++g)
      for (int h = 0; h < K; ++h) {
        if (g == h) continue;
        f.z[g * kMaxGluons + h] = take(1 << g | 1 << h, 16);
        if (K >= 4) f.qq[g * kMaxGluons + h] = take(1 << g | 1 << h, 16);
      }
    for (int i = 0; i < t.nfull; ++i) f.full[i] = take((1 << K) - 1, 4);
    for (int s = 0; s < t.nseq; ++s) {
      if (has_u(s)) f.u[s] = take(t.seq_mask[s], 16);
      if (t.seq_len[s] <= K - 2) f.d[s] = take(t.seq_mask[s], 4);
      for (int r = 0; r < s; ++r)
        if (has_dot(r, s)) f.dot[r][s] = f.dot[s][r] = take(t.seq_mask[r] | t.seq_mask[s], 1);
    }
    if (K == 5)
      for (int s = 0; s < t.nseq; ++s)
        for (int g = 0; g < K; ++g)
          if (t.seq_len[s] == 2 && !((t.seq_mask[s] >> g) & 1)) f.y[s][g] = take(t.seq_mask[s] | 1 << g, 16);
    if (own) o.nlocl = at;
    else if (at > o.stride) o.stride = at;
  }
  // ---- tasks ----
  int nt = 0, ntl = 0;
  o.nltask = o.nltaskl = 0;
  auto tasksl = [&](Tab64::Type type, int a, int b, int mask) {
    const uint32_t base = static_cast<uint32_t>(type) | static_cast<uint32_t>(a) << 4 | static_cast<uint32_t>(b) << 14;
    o.ltaskl[o.nltaskl++] = base;
    for (int gc = 0; gc < (1 << K); ++gc)
      if ((gc & ~mask) == 0) o.taskl[ntl++] = base | static_cast<uint32_t>(gc) << 20;
  };
  auto tasks = [&](Tab64::Type type, int a, int b, int mask) {
    if (type != Tab64::kY || K == 5) tasksl(type, a, b, mask);
    const uint32_t base = static_cast<uint32_t>(type) | static_cast<uint32_t>(a) << 4 | static_cast<uint32_t>(b) << 14;
    o.ltask[o.nltask++] = base;
    for (int gc = 0; gc < top; ++gc)
      if ((gc & ~mask) == 0) o.task[nt++] = base | static_cast<uint32_t>(gc) << 20;
  };
  auto seqs = [&](Tab64::Type type, int len) {
    for (int s = 0; s < t.nseq; ++s)
      if (t.seq_len[s] == len) tasks(type, s, 0, t.seq_mask[s]);
  };
  auto psis = [&](int m) {
    for (int p = 0; p < t.ncol / fact(K - m); ++p) tasks(Tab64::kPsi, p, m, t.prefix_mask[p * fact(K - m)][m]);
  };
  auto next_pass = [&] {
    o.pass0[++o.npass] = nt;
    o.pass0l[o.npass] = ntl;
  };
  for (int g = 0; g < K; ++g) tasks(Tab64::kJ1, g, 0, 1 << g);
  tasks(Tab64::kJq0, 0, 0, 0);
  psis(1);
  if (K == 3) next_pass();   // (three gluons: four short passes instead of two)
  for (int g = 0; g < K; ++g) tasks(Tab64::kChi, g, 0, 1 << g);
  // (linear polarisations) quark current and gluon, products of two currents of la and lb gluons
  auto us = [&](int len) {
    for (int s = 0; s < t.nseq; ++s)
      if (t.seq_len[s] == len && has_u(s)) tasksl(Tab64::kU, s, 0, t.seq_mask[s]);
  };
  auto dots = [&](int la, int lb) {
    for (int s = 0; s < t.nseq; ++s)
      for (int r = 0; r < s; ++r)
        if (t.seq_len[r] == la && t.seq_len[s] == lb && has_dot(r, s)) tasksl(Tab64::kDot, r, s, t.seq_mask[r] | t.seq_mask[s]);
  };
  if (K == 3) us(1);
  next_pass();
  seqs(Tab64::kSeq, 2);
  dots(1, 1);
  if (K >= 4) us(1);
  if (K >= 4)
    for (int g = 0; g < K; ++g)
      for (int h = 0; h < K; ++h)
        if (g != h) {
          if (K == 5) tasks(Tab64::kQQ, g, h, 1 << g | 1 << h);
          else tasksl(Tab64::kQQ, g, h, 1 << g | 1 << h);
        }
  next_pass();
  if (K >= 4) {
    seqs(Tab64::kSeq, 3);
    for (int s = 0; s < t.nseq; ++s)
      for (int g = 0; g < K; ++g)
        if (o.sh.y[s][g] >= 0) tasks(Tab64::kY, s, g, t.seq_mask[s] | 1 << g);
    psis(2);
    us(2);
    dots(1, 2);
    if (K == 5) dots(2, 2);
  }
  seqs(Tab64::kZ, 2);
  auto fulls = [&] {
    for (int i = 0; i < t.nfull; ++i) tasks(Tab64::kFull, i, 0, (1 << K) - 1);
    next_pass();
  };
  if (K == 3) {
    fulls();
  } else {
    next_pass();
    if (K == 5) {
      seqs(Tab64::kSeq, 4);
      psis(3);
      dots(1, 3);
      next_pass();
    }
    fulls();
  }
  // ---- terms of the amplitudes ----
  std::vector<int> p(K);
  std::iota(p.begin(), p.end(), 0);
  std::map<std::vector<int>, int> rank;
  std::vector<std::vector<int>> perms;
  do { rank[p] = static_cast<int>(perms.size()); perms.push_back(p); } while (std::next_permutation(p.begin(), p.end()));
  auto reversed = [&](int c, int i, int j) {   // the ordering with positions [i, j) reversed
    std::vector<int> q = perms[c];
    std::reverse(q.begin() + i, q.begin() + j);
    return rank.at(q);
  };
  for (int c = 0; c < t.ncol; ++c)
    if (t.full_idx[c] >= 0) {
      o.full_c[t.full_idx[c]] = static_cast<int16_t>(c);
      o.full_cr[t.full_idx[c]] = static_cast<int16_t>(reversed(c, 0, K));
    }
  auto entry = [&](int16_t* e, int c, int i, int j) {
    e[0] = static_cast<int16_t>(t.sub[c][i][j] >> 1);
    e[1] = static_cast<int16_t>(c);
    e[2] = static_cast<int16_t>(reversed(c, i, j));
  };
  int n1 = 0, n2 = 0, n3 = 0;
  for (int g = 0; g < K; ++g)
    for (int c = 0; c < t.ncol; ++c) {
      const std::vector<int>& s = perms[c];
      if (s[K - 1] == g && s[0] < s[K - 2]) entry(o.t1[n1++], c, 0, K - 1);
      if (K == 5 && s[0] == g && s[1] < s[4]) entry(o.t2[n2++], c, 1, 5);
    }
  if (K == 5)
    for (int g = 0; g < K; ++g)
      for (int h = 0; h < K; ++h) {
        if (g == h) continue;
        o.t3q[n3 / 3][0] = static_cast<int16_t>(g);
        o.t3q[n3 / 3][1] = static_cast<int16_t>(h);
        for (int c = 0; c < t.ncol; ++c) {
          const std::vector<int>& s = perms[c];
          if (s[0] == g && s[4] == h && s[1] < s[3]) entry(o.t3[n3++], c, 1, 4);
        }
      }
  for (int g = 0; g < t.ncol / 6; ++g)
    for (int i = 0; i < 6; ++i) {
      const int c = 6 * g + i;
      const std::vector<int>& s = perms[c];
      o.gz[g][i] = static_cast<int16_t>(s[K - 2] * kMaxGluons + s[K - 1]);
      if (K >= 4) {
        if (i < 3) o.g3[g][i] = static_cast<int16_t>(t.sub[c][K - 3][K] >> 1);
        const int y = i == 0 ? 0 : i == 1 ? 1 : i == 3 ? 2 : -1;
        if (y >= 0) {
          o.gy[g][y][0] = static_cast<int16_t>(t.sub[c][K - 3][K - 1] >> 1);
          o.gy[g][y][1] = static_cast<int16_t>(s[K - 1]);
        }
      }
    }
  // ---- colour sum in the symmetry-adapted basis (4 and 5 gluons) ----
  if (K < 4) return;
  auto image = [&](int c, int m) {   // ordering c with gluons 0,1 and 2,3 swapped and reversed as m's bits say
    std::vector<int> q = perms[c];
    for (int& g : q) {
      if ((m & 1) && g < 2) g = 1 - g;
      else if ((m & 2) && (g == 2 || g == 3)) g = 5 - g;
    }
    if (m & 4) std::reverse(q.begin(), q.end());
    return rank.at(q);
  };
  std::vector<bool> seen(t.ncol, false);
  // a basis combination: the jamp index it replaces, its jamps with their signs
  struct Vec { int at; std::vector<std::pair<int, int>> sign; int norm; };
  std::vector<Vec> blocks[8];
  for (int c = 0; c < t.ncol; ++c) {
    if (seen[c]) continue;
    int self = 0;   // the product of swaps that equals the reversal on this orbit, if any (never the identity)
    for (int m = 1; m < 4; ++m)
      if (image(c, m) == image(c, 4)) self = m;
    const int n = self ? 4 : 8;
    uint8_t* orb = self ? o.orb4[o.n4++] : o.orb8[o.n8++];
    for (int m = 0; m < n; ++m) {
      orb[m] = static_cast<uint8_t>(image(c, m));
      seen[orb[m]] = true;
    }
    for (int k = 0; k < n; ++k) {
      Vec v{orb[k], {}, n};
      for (int m = 0; m < n; ++m) v.sign.push_back({orb[m], __builtin_popcount(k & m) & 1 ? -1 : 1});
      blocks[self ? k | (__builtin_popcount(k & self) & 1) << 2 : k].push_back(v);
    }
  }
  o.nblk = 8;
  int nc = 0;
  for (int b = 0; b < 8; ++b) {
    o.blk_n[b] = static_cast<uint8_t>(blocks[b].size());
    for (size_t i = 0; i < blocks[b].size(); ++i) {
      o.blk[b][i] = static_cast<uint8_t>(blocks[b][i].at);
      for (size_t j = i; j < blocks[b].size(); ++j) {
        int64_t s = 0;
        for (const auto& x : blocks[b][i].sign)
          for (const auto& y : blocks[b][j].sign)
            s += num[static_cast<size_t>(x.first) * t.ncol + y.first] * (x.second * y.second);
        // (exact: an integer over a power of two)
        o.blk_c[nc++] = (i == j ? 1.0 : 2.0) * static_cast<double>(s) / (blocks[b][i].norm * blocks[b][j].norm);
      }
    }
  }
}

const Tab64& tab64_host(int K) {
  static Tab64 tabs[kMaxGluons + 1];
  static std::once_flag once[kMaxGluons + 1];
  std::call_once(once[K], [K] {
    Tables* t = new Tables;
    build_tables(K, *t);
    std::vector<int64_t> num;
    int64_t den;
    colour_matrix_exact(K, num, den);
    build_tab64(K, *t, num, tabs[K]);
    delete t;
  });
  return tabs[K];
}

}  // namespace mg
