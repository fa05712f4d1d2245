"""Host tables of the FP64 matrix elements of 3 to 5 gluons (mg_tables64.cpp), checked by a small C++ program: the colour
sum in the symmetry-adapted basis equals the full quadratic form exactly (integer jamps: every number involved is exact in
FP64), every item lies inside its buffer without overlapping another, and the task and amplitude tables stay in range."""
import os
import shutil
import subprocess

import pytest

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))
CSRC = os.path.join(ROOT, "paper_2210_11122_gb300", "csrc")

CHECKER = r"""
#include "mg_internal.h"
#include <cstdio>
#include <cstdlib>
#include <vector>
using namespace mg;
#define CHECK(x) do { if (!(x)) { std::printf("K=%d line %d: %s\n", K, __LINE__, #x); return 1; } } while (0)
static int nh(int K, int mask, bool own, bool lin) {
  return own ? 1 : 1 << __builtin_popcount(lin ? mask : mask & ((1 << (K - 1)) - 1));
}
int run(int K) {
  const Tab64& o = tab64_host(K);
  Tables* t = new Tables;
  build_tables(K, *t);
  std::vector<int64_t> num;
  int64_t den;
  colour_matrix_exact(K, num, den);
  const int n = t->ncol;
  if (K >= 4)
    for (int rep = 0; rep < 4; ++rep) {
      std::vector<double> A(n);
      unsigned s = 17 * rep + 5;
      for (double& x : A) { s = s * 1664525u + 1013904223u; x = static_cast<int>(s >> 24) - 128; }
      double ref = 0;
      for (int i = 0; i < n; ++i)
        for (int j = 0; j < n; ++j) ref += static_cast<double>(num[i * n + j]) * A[i] * A[j];
      auto sums = [&](const uint8_t* orb, int m) {
        for (int b = 1; b < m; b <<= 1)
          for (int k = 0; k < m; ++k)
            if (!(k & b)) { double x = A[orb[k]], y = A[orb[k | b]]; A[orb[k]] = x + y; A[orb[k | b]] = x - y; }
      };
      for (int i = 0; i < o.n8; ++i) sums(o.orb8[i], 8);
      for (int i = 0; i < o.n4; ++i) sums(o.orb4[i], 4);
      CHECK(8 * o.n8 + 4 * o.n4 == n);
      double got = 0;
      int c = 0;
      for (int b = 0; b < o.nblk; ++b)
        for (int i = 0; i < o.blk_n[b]; ++i)
          for (int j = i; j < o.blk_n[b]; ++j) got += o.blk_c[c++] * A[o.blk[b][i]] * A[o.blk[b][j]];
      CHECK(c <= 964 && got == ref);
    }
  // items: disjoint and inside the buffers (either basis, shared and own)
  for (int lin = 0; lin < 2; ++lin)
    for (int own = 0; own < 2; ++own) {
      const int size = own ? (lin ? o.nlocl : o.nloc) : o.stride;
      std::vector<char> u(size, 0);
      bool ok = true;
      auto item = [&](int off, int mask, int doubles) {
        if (off < 0) return;
        for (int i = 0; i < doubles * nh(K, mask, own, lin); ++i) {
          if (off + i >= size || u[off + i]) { ok = false; return; }
          u[off + i] = 1;
        }
      };
      const Tab64::Off& h = own ? o.loc : o.sh;
      const Tab64::OffL& l = own ? o.locl : o.shl;
      const int full = (1 << K) - 1;
      for (int s = 0; s < t->nseq; ++s) {
        const int m = t->seq_mask[s];
        if (lin) {
          item(l.J[s], m, 4); item(l.u[s], m, 16); item(l.d[s], m, 4);
          for (int r = 0; r < s && s < Tab64::kMaxSeq3; ++r) item(l.dot[r][s], m | t->seq_mask[r], 1);
        } else {
          item(h.J[s], m, 8); item(h.X[s], m, 16);
        }
        for (int g = 0; g < K; ++g) item(lin ? l.y[s][g] : h.y[s][g], m | 1 << g, 16);
      }
      int f = 1;
      for (int i = 2; i <= K; ++i) f *= i;
      for (int m = 1, per = f; m <= K - 2; ++m) {
        per /= K - m + 1;
        for (int p = 0; p < n / per; ++p) {
          const int mask = t->prefix_mask[p * per][m];
          if (lin) { item(l.psi[m][p], mask, 8); item(l.qv[m][p], mask, 16); }
          else item(h.psi[m][p], mask, 16);
        }
      }
      for (int g = 0; g < K; ++g) {
        item(lin ? l.chi[g] : h.chi[g], 1 << g, 16);
        item(lin ? l.qg[g] : h.qg[g], 1 << g, lin ? 16 : 32);
        for (int q = 0; q < K; ++q) {
          if (q == g) continue;
          const int i = g * kMaxGluons + q, m = 1 << g | 1 << q;
          item(lin ? l.z[i] : h.z[i], m, 16);
          item(lin ? l.qq[i] : h.qq[i], m, lin ? 16 : 32);
        }
      }
      item(lin ? l.q0 : h.q0, 0, lin ? 16 : 32);
      for (int i = 0; i < t->nfull; ++i) item(lin ? l.full[i] : h.full[i], full, lin ? 4 : 8);
      CHECK(ok);
    }
  CHECK(o.npass <= Tab64::kMaxPass && o.pass0[o.npass] <= Tab64::kMaxTask && o.pass0l[o.npass] <= Tab64::kMaxTaskL);
  CHECK(o.nltask <= Tab64::kMaxLTask && o.nltaskl <= Tab64::kMaxLTask);
  for (int i = 0; i < n / 2; ++i) CHECK(o.t1[i][1] != o.t1[i][2] && o.full_c[i] != o.full_cr[i]);
  delete t;
  return 0;
}
int main() { return run(3) || run(4) || run(5); }
"""


def test_tables_of_the_fp64_matrix_elements(tmp_path):
    cxx = shutil.which("g++") or shutil.which("c++")
    if not cxx:
        pytest.skip("no host C++ compiler")
    src = tmp_path / "check.cpp"
    src.write_text(CHECKER)
    exe = tmp_path / "check"
    cmd = [cxx, "-std=c++17", "-O1", "-I", CSRC, "-I", os.path.join(ROOT, "include"), str(src)]
    cmd += [os.path.join(CSRC, f) for f in ("mg_tables.cpp", "mg_tables64.cpp", "mg_colour.cpp")] + ["-o", str(exe)]
    r = subprocess.run(cmd, capture_output=True, text=True)
    assert r.returncode == 0, r.stderr[-3000:]
    r = subprocess.run([str(exe)], capture_output=True, text=True)
    assert r.returncode == 0, r.stdout
