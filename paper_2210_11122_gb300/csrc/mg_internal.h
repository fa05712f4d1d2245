// mg_internal.h -- declarations shared by the engine's own translation units.
#pragma once

#include <cstdint>
#include <vector>

#include "../../include/mg.h"

namespace mg {

constexpr int kMaxGluons = 5;      // g g -> t tbar g g g
constexpr int kMaxNcol = 120;      // 5!
constexpr int kMaxSeq = 105;       // canonical gluon sequences of length 1..K-1 for K = 5
constexpr int kPage = 32;          // AoSoA page: events per page

// Count one kernel launch of this library (process-wide, thread-safe; read by mg_kernel_launches).
void note_launch();

inline int gluons_of(mg_process p) { return static_cast<int>(p) + 2; }
inline int npar_of(mg_process p) { return static_cast<int>(p) + 4; }
inline int factorial(int n) { int f = 1; for (int i = 2; i <= n; ++i) f *= i; return f; }

// ----------------------------------------------------------------------------------------
// Exact colour matrix of one quark line + K gluons (mg_colour.cpp):
// C(sigma,tau) = Tr(T^sigma (T^tau)^dagger) = num / den.
// ----------------------------------------------------------------------------------------
void colour_matrix_exact(int K, std::vector<int64_t>& num, int64_t& den);

// ----------------------------------------------------------------------------------------
// Recursion tables for K gluons (mg_tables.cpp).  A "slot reference" packs a canonical gluon
// sequence slot and a sign: ref = (slot << 1) | negative.  Canonical sequences of length >= 2
// have seq[0] < seq[L-1]; the reversed sequence carries the sign (-1)^(L+1) (reflection
// identity of colour-ordered gluon currents).
// ----------------------------------------------------------------------------------------
struct Tables {
  int K, ncol, nseq;
  // canonical sequences: length, subset mask; splits into (L,R) and (A,B,C) as slot refs
  uint8_t seq_len[kMaxSeq];
  uint8_t seq_mask[kMaxSeq];
  int16_t seq_v3[kMaxSeq][kMaxGluons - 1][2];
  int16_t seq_v4[kMaxSeq][6][3];
  uint8_t seq_nv3[kMaxSeq], seq_nv4[kMaxSeq];
  // permutations sigma in lexicographic order (= jamp index)
  uint8_t perm[kMaxNcol][kMaxGluons];
  uint8_t lcp[kMaxNcol];                        // common prefix length with the previous sigma
  uint8_t prefix_mask[kMaxNcol][kMaxGluons];    // mask of sigma[0..m) for m = 0..K-1
  // sub[c][j][m] = slot ref of sigma[j..m), 0 <= j < m <= K, (j, m) != (0, K)
  int16_t sub[kMaxNcol][kMaxGluons][kMaxGluons + 1];
  // full-length sigma: canonical flag, index into the full-current table, its splits
  int16_t full_idx[kMaxNcol];                   // >= 0: canonical, own index; < 0: -(idx of reverse)-1
  int nfull;
  int16_t full_v3[kMaxNcol / 2][kMaxGluons - 1][2];
  int16_t full_v4[kMaxNcol / 2][6][3];
  uint8_t full_nv3[kMaxNcol / 2], full_nv4[kMaxNcol / 2];
  uint8_t full_split_mask[kMaxNcol / 2][kMaxGluons - 1];   // mask of the left part of each V3 split
};

// helicity bits of the gluons in mask, packed (bit g of gc -> the rank of g among mask's bits), and back
inline constexpr int pext_bits(int gc, int mask) {
  int r = 0, k = 0;
  for (int g = 0; g < kMaxGluons; ++g)
    if ((mask >> g) & 1) r |= ((gc >> g) & 1) << k++;
  return r;
}
inline constexpr int pdep_bits(int h, int mask) {
  int r = 0, k = 0;
  for (int g = 0; g < kMaxGluons; ++g)
    if ((mask >> g) & 1) r |= ((h >> k++) & 1) << g;
  return r;
}

void build_tables(int K, Tables& t);

// ----------------------------------------------------------------------------------------
// FP64 matrix elements of 3 to 5 gluons (mg_me64.cuh): the items shared between gluon-helicity combinations, the
// tasks that compute them, and the terms of the colour-ordered amplitudes.  Offsets are in doubles per event; an item
// of a gluon set holds one entry per helicity assignment of the set without gluon K-1 (which has helicity -1), in
// pext_bits order; entries are 8 doubles (4 complex) times what the comment says.
// ----------------------------------------------------------------------------------------
struct Tab64 {
  enum Type { kJ1, kJq0, kChi, kPsi, kSeq, kZ, kY, kFull, kU, kDot, kQQ };
  static constexpr int kMaxTask = 2500, kMaxTaskL = 5800, kMaxLTask = 480, kMaxPass = 6;
  static constexpr int kMaxSeq3 = 45;      // canonical sequences of at most 3 gluons
  struct Off {
    int J[kMaxSeq];                        // current of a canonical sequence (1)
    int X[kMaxSeq];                        // (gamma.J) v, three or more gluons (antitop helicity: 2); -1: none
    int psi[kMaxGluons - 1][60];           // row spinor after m gluons, prefix = ordering / (K - m)! (top helicity: 2)
    int chi[kMaxGluons];                   // column spinor before the last gluon (2)
    int qg[kMaxGluons];                    // ubar gamma^mu chi(g) (2 top + antitop: 4)
    int q0;                                // ubar gamma^mu v (4)
    int z[kMaxGluons * kMaxGluons];        // last two gluons (2)
    int y[kMaxSeq][kMaxGluons];            // (gamma.J_pair) chi(g) (2); -1: none
    int full[kMaxNcol / 2];                // ubar gamma^mu v times a canonical full current (4 complex numbers)
    int qq[kMaxGluons * kMaxGluons];       // psi_1(g) gamma^mu chi(h), 5 gluons (4)
  };
  // Linear gluon polarisations (mg_me64l.cuh): one entry per polarisation combination of the whole gluon set; currents
  // are real (4 doubles), the others 8 doubles times what the comment says, top helicity -1 only.
  struct OffL {
    int J[kMaxSeq];
    int psi[kMaxGluons - 1][60];           // (1)
    int qv[kMaxGluons - 1][60];            // psi_m gamma^mu v, m <= K - 3 (antitop helicity: 2)
    int chi[kMaxGluons], qg[kMaxGluons];   // (2)
    int q0;                                // (2)
    int z[kMaxGluons * kMaxGluons];        // (2)
    int y[kMaxSeq][kMaxGluons];            // 5 gluons (2)
    int full[kMaxNcol / 2];                // 2 complex numbers (4 doubles)
    int u[kMaxSeq];                        // one and two gluons: ubar gamma^mu v joined to J by a three-gluon vertex (2)
    int d[kMaxSeq];                        // up to K-2 gluons: ubar gamma^mu v . J, 2 complex numbers (4 doubles)
    int dot[kMaxSeq3][kMaxSeq3];           // g J . J' of disjoint sequences of together at most K-1 gluons (1 double)
    int qq[kMaxGluons * kMaxGluons];       // 4 and 5 gluons (2)
  };
  int K, stride;                           // doubles per event of the shared buffer (either basis)
  int nloc, nlocl;                         // doubles of one combination's own items
  Off sh, loc;
  OffL shl, locl;
  int npass, pass0[kMaxPass + 1];
  uint32_t task[kMaxTask];                 // type | a << 4 | b << 14 | gluon helicities << 20, by pass
  int pass0l[kMaxPass + 1];
  uint32_t taskl[kMaxTaskL];               // the same for linear polarisations
  int nltaskl;
  uint32_t ltaskl[kMaxLTask];
  int nltask;
  uint32_t ltask[kMaxLTask];               // the same tasks without helicities, in an order that respects dependences
  int16_t full_c[kMaxNcol / 2], full_cr[kMaxNcol / 2];   // orderings of a full current and of its reversal
  int16_t t1[kMaxNcol / 2][3];             // by last gluon: sequence of K-1, ordering, ordering reversed in the sequence
  int16_t t2[kMaxNcol / 2][3];             // 5 gluons, by first gluon: sequence of the last 4, ordering, reversed
  int16_t t3[kMaxNcol / 2][3];             // 5 gluons, by (first, last) gluon: sequence of the middle 3, ordering, reversed
  int16_t t3q[kMaxGluons * (kMaxGluons - 1)][2];   // t3's (first, last) gluons, three entries each
  int16_t g3[kMaxNcol / 6][3];             // six orderings with a common prefix of K-3: sequences xyz, xzy, yxz
  int16_t gy[kMaxNcol / 6][3][2];          // (pair, last): (xy, z), (xz, y), (yz, x)
  int16_t gz[kMaxNcol / 6][6];             // last two gluons, first * 5 + second, of the six orderings
  // Colour sum of 4 and 5 gluons in a basis that block-diagonalises the colour matrix C.  C is unchanged when both
  // orderings have gluons 0 and 1 swapped, gluons 2 and 3 swapped, or are reversed; on an orbit of these three commuting
  // involutions (8 orderings, or 4 where the reversal equals a product of swaps) the sums with signs (-1)^(k & m) have
  // no C entries between different sign patterns k.  Orbit member m = bit 0: 0 <-> 1, bit 1: 2 <-> 3, bit 2:
  // reversed; the combination of pattern k replaces the jamp of member k.
  int n8, n4, nblk;                        // orbits of 8 and of 4; blocks
  uint8_t orb8[14][8], orb4[2][4];         // jamp indices
  uint8_t blk_n[8], blk[8][16];            // a block's size and jamp indices
  double blk_c[964];                       // its packed upper triangle (off-diagonal doubled), block after block
};

// num: the integer colour matrix (colour_matrix_exact)
void build_tab64(int K, const Tables& t, const std::vector<int64_t>& num, Tab64& o);
const Tab64& tab64_host(int K);            // built once per process (K = 3..5)

}  // namespace mg
