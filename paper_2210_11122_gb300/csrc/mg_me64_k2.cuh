// mg_me64_k2.cuh -- the FP64 matrix element of g g -> t tbar in one kernel: record, amplitudes, colour sum and
// helicity sum of 32 events by a block of 4 warps.
//
// With two gluons the work is small (about 1,500 FP64 instructions per event), so what counts is how it is spread: the
// chain record -> amplitudes -> sum as three kernels of one long thread each took 57 us for one page of events (a
// warp issues an FP64 instruction every 64 cycles at best) and 100 us for 16,384; the slot threads formed column spinors
// that the other slots formed too.  Here every item is formed once per block and the warps share the chain
// (mg_me64.cuh's cut of the quark line, of which two gluons leave only the last piece): 18 us and 54 us.
//   1. record: warp 0 subset momenta and propagators, 1 polarisations, 2 ubar, 3 v;
//   2. chi(g, helicity, antitop helicity) (6) and the pair current (2), two per warp;
//   3. warp = (helicity of gluon 0, antitop helicity): A(01) = ubar . [(gamma.J_0) chi(1) + (gamma.J_01) v] and A(10) for
//      both top helicities, their colour sums, weighted (gluon 1 has helicity -1: hel_weight); 4. the sum of the warps.
#pragma once

#include "mg_me64.cuh"

namespace mg {
namespace m64 {

// An external gluon: J_0 = 0 and J_3 real, so gamma.J has real diagonal entries +- J_3; without the complex products with zeros of
// the general forms 16,384 events take 54 instead of 61 us (the same bits)
struct ExtGluon {
  cx<double> j1, j2;
  double j3;
  __device__ __forceinline__ cx<double> jm() const { return {j1.r + j2.i, j1.i - j2.r}; }   // J1 - i J2
  __device__ __forceinline__ cx<double> jp() const { return {j1.r - j2.i, j1.i + j2.r}; }
  // o += (gamma.J) v
  __device__ __forceinline__ void col_acc(cx<double>* o, const cx<double>* v) const {
    const cx<double> m = jm(), p = jp();
    v2::cmacr(o[0], -j3, v[2]); v2::cmsub(o[0], m, v[3]);
    v2::cmacr(o[1], j3, v[3]); v2::cmsub(o[1], p, v[2]);
    v2::cmacr(o[2], j3, v[0]); v2::cmac(o[2], m, v[1]);
    v2::cmac(o[3], p, v[0]); v2::cmacr(o[3], -j3, v[1]);
  }
  __device__ __forceinline__ cx<double> dot(const double* P) const {   // J . P, real P
    cx<double> r = {-(P[1] * j1.r), -(P[1] * j1.i)};
    v2::cmacr(r, -P[2], j2);
    r.r = fma(-P[3], j3, r.r);
    return r;
  }
};

// v3_acc of two external gluons
__device__ __forceinline__ void ext_v3(cx<double>* acc, const ExtGluon& L, const ExtGluon& R, const double* PL,
                                       const double* PR) {
  cx<double> jj = {}, cl = v2::cscale(2.0, L.dot(PR)), cr = v2::cscale(2.0, R.dot(PL));
  v2::cmsub(jj, L.j1, R.j1);
  v2::cmsub(jj, L.j2, R.j2);
  jj.r = fma(-L.j3, R.j3, jj.r);
#pragma unroll
  for (int m = 0; m < 4; ++m) acc[m] = v2::cscale(PL[m] - PR[m], jj);
  v2::cmac(acc[1], cl, R.j1); v2::cmsub(acc[1], cr, L.j1);
  v2::cmac(acc[2], cl, R.j2); v2::cmsub(acc[2], cr, L.j2);
  v2::cmacr(acc[3], R.j3, cl); v2::cmacr(acc[3], -L.j3, cr);
}

struct K2Block {
  using L = v2::EvLayout<2>;
  double rec[L::NBASE][kPage];
  double chi[6][8][kPage];     // (gluon 0, -), (gluon 0, +), (gluon 1, -), each antitop helicity
  double j2[2][8][kPage];      // pair current, helicity of gluon 0
  double part[4][kPage];
};

// me[e] of the 32 events of page `page`; all 128 threads of the block call it
__device__ __forceinline__ void k2_page(K2Block& s, const double* __restrict__ mom, int64_t nevt, int64_t page,
                                        const uint32_t* __restrict__ mask, const double* __restrict__ ctri,
                                        const MeConst& cst, double norm, double* __restrict__ me) {
  using L = K2Block::L;
  const int lane = threadIdx.x % kPage, warp = threadIdx.x / kPage;
  const int64_t e = page * kPage + lane;
  const bool live = e < nevt;
  auto rec = [&](int i) { return s.rec[i][lane]; };
  auto put = [&](int i, double v) { s.rec[i][lane] = v; };
  auto spinor = [&](int item, cx<double>* v) {
#pragma unroll
    for (int q = 0; q < 4; ++q) v[q] = {rec(item + 2 * q), rec(item + 2 * q + 1)};
  };
  auto ld = [&](const double (*p)[kPage], cx<double>* v) {
#pragma unroll
    for (int m = 0; m < 4; ++m) v[m] = {p[2 * m][lane], p[2 * m + 1][lane]};
  };
  auto st = [&](double (*p)[kPage], const cx<double>* v) {
#pragma unroll
    for (int m = 0; m < 4; ++m) {
      p[2 * m][lane] = v[m].r;
      p[2 * m + 1][lane] = v[m].i;
    }
  };
  auto gluon = [&](int g, int lam) -> ExtGluon {   // (ext_gluon, incoming)
    const int o = L::EPS + 5 * g;
    return {{lam > 0 ? -rec(o) : rec(o), -rec(o + 3)}, {lam > 0 ? -rec(o + 1) : rec(o + 1), -rec(o + 4)},
            lam > 0 ? -rec(o + 2) : rec(o + 2)};
  };
  if (live) {
    double p[4][4];
    const double* base = mom + page * 16 * kPage + lane;
#pragma unroll
    for (int i = 0; i < 4; ++i)
#pragma unroll
      for (int m = 0; m < 4; ++m) p[i][m] = __ldg(base + (i * 4 + m) * kPage);
    if (warp == 0) v2::record_subsets<2, double, 0, 4>(p, cst, put);
    else if (warp == 1) v2::record_pols<2, double>(p, put);
    else
#pragma unroll
      for (int l = 0; l < 2; ++l) {
        cx<double> w[4];
        if (warp == 2) v2::top_ubar<double>(p[2], cst.mt, l ? 1 : -1, w);
        else v2::top_v<double>(p[3], cst.mt, l ? 1 : -1, w);
#pragma unroll
        for (int a = 0; a < 4; ++a) {
          put((warp == 2 ? L::UB : L::VV) + (l * 4 + a) * 2, w[a].r);
          put((warp == 2 ? L::UB : L::VV) + (l * 4 + a) * 2 + 1, w[a].i);
        }
      }
  }
  __syncthreads();
  if (live) {
#pragma unroll
    for (int k = 0; k < 2; ++k) {
      const int t = warp + 4 * k;
      if (t < 6) {
        const int g = t >> 2, b = t & 1;
        cx<double> v[4], X[4] = {}, chi[4];
        spinor(L::VV + 8 * b, v);
        gluon(g, t >> 1 == 1 ? 1 : -1).col_acc(X, v);
        double q[5];
#pragma unroll
        for (int i = 0; i < 5; ++i) q[i] = rec(L::QC + 5 * (3 ^ (1 << g)) + i);
        col_prop(X, q, chi);
        st(s.chi[t], chi);
      } else {
        cx<double> acc[4];
        double P0[4], P1[4];
#pragma unroll
        for (int m = 0; m < 4; ++m) {
          P0[m] = rec(L::PT + 4 + m);
          P1[m] = rec(L::PT + 8 + m);
        }
        ext_v3(acc, gluon(0, t == 7 ? 1 : -1), gluon(1, -1), P0, P1);
        const double f = rec(L::GP + 3);
#pragma unroll
        for (int m = 0; m < 4; ++m) acc[m] = v2::cscale(f, acc[m]);
        st(s.j2[t - 6], acc);
      }
    }
  }
  __syncthreads();
  if (live) {
    const int g0 = warp >> 1, b = warp & 1;   // helicity of gluon 0, antitop helicity
    cx<double> J[4], v[4], z0[4], z1[4], c[4];
    ld(s.j2[g0], J);
    spinor(L::VV + 8 * b, v);
    v2::gamma_col(J, v, z0);
#pragma unroll
    for (int i = 0; i < 4; ++i) z1[i] = v2::cneg(z0[i]);
    ld(s.chi[4 + b], c);
    gluon(0, g0 ? 1 : -1).col_acc(z0, c);
    ld(s.chi[2 * g0 + b], c);
    gluon(1, -1).col_acc(z1, c);
    double total = 0.0;
#pragma unroll
    for (int a = 0; a < 2; ++a) {
      const int w = hel_weight(mask, g0 << 3 | a << 1 | b, 4, 1);
      if (!w) continue;
      cx<double> u[4], A[2] = {};
      spinor(L::UB + 8 * a, u);
      v2::sdot_acc(A[0], u, z0, false);
      v2::sdot_acc(A[1], u, z1, false);
      const double x = v2::colour_sum<2, double>(A, ctri);
      total += w > 1 ? x + x : x;
    }
    s.part[warp][lane] = total;
  }
  __syncthreads();
  if (warp == 0 && live)
    me[e] = ((s.part[0][lane] + s.part[1][lane]) + (s.part[2][lane] + s.part[3][lane])) * (cst.colour_scale * norm);
}

}  // namespace m64
}  // namespace mg
