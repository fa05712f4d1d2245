// mg_me64.cu -- launches of the FP64 matrix elements of 3 to 5 gluons (mg_me64.cuh): the passes that fill the
// shared items, and the slot kernel reading them.
#include <cuda_runtime.h>

#include "mg_internal.h"
#include "mg_kernels.h"
#include "mg_me64_k2.cuh"
#include "mg_me64l.cuh"

namespace mg {
namespace m64 {

// One thread per (event, task of pass p), warps on one task of 32 consecutive events; lin null or *lin != 0: the
// linear polarisations' tasks.  Bound by the FP64 pipe.
template <int K>
__global__ void __launch_bounds__(128)
k_pass64(const double* __restrict__ rec, int64_t nevt, const Tables* __restrict__ tab, const Tab64* __restrict__ t64,
         double gs, int p, const int* __restrict__ lin, double* __restrict__ share) {
  const int64_t npage = (nevt + kPage - 1) / kPage;
  const int64_t t = static_cast<int64_t>(blockIdx.x) * blockDim.x + threadIdx.x;
  const int64_t j = t / (npage * kPage);
  const int64_t e = t - j * npage * kPage;
  if (e >= nevt) return;
  const double* in = rec + (e / kPage) * v2::EvLayout<K>::NITEM * kPage + (e % kPage);
  double* buf = share + (e / kPage) * static_cast<int64_t>(t64->stride) * kPage + (e % kPage);
  if (!lin || *lin) {
    if (j >= t64->pass0l[p + 1] - t64->pass0l[p]) return;
    const uint32_t task = t64->taskl[t64->pass0l[p] + j];
    run_task_l<K, false>(ViewL<K, false>{in, buf, tab, t64, &t64->shl, static_cast<int>(task >> 20), gs}, task);
  } else {
    if (j >= t64->pass0[p + 1] - t64->pass0[p]) return;
    const uint32_t task = t64->task[t64->pass0[p] + j];
    run_task<K, false>(View<K, false>{in, buf, tab, t64, &t64->sh, static_cast<int>(task >> 20), gs}, task);
  }
}

// One block per (event tile of 32, block of the tile); slot_major: all blocks of a tile are dispatched together.
template <int K, bool AMP, bool LOCAL, int MINB>
__global__ void __launch_bounds__(kMeThreads, MINB)
k_me64(const double* __restrict__ rec, int64_t nevt, const Tables* __restrict__ tab, const Tab64* __restrict__ t64,
       const int* __restrict__ hslots, const int* __restrict__ nslot, const int* __restrict__ lin,
       const uint32_t* __restrict__ mask, const double* __restrict__ ctri, MeConst cst, double* __restrict__ out,
       int64_t stride, int slot_major, const double* __restrict__ share) {
  const unsigned tile = slot_major ? blockIdx.y : blockIdx.x;
  const int blk = static_cast<int>(slot_major ? blockIdx.x : blockIdx.y);
  thread64<K, AMP, LOCAL>(rec, nevt, tile, blk, tab, t64, hslots, nslot, lin, mask, ctri, cst, out, stride, share);
}

// One thread per (event, ordering, antitop helicity): the linear polarisations' amplitudes of k_me64<AMP> turned into the
// helicities'.  jout: as FP32 jamps, rows 2 * gluon helicities + antitop helicity (2^(K+1) per event), through shared
// memory so that a warp writes runs of 8 orderings; else in place (the same rows), with the weighted sum of |jamp|^2
// over the helicities in j2[(b * ncol + sigma) * stride + e].  Bound by its memory traffic, a few per cent of a call; it
// replaces amplitudes formed per helicity from complex currents: gg->ttggg + TC colour 5.35 vs 7.61 ms per 2,049 events,
// LHE choices of gg->ttgg 6.48 vs 8.69 ms per 32,768.
constexpr int kTrC = 4;   // orderings per block (one warp each)
template <int K, bool JAMPS>
__global__ void __launch_bounds__(32 * kTrC)
k_helicities(double* __restrict__ amp, int64_t nevt, const uint32_t* __restrict__ mask, float2* __restrict__ jout,
             double* __restrict__ j2, int64_t stride) {
  constexpr int NCOL = v2::Sizes<K>::ncol, NG = 1 << K;
  const int b = blockIdx.z, c = blockIdx.y * kTrC + threadIdx.x / 32, lane = threadIdx.x % 32;
  const int64_t e = static_cast<int64_t>(blockIdx.x) * 32 + lane;
  const bool live = e < nevt && c < NCOL;
  cx<double> a[NG];
  if (live) {
#pragma unroll
    for (int x = 0; x < NG; ++x) {
      const double* p = amp_at<K>(amp, e, 2 * x + b, c);
      a[x] = {p[0], p[kPage]};
    }
    to_helicities<K>(a);
  }
  if constexpr (JAMPS) {
    __shared__ float2 tile[32][kTrC];
    const int te = threadIdx.x / kTrC, tc = blockIdx.y * kTrC + threadIdx.x % kTrC;   // writer's event and ordering
    const int64_t we = static_cast<int64_t>(blockIdx.x) * 32 + te;
#pragma unroll
    for (int x = 0; x < NG; ++x) {
      if (live) tile[lane][threadIdx.x / 32] = make_float2(static_cast<float>(a[x].r), static_cast<float>(a[x].i));
      __syncthreads();
      if (we < nevt && tc < NCOL) jout[(we * (2 * NG) + 2 * x + b) * NCOL + tc] = tile[te][threadIdx.x % kTrC];
      __syncthreads();
    }
  } else if (live) {
    double s = 0.0;
#pragma unroll
    for (int x = 0; x < NG; ++x) {
      double* p = amp_at<K>(amp, e, 2 * x + b, c);
      p[0] = a[x].r;
      p[kPage] = a[x].i;
      const int w = hel_weight(mask, hel_of_row<K>(x, b), K + 2, 1);
      if (w) s = fma(static_cast<double>(w), fma(a[x].r, a[x].r, a[x].i * a[x].i), s);
    }
    j2[(b * NCOL + c) * stride + e] = s;
  }
}

// One thread per (event, row): the colour sum of the row's amplitudes, out[row * stride + e].
template <int K>
__global__ void __launch_bounds__(kMeThreads, 4)
k_colour64(double* __restrict__ amp, int64_t nevt, const Tab64* __restrict__ t64, const double* __restrict__ ctri,
           double scale, double* __restrict__ out, int64_t stride) {
  constexpr int NCOL = v2::Sizes<K>::ncol;
  const int64_t e = static_cast<int64_t>(blockIdx.x) * kPage + threadIdx.x % kPage;
  const int row = blockIdx.y * (kMeThreads / kPage) + threadIdx.x / kPage;
  if (e >= nevt) return;
  cx<double> A[NCOL];
  const double* p = amp_at<K>(amp, e, row, 0);
  for (int c = 0; c < NCOL; ++c) A[c] = {p[2 * c * kPage], p[(2 * c + 1) * kPage]};
  out[row * stride + e] = colour_sum64<K>(A, t64, ctri) * scale;
}

template <int K>
static cudaError_t launch_pass(const double* rec, int64_t nevt, const Tables* tab, const Tab64* t64, const MeConst& cst,
                               const int* lin, double* share, cudaStream_t st) {
  const Tab64& h = tab64_host(K);
  const int64_t lanes = (nevt + kPage - 1) / kPage * kPage;
  if (lanes <= 0) return cudaSuccess;
  for (int p = 0; p < h.npass; ++p) {
    // (the basis is known on the device only: enough threads for either)
    const int nh = h.pass0[p + 1] - h.pass0[p], nl = h.pass0l[p + 1] - h.pass0l[p], n = !lin || nl > nh ? nl : nh;
    { k_pass64<K><<<static_cast<unsigned>((lanes * n + 127) / 128), 128, 0, st>>>(rec, nevt, tab, t64, cst.gs, p, lin,
                                                                                  share); mg::note_launch(); }
    const cudaError_t e = cudaGetLastError();
    if (e != cudaSuccess) return e;
  }
  return cudaSuccess;
}

template <int K, bool AMP>
static cudaError_t launch_k(const double* rec, int64_t nevt, const Tables* tab, const Tab64* t64, const int* hslots,
                            const int* nslot, const int* lin, const uint32_t* mask, const double* ctri,
                            const MeConst& cst, double* out, int64_t stride, MeShape shape, const double* share,
                            cudaStream_t st) {
  constexpr unsigned NBLK = 1 << (K - 1);
  const unsigned tiles = static_cast<unsigned>((nevt + kPage - 1) / kPage);
  if (tiles == 0) return cudaSuccess;
  if (!share && (tab64_host(K).nloc > Loc<K>::n || tab64_host(K).nlocl > LocL<K>::n)) return cudaErrorInvalidValue;
  // (a grid's y extent is limited to 65,535: event tiles beyond it go to x)
  const int sm = shape.slot_major && tiles <= 65535 ? 1 : 0;
  const dim3 grid = sm ? dim3(NBLK, tiles) : dim3(tiles, NBLK);
  if (share)
    k_me64<K, AMP, false, 4><<<grid, kMeThreads, 0, st>>>(rec, nevt, tab, t64, hslots, nslot, lin, mask, ctri, cst, out, stride,
                                                          sm, share);
  else
    k_me64<K, AMP, true, 2><<<grid, kMeThreads, 0, st>>>(rec, nevt, tab, t64, hslots, nslot, lin, mask, ctri, cst, out, stride,
                                                         sm, nullptr);
  mg::note_launch();
  return cudaGetLastError();
}

template <int K>
static cudaError_t launch_hel_k(double* amp, int64_t nevt, const Tab64* t64, const uint32_t* mask, const double* ctri,
                                double scale, double* out, int64_t stride, float2* jout, double* j2, cudaStream_t st) {
  const unsigned tiles = static_cast<unsigned>((nevt + kPage - 1) / kPage);
  if (tiles == 0) return cudaSuccess;
  const dim3 grid(tiles, (v2::Sizes<K>::ncol + kTrC - 1) / kTrC, 2);
  if (jout)
    k_helicities<K, true><<<grid, 32 * kTrC, 0, st>>>(amp, nevt, mask, jout, nullptr, stride);
  else
    k_helicities<K, false><<<grid, 32 * kTrC, 0, st>>>(amp, nevt, mask, nullptr, j2, stride);
  mg::note_launch();
  if (!jout) {
    k_colour64<K><<<dim3(tiles, (2 << K) / (kMeThreads / kPage)), kMeThreads, 0, st>>>(amp, nevt, t64, ctri, scale, out, stride);
    mg::note_launch();
  }
  return cudaGetLastError();
}

}  // namespace m64

namespace m64 {
__global__ void __launch_bounds__(kMeThreads, 4)
k_me64_k2(const double* __restrict__ mom, int64_t nevt, const uint32_t* __restrict__ mask, const double* __restrict__ ctri,
          MeConst cst, double norm, double* __restrict__ me) {
  __shared__ K2Block s;
  k2_page(s, mom, nevt, blockIdx.x, mask, ctri, cst, norm, me);
}
}  // namespace m64

cudaError_t launch_me64_k2(const double* mom, int64_t nevt, const uint32_t* mask, const double* ctri, const MeConst& cst,
                           double norm, double* me, cudaStream_t st) {
  const unsigned pages = static_cast<unsigned>((nevt + kPage - 1) / kPage);
  if (pages == 0) return cudaSuccess;
  { m64::k_me64_k2<<<pages, kMeThreads, 0, st>>>(mom, nevt, mask, ctri, cst, norm, me); mg::note_launch(); }
  return cudaGetLastError();
}

cudaError_t launch_pass64(int K, const double* rec, int64_t nevt, const Tables* tab, const Tab64* t64, const MeConst& cst,
                          const int* lin, double* share, cudaStream_t st) {
  switch (K) {
    case 3: return m64::launch_pass<3>(rec, nevt, tab, t64, cst, lin, share, st);
    case 4: return m64::launch_pass<4>(rec, nevt, tab, t64, cst, lin, share, st);
    case 5: return m64::launch_pass<5>(rec, nevt, tab, t64, cst, lin, share, st);
    default: return cudaErrorInvalidValue;
  }
}

cudaError_t launch_me64(int K, const double* rec, int64_t nevt, const Tables* tab, const Tab64* t64, const int* hslots,
                        const int* nslot, const int* lin, const uint32_t* mask, const double* ctri, const MeConst& cst,
                        double* out, int64_t stride, MeShape shape, const double* share, cudaStream_t st) {
#define MG_64_CASE(KK)                                                                                                   \
  case KK:                                                                                                               \
    if (!lin) return m64::launch_k<KK, true>(rec, nevt, tab, t64, hslots, nslot, lin, mask, ctri, cst, out, stride, shape, \
                                             share, st);                                                                 \
    return m64::launch_k<KK, false>(rec, nevt, tab, t64, hslots, nslot, lin, mask, ctri, cst, out, stride, shape, share, st);
  switch (K) {
    MG_64_CASE(3)
    MG_64_CASE(4)
    MG_64_CASE(5)
    default: return cudaErrorInvalidValue;
  }
#undef MG_64_CASE
}

cudaError_t launch_helicities(int K, double* amp, int64_t nevt, const Tab64* t64, const uint32_t* mask, const double* ctri,
                              double scale, double* out, int64_t stride, float2* jout, double* j2, cudaStream_t st) {
  switch (K) {
    case 3: return m64::launch_hel_k<3>(amp, nevt, t64, mask, ctri, scale, out, stride, jout, j2, st);
    case 4: return m64::launch_hel_k<4>(amp, nevt, t64, mask, ctri, scale, out, stride, jout, j2, st);
    case 5: return m64::launch_hel_k<5>(amp, nevt, t64, mask, ctri, scale, out, stride, jout, j2, st);
    default: return cudaErrorInvalidValue;
  }
}

}  // namespace mg
