// mg_me64.cu -- launches of the FP64 matrix elements of 3 to 5 gluons (mg_me64.cuh): the passes that fill the
// shared items, and the slot kernel reading them.
#include <cuda_runtime.h>

#include "mg_internal.h"
#include "mg_kernels.h"
#include "mg_me64l.cuh"

namespace mg {
namespace m64 {

// One thread per (event, task of pass p), warps on one task of 32 consecutive events; *lin != 0 (lin may be null): the
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
  if (lin && *lin) {
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
template <int K, int MODE, bool LOCAL, int MINB>
__global__ void __launch_bounds__(kMeThreads, MINB)
k_me64(const double* __restrict__ rec, int64_t nevt, const Tables* __restrict__ tab, const Tab64* __restrict__ t64,
       const int* __restrict__ hslots, const int* __restrict__ nslot, const int* __restrict__ lin,
       const uint32_t* __restrict__ mask, const double* __restrict__ ctri, MeConst cst, double* __restrict__ out,
       int64_t stride, float2* __restrict__ jout, int slot_major, const double* __restrict__ share, double* __restrict__ j2) {
  const unsigned tile = slot_major ? blockIdx.y : blockIdx.x;
  const int blk = static_cast<int>(slot_major ? blockIdx.x : blockIdx.y);
  thread64<K, MODE, LOCAL>(rec, nevt, tile, blk, tab, t64, hslots, nslot, lin, mask, ctri, cst, out, stride, jout, share, j2);
}

template <int K>
static cudaError_t launch_pass(const double* rec, int64_t nevt, const Tables* tab, const Tab64* t64, const MeConst& cst,
                               const int* lin, double* share, cudaStream_t st) {
  const Tab64& h = tab64_host(K);
  const int64_t lanes = (nevt + kPage - 1) / kPage * kPage;
  if (lanes <= 0) return cudaSuccess;
  for (int p = 0; p < h.npass; ++p) {
    // (the basis is known on the device only: enough threads for either)
    const int nh = h.pass0[p + 1] - h.pass0[p], nl = h.pass0l[p + 1] - h.pass0l[p], n = lin && nl > nh ? nl : nh;
    { k_pass64<K><<<static_cast<unsigned>((lanes * n + 127) / 128), 128, 0, st>>>(rec, nevt, tab, t64, cst.gs, p, lin,
                                                                                  share); mg::note_launch(); }
    const cudaError_t e = cudaGetLastError();
    if (e != cudaSuccess) return e;
  }
  return cudaSuccess;
}

template <int K, int MODE>
static cudaError_t launch_k(const double* rec, int64_t nevt, const Tables* tab, const Tab64* t64, const int* hslots,
                            const int* nslot, const int* lin, const uint32_t* mask, const double* ctri,
                            const MeConst& cst, double* out, int64_t stride, float2* jout, MeShape shape,
                            const double* share, double* j2, cudaStream_t st) {
  constexpr unsigned NBLK = 1 << (K - 1);
  const unsigned tiles = static_cast<unsigned>((nevt + kPage - 1) / kPage);
  if (tiles == 0) return cudaSuccess;
  if (!share && (tab64_host(K).nloc > Loc<K>::n || tab64_host(K).nlocl > LocL<K>::n)) return cudaErrorInvalidValue;
  // (a grid's y extent is limited to 65,535: event tiles beyond it go to x)
  const int sm = shape.slot_major && tiles <= 65535 ? 1 : 0;
  const dim3 grid = sm ? dim3(NBLK, tiles) : dim3(tiles, NBLK);
  if (share)
    k_me64<K, MODE, false, 4><<<grid, kMeThreads, 0, st>>>(rec, nevt, tab, t64, hslots, nslot, lin, mask, ctri, cst, out, stride,
                                                           jout, sm, share, j2);
  else
    k_me64<K, MODE, true, 2><<<grid, kMeThreads, 0, st>>>(rec, nevt, tab, t64, hslots, nslot, lin, mask, ctri, cst, out, stride,
                                                          jout, sm, nullptr, j2);
  mg::note_launch();
  return cudaGetLastError();
}

}  // namespace m64

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
                        double* out, int64_t stride, float2* jout, MeShape shape, const double* share, double* j2,
                        cudaStream_t st) {
#define MG_64_CASE(KK)                                                                                                     \
  case KK:                                                                                                                 \
    if (jout) return m64::launch_k<KK, m64::kJamps>(rec, nevt, tab, t64, hslots, nslot, lin, mask, ctri, cst, out, stride, jout, \
                                                    shape, share, nullptr, st);                                            \
    if (j2) return m64::launch_k<KK, m64::kLhe>(rec, nevt, tab, t64, hslots, nslot, lin, mask, ctri, cst, out, stride, nullptr,  \
                                                shape, share, j2, st);                                                     \
    return m64::launch_k<KK, m64::kME>(rec, nevt, tab, t64, hslots, nslot, lin, mask, ctri, cst, out, stride, nullptr, shape,    \
                                       share, nullptr, st);
  switch (K) {
    MG_64_CASE(3)
    MG_64_CASE(4)
    MG_64_CASE(5)
    default: return cudaErrorInvalidValue;
  }
#undef MG_64_CASE
}

}  // namespace mg
