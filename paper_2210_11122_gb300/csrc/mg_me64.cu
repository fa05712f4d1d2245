// mg_me64.cu -- launches of the FP64 matrix elements of 3 to 5 gluons (mg_me64.cuh): the passes that fill the
// shared items, and the slot kernel reading them.
#include <cuda_runtime.h>

#include "mg_internal.h"
#include "mg_kernels.h"
#include "mg_me64.cuh"

namespace mg {
namespace m64 {

// One block per (event tile, combination); slot_major: all combinations of an event tile are dispatched together.
template <int K, int MODE, bool LOCAL, int MINB>
__global__ void __launch_bounds__(kMeThreads, MINB)
k_me64(const double* __restrict__ rec, int64_t nevt, const Tables* __restrict__ tab, const Tab64* __restrict__ t64,
       const int* __restrict__ hslots, const int* __restrict__ nslot, const uint32_t* __restrict__ mask,
       const double* __restrict__ ctri, MeConst cst, double* __restrict__ out, int64_t stride, float2* __restrict__ jout,
       int slot_major, const double* __restrict__ share, double* __restrict__ j2) {
  const unsigned tile = slot_major ? blockIdx.y : blockIdx.x;
  const int slot = static_cast<int>(slot_major ? blockIdx.x : blockIdx.y);
  if (slot >= *nslot) return;
  thread64<K, MODE, LOCAL>(rec, nevt, tile, slot, hslots[slot], tab, t64, mask, ctri, cst, out, stride, jout, share, j2);
}

template <int K>
static cudaError_t launch_pass(const double* rec, int64_t nevt, const Tables* tab, const Tab64* t64, const MeConst& cst,
                               double* share, cudaStream_t st) {
  const Tab64& h = tab64_host(K);
  const int64_t lanes = (nevt + kPage - 1) / kPage * kPage;
  if (lanes <= 0) return cudaSuccess;
  for (int p = 0; p < h.npass; ++p) {
    const int n = h.pass0[p + 1] - h.pass0[p];
    { k_pass64<K><<<static_cast<unsigned>((lanes * n + 127) / 128), 128, 0, st>>>(rec, nevt, tab, t64, cst.gs, h.pass0[p],
                                                                                  n, share); mg::note_launch(); }
    const cudaError_t e = cudaGetLastError();
    if (e != cudaSuccess) return e;
  }
  return cudaSuccess;
}

template <int K, int MODE>
static cudaError_t launch_k(const double* rec, int64_t nevt, const Tables* tab, const Tab64* t64, const int* hslots,
                            const int* nslot, const uint32_t* mask, const double* ctri, const MeConst& cst, double* out,
                            int64_t stride, float2* jout, MeShape shape, const double* share, double* j2,
                            cudaStream_t st) {
  constexpr unsigned MAXSLOT = 1 << (K - 1);
  const int nev = share ? events_per_block<false>() : events_per_block<true>();
  const unsigned tiles = static_cast<unsigned>((nevt + nev - 1) / nev);
  if (tiles == 0) return cudaSuccess;
  // (a grid's y extent is limited to 65,535: event tiles beyond it go to x)
  const int sm = shape.slot_major && tiles <= 65535 ? 1 : 0;
  const dim3 grid = sm ? dim3(MAXSLOT, tiles) : dim3(tiles, MAXSLOT);
  if (share)
    k_me64<K, MODE, false, 4><<<grid, kMeThreads, 0, st>>>(rec, nevt, tab, t64, hslots, nslot, mask, ctri, cst, out, stride,
                                                           jout, sm, share, j2);
  else
    k_me64<K, MODE, true, 2><<<grid, kMeThreads, 0, st>>>(rec, nevt, tab, t64, hslots, nslot, mask, ctri, cst, out, stride,
                                                          jout, sm, nullptr, j2);
  mg::note_launch();
  return cudaGetLastError();
}

}  // namespace m64

cudaError_t launch_pass64(int K, const double* rec, int64_t nevt, const Tables* tab, const Tab64* t64, const MeConst& cst,
                          double* share, cudaStream_t st) {
  switch (K) {
    case 3: return m64::launch_pass<3>(rec, nevt, tab, t64, cst, share, st);
    case 4: return m64::launch_pass<4>(rec, nevt, tab, t64, cst, share, st);
    case 5: return m64::launch_pass<5>(rec, nevt, tab, t64, cst, share, st);
    default: return cudaErrorInvalidValue;
  }
}

cudaError_t launch_me64(int K, const double* rec, int64_t nevt, const Tables* tab, const Tab64* t64, const int* hslots,
                        const int* nslot, const uint32_t* mask, const double* ctri, const MeConst& cst, double* out,
                        int64_t stride, float2* jout, MeShape shape, const double* share, double* j2, cudaStream_t st) {
#define MG_64_CASE(KK)                                                                                                     \
  case KK:                                                                                                                 \
    if (jout) return m64::launch_k<KK, m64::kJamps>(rec, nevt, tab, t64, hslots, nslot, mask, ctri, cst, out, stride, jout, \
                                                    shape, share, nullptr, st);                                            \
    if (j2) return m64::launch_k<KK, m64::kLhe>(rec, nevt, tab, t64, hslots, nslot, mask, ctri, cst, out, stride, nullptr,  \
                                                shape, share, j2, st);                                                     \
    return m64::launch_k<KK, m64::kME>(rec, nevt, tab, t64, hslots, nslot, mask, ctri, cst, out, stride, nullptr, shape,    \
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
