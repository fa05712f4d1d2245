// mg_me64.cu -- launches of the FP64 matrix elements of 3 to 5 gluons (mg_me64.cuh): the passes that fill the
// shared items, and the slot kernel reading them.
#include <cuda_runtime.h>

#include "mg_internal.h"
#include "mg_kernels.h"
#include "mg_me64.cuh"

namespace mg {
namespace m64 {

// MINB resident blocks per SM: 4 for 3 gluons (at most 128 registers), 3 for 4 and 5 (at most 168).
template <int K, int MODE, bool LOCAL, int MINB>
__global__ void __launch_bounds__(kMeThreads, MINB)
k_me64(const double* __restrict__ rec, int64_t nevt, const Tables* __restrict__ tab, const Tab64* __restrict__ t64,
       const int* __restrict__ hslots, const int* __restrict__ nslot, const uint32_t* __restrict__ mask,
       const double* __restrict__ ctri, MeConst cst, double* __restrict__ out, int64_t stride, float2* __restrict__ jout,
       int tile_ev, int slot_major, const double* __restrict__ share, double* __restrict__ j2) {
  const int tile_sl = static_cast<int>(blockDim.x) / tile_ev;   // slots per block
  const unsigned bev = slot_major ? blockIdx.y : blockIdx.x, bsl = slot_major ? blockIdx.x : blockIdx.y;
  const int64_t e = static_cast<int64_t>(bev) * tile_ev + threadIdx.x % tile_ev;
  const int slot = static_cast<int>(bsl) * tile_sl + static_cast<int>(threadIdx.x) / tile_ev;
  if (e >= nevt || slot >= *nslot) return;
  thread64<K, MODE, LOCAL>(rec, e, slot, hslots[slot], tab, t64, mask, ctri, cst, out, stride, jout, share, j2);
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

static int sm_count() {
  int dev = 0, n = 0;
  if (cudaGetDevice(&dev) != cudaSuccess || cudaDeviceGetAttribute(&n, cudaDevAttrMultiProcessorCount, dev) != cudaSuccess) {
    cudaGetLastError();
    return 1;
  }
  return n;
}

template <int K, int MODE>
static cudaError_t launch_k(const double* rec, int64_t nevt, const Tables* tab, const Tab64* t64, const int* hslots,
                            const int* nslot, const uint32_t* mask, const double* ctri, const MeConst& cst, double* out,
                            int64_t stride, float2* jout, MeShape shape, const double* share, double* j2,
                            cudaStream_t st) {
  constexpr int MAXSLOT = 1 << (K - 1);
  int tev = shape.tile_ev;
  if (tev != 32 && tev != 64 && tev != 128) tev = 128;
  int threads = kMeThreads;
  // a grid of fewer than 4 blocks per SM: blocks of 2 warps, so that the busiest sub-partition holds at most half
  // a warp more than the average instead of a whole one
  if ((nevt + tev - 1) / tev * ((MAXSLOT + kMeThreads / tev - 1) / (kMeThreads / tev)) < 4 * static_cast<int64_t>(sm_count())) {
    threads = kMeThreads / 2;
    if (tev > threads) tev = threads;
  }
  const int tsl = threads / tev;
  const unsigned nev_t = static_cast<unsigned>((nevt + tev - 1) / tev), nsl_t = (MAXSLOT + tsl - 1) / tsl;
  const int sm = shape.slot_major ? 1 : 0;
  const dim3 grid = sm ? dim3(nsl_t, nev_t) : dim3(nev_t, nsl_t);
  if (nev_t == 0) return cudaSuccess;
  if (share)
    k_me64<K, MODE, false, (K == 3 ? 4 : 3)><<<grid, threads, 0, st>>>(rec, nevt, tab, t64, hslots, nslot, mask, ctri, cst, out,
                                                                       stride, jout, tev, sm, share, j2);
  else
    k_me64<K, MODE, true, 2><<<grid, threads, 0, st>>>(rec, nevt, tab, t64, hslots, nslot, mask, ctri, cst, out, stride,
                                                       jout, tev, sm, nullptr, j2);
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
