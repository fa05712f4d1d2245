// mg_persist.cu -- the FP64 matrix elements of several jobs (any mix of the four processes) in ONE
// persistent kernel launch.
//
// The paper (Sec. 4) finds the GPU throughput still growing up to batches of ~16k events: smaller batches
// leave the device underfilled.  A batch of many small jobs therefore runs better as one launch whose
// thread blocks drain a common queue of work tiles than as one launch per job.  Here the queue holds
// (job, block of helicities, tile of 32 events) triples, the jobs ordered by falling cost per tile (more
// gluons first, so the longest tiles start first); each 128-thread block takes the next tile from an
// atomic counter until the queue is empty, and runs the same per-thread FP64 work as the
// single-job kernels (the per-event record
// from k_event_prep; the items shared between a job's gluon-helicity combinations from its
// launch_pass64 where its context's FP64 shape shares them, else built in the thread; a job whose items exceed
// 2 GiB runs in launches of its own).  The results are
// bit-identical to mg_sigmakin(MG_FP64), with or without the shared currents.
#include <cuda_runtime.h>

#include <algorithm>
#include <cmath>
#include <vector>

#include "mg_alloc.h"
#include "mg_ctx.h"
#include "mg_internal.h"
#include "mg_kernels.h"
#include "mg_me64_k2.cuh"
#include "mg_me64l.cuh"

namespace mg {
namespace pers {

constexpr int kMaxJobs = 64;   // the job table travels as the kernel's parameter (8 KB)

struct PJob {
  const double* rec;        // per-event FP64 record
  const Tables* tab;
  const int* gslots;        // gluon-helicity combinations (one of each flipped pair) with a good helicity
  const int* nslot;
  const int* lin;           // nonzero: linear polarisations (3 to 5 gluons)
  const uint32_t* mask;
  const double* ctri;
  const Tab64* t64;
  const double* share;      // the job's shared items (launch_pass64), or null: every combination on its own
  double* part;             // part[row * stride + e]
  double norm;              // (2 gluons: rec holds the momenta, part the MEs, which are norm * the helicity sum)
  int64_t nevt, stride, tile0;
  int K, ntile_ev;
  MeConst cst;
};

struct PBatch {
  int njobs;
  int64_t ntiles;
  PJob job[kMaxJobs];
};

template <int K, bool OWN>
__device__ __forceinline__ void run64(const PJob& J, int64_t tile, int blk) {
  if (!OWN || J.share)
    m64::thread64<K, false, false>(J.rec, J.nevt, tile, blk, J.tab, J.t64, J.gslots, J.nslot, J.lin, J.mask, J.ctri, J.cst,
                                   J.part, J.stride, J.share);
  else if constexpr (OWN)
    m64::thread64<K, false, true>(J.rec, J.nevt, tile, blk, J.tab, J.t64, J.gslots, J.nslot, J.lin, J.mask, J.ctri, J.cst,
                                  J.part, J.stride, nullptr);
}

// OWN: some job of 3 to 5 gluons runs without shared items.  Its threads keep their items in 50 KB of local memory, which
// the driver reserves for every thread the GPU can hold (14.7 GB of device memory in all, against 2.7), so batches whose jobs all
// share have a kernel without that code.
template <bool OWN>
__global__ void __launch_bounds__(kMeThreads, 3) k_me_persistent(const __grid_constant__ PBatch b,
                                                              unsigned long long* __restrict__ next) {
  __shared__ long long s_tile;
  __shared__ m64::K2Block s_k2;
  for (;;) {
    if (threadIdx.x == 0) s_tile = static_cast<long long>(atomicAdd(next, 1ull));
    __syncthreads();
    const int64_t tile = s_tile;
    __syncthreads();
    if (tile >= b.ntiles) return;
    int lo = 0, hi = b.njobs - 1;   // the job holding the tile: the last one with tile0 <= tile
    while (lo < hi) {
      const int mid = (lo + hi + 1) >> 1;
      if (b.job[mid].tile0 <= tile) lo = mid;
      else hi = mid - 1;
    }
    const PJob& J = b.job[lo];
    const int64_t t = tile - J.tile0;
    const int slot = static_cast<int>(t / J.ntile_ev);
    const int64_t etile = t - static_cast<int64_t>(slot) * J.ntile_ev;
    switch (J.K) {
      case 2: m64::k2_page(s_k2, J.rec, J.nevt, etile, J.mask, J.ctri, J.cst, J.norm, J.part); break;
      case 3: run64<3, OWN>(J, etile, slot); break;
      case 4: run64<4, OWN>(J, etile, slot); break;
      default: run64<5, OWN>(J, etile, slot); break;
    }
  }
}

}  // namespace pers
}  // namespace mg

namespace {

int64_t pad_pg(int64_t n) { return (n + mg::kPage - 1) / mg::kPage * mg::kPage; }

mg_status grow_d(double** buf, int64_t* cap, int64_t need) {
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

}  // namespace

extern "C" mg_status mg_sigmakin_batch(const mg_batch_job* jobs, int njobs, void* stream) {
  if (!jobs || njobs < 1 || njobs > mg::pers::kMaxJobs) return MG_EINVAL;
  for (int i = 0; i < njobs; ++i) {
    const mg_batch_job& j = jobs[i];
    if (!j.ctx || j.nevt < 0 || (j.nevt > 0 && (!j.mom_dev || !j.me_dev))) return MG_EINVAL;
    if (j.ctx->prm.wt != 0.0) return MG_ENOTSUP;
    for (int k = 0; k < i; ++k)
      if (jobs[k].ctx == j.ctx) return MG_EINVAL;   // one context per job: the scratch is per context
  }
  cudaStream_t st = static_cast<cudaStream_t>(stream);
  // per job: helicity mask (first call), scratch, per-event record; the tile table, costliest jobs first
  std::vector<int> order(njobs);
  for (int i = 0; i < njobs; ++i) order[i] = i;
  std::stable_sort(order.begin(), order.end(), [&](int a, int b) { return jobs[a].ctx->K > jobs[b].ctx->K; });
  mg::pers::PBatch* batch = new (std::nothrow) mg::pers::PBatch;
  if (!batch) return MG_ENOMEM;
  batch->njobs = 0;
  batch->ntiles = 0;
  mg_status s = MG_OK;
  bool own = false;
  for (int oi = 0; oi < njobs && s == MG_OK; ++oi) {
    const mg_batch_job& j = jobs[order[oi]];
    mg_ctx* c = j.ctx;
    if (j.nevt == 0) continue;
    if (!c->mask_ready) s = mg_hel_filter(c, j.mom_dev, j.nevt, stream);
    const int64_t stride = pad_pg(j.nevt);
    if (s == MG_OK) s = grow_d(&c->d_part, &c->part_cap, stride * c->nhel);
    if (s == MG_OK) s = grow_d(&c->d_prep, &c->prep_cap, stride * mg::event_record_bytes(c->K, false) / 8 + 1);
    if (s != MG_OK) break;
    c->last = st;
    mg::MeConst cst;
    cst.gs = std::sqrt(4.0 * 3.14159265358979323846 * c->prm.alphas);
    cst.mt = c->prm.mt;
    cst.wt = c->prm.wt;
    cst.conj = 1;   // one of each pair of flipped helicities
    cst.colour_scale = cst.gs * cst.gs / static_cast<double>(c->colour_den);
    if (c->K >= 3 && mg::launch_event_prep(c->K, false, j.mom_dev, j.nevt, cst, c->d_prep, st) != cudaSuccess) { s = MG_ECUDA; break; }
    // the job's items shared between its gluon-helicity combinations, where its
    // context's FP64 shape asks for them
    const double* share = nullptr;
    if (c->shape[MG_FP64].shared && c->K >= 3) {
      const int64_t chunk = mg::item_chunk(c, stride);
      s = grow_d(&c->d_share, &c->share_cap, mg::item_chunk_max(c, stride) * mg::share_doubles(c->K));
      if (s != MG_OK) break;
      if (chunk < stride) {
        // items over 2 GiB: the job's matrix elements in chunks and launches of its own, as mg_sigmakin's.  In the
        // persistent launch without items 7,008 gg -> t tbar g g g events took 43.3 ms, now 15.3, 60,000
        // gg -> t tbar g g events 33.3, now 9.4
        const int64_t nitem = mg::event_record_bytes(c->K, false) / 8;
        for (int64_t e0 = 0; e0 < j.nevt && s == MG_OK; e0 += chunk)
          if (mg::fp64_slots(c, c->d_prep + (e0 / mg::kPage) * nitem * mg::kPage, j.nevt - e0 < chunk ? j.nevt - e0 : chunk,
                             true, cst, c->d_part + e0, stride, c->shape[MG_FP64], st) != cudaSuccess)
            s = MG_ECUDA;
        continue;
      }
      if (mg::launch_pass64(c->K, c->d_prep, j.nevt, c->d_tab, c->d_tab64, cst, c->d_lin, c->d_share, st) != cudaSuccess) { s = MG_ECUDA; break; }
      share = c->d_share;
    }
    own = own || (c->K >= 3 && !share);
    mg::pers::PJob& p = batch->job[batch->njobs++];
    p.share = share;
    p.rec = c->K == 2 ? j.mom_dev : c->d_prep;
    p.norm = 1.0 / (256.0 * mg::factorial(c->ng));
    p.tab = c->d_tab;
    p.t64 = c->d_tab64;
    p.gslots = c->d_hslots;
    p.nslot = c->d_nhslots;
    p.lin = c->d_lin;
    p.mask = c->d_mask;
    p.ctri = c->d_ctri;
    p.part = c->K == 2 ? j.me_dev : c->d_part;
    p.nevt = j.nevt;
    p.stride = stride;
    p.K = c->K;
    p.ntile_ev = static_cast<int>((j.nevt + mg::kPage - 1) / mg::kPage);
    p.tile0 = batch->ntiles;
    p.cst = cst;
    // 3 to 5 gluons: 2^(K-1) blocks of work per event tile (thread64); 2: one
    batch->ntiles += static_cast<int64_t>(p.ntile_ev) << (c->K == 2 ? 0 : c->K - 1);
  }
  if (s == MG_OK && batch->njobs > 0) {
    // the tile counter of the costliest job's context (a context's work is ordered on one stream at a time)
    unsigned long long* counter_dev = jobs[order[0]].ctx->d_tiles;
    int dev = 0, nsm = 0, per_sm = 0;
    cudaGetDevice(&dev);
    cudaDeviceGetAttribute(&nsm, cudaDevAttrMultiProcessorCount, dev);
    const auto kernel = own ? mg::pers::k_me_persistent<true> : mg::pers::k_me_persistent<false>;
    if (cudaOccupancyMaxActiveBlocksPerMultiprocessor(&per_sm, kernel, mg::kMeThreads, 0) != cudaSuccess ||
        per_sm < 1)
      per_sm = 1;
    int64_t blocks = static_cast<int64_t>(nsm) * per_sm;
    if (blocks > batch->ntiles) blocks = batch->ntiles;
    if (cudaMemsetAsync(counter_dev, 0, sizeof(unsigned long long), st) != cudaSuccess) s = MG_ECUDA;
    if (s == MG_OK) {
      kernel<<<static_cast<unsigned>(blocks), mg::kMeThreads, 0, st>>>(*batch, counter_dev);
      mg::note_launch();
      if (cudaGetLastError() != cudaSuccess) s = MG_ECUDA;
    }
  }
  for (int i = 0; i < njobs && s == MG_OK; ++i) {
    const mg_batch_job& j = jobs[i];
    if (j.nevt == 0 || j.ctx->K == 2) continue;
    const double norm = 1.0 / (256.0 * mg::factorial(j.ctx->ng));
    if (mg::fp64_hel_sum(j.ctx, j.nevt, pad_pg(j.nevt), norm, j.me_dev, st) != cudaSuccess)
      s = MG_ECUDA;
  }
  delete batch;
  return s;
}
