// ---------------------------------------------------------------------------
// Batched solve of many systems (uneven n, m, shift counts) in one persistent
// launch.  A plan fixes the device-side system descriptors, the cost-ordered
// (system, shift) worklist and the scratch, so that running it is one kernel
// launch with fixed arguments (capturable in a CUDA graph and replayable after
// the caller rewrites the shift buffers in place).
// ---------------------------------------------------------------------------
#include "batch.cuh"

namespace ssv {

int batch_create(int nsys, const Handle* const* hs, const int* s, const double* const* shifts,
                 const ssv_opts* o, double* const* outs, const long long* ldos, int* const* status,
                 BatchPlan** out, cudaStream_t stream_ordered) {
  *out = nullptr;
  if ((o->precision != SSV_FP64 && o->precision != SSV_DFLOAT) || o->mode == SSV_X) return SSV_ENOTSUP;
  BatchPlan* bp = new (std::nothrow) BatchPlan();
  if (!bp) return SSV_ENOMEM;
  bp->dfloat = o->precision == SSV_DFLOAT;
  cudaGetDevice(&bp->dev);
  bp->stream_ordered = stream_ordered != nullptr;
  bp->stream = stream_ordered;
  std::vector<FpSys> sys(nsys);
  std::vector<std::pair<double, unsigned long long>> work;
  const bool track_t = (o->mode == SSV_XHAT);
  for (int k = 0; k < nsys; ++k) {
    const Handle* h = hs[k];
    FpSys& d = sys[k];
    d.n = h->n; d.m = h->m; d.p = h->p;
    d.nb = o->nb > 0 ? o->nb : tuned_nb(h->n, h->m, h->p, o->precision, o->mode);
    if (d.nb > kNB || h->m > 32) { delete bp; return SSV_ENOTSUP; }
    d.mode = o->mode; d.H = h->H; d.Ct = h->Ct; d.ldct = h->p > 0 ? h->p : 1; d.R = h->R;
    d.shifts = reinterpret_cast<const cd*>(shifts[k]);
    d.out = reinterpret_cast<cd*>(outs[k]); d.ldo = ldos[k];
    d.status = status ? status[k] : nullptr;
    d.xhat_copy = nullptr; d.ldxc = 0; d.hnorm = h->hnorm2; d.bhat = nullptr; d.ldb = 0;
    d.rhs = nullptr; d.ldr = 0; d.flip_out = 0;
    d.Hhi = h->Hhi; d.Hlo = h->Hlo;
    d.gfull = GivensSched{nullptr, nullptr, 0};
    d.gtail = d.gfull;
    bp->maxm = std::max(bp->maxm, h->m);
    bp->slot = std::max(bp->slot, (size_t)(h->p + h->n) * h->m + (track_t ? (size_t)h->n * h->m : 0));
    const double cost = (double)h->n * h->n * h->m * (1.0 + 2.0 * h->m / d.nb);
    for (int j = 0; j < s[k]; ++j) work.push_back({cost, ((unsigned long long)k << 32) | (unsigned)j});
  }
  std::stable_sort(work.begin(), work.end(),
                   [](const std::pair<double, unsigned long long>& a,
                      const std::pair<double, unsigned long long>& b) { return a.first > b.first; });
  bp->nitems = (int)work.size();
  std::vector<unsigned long long> items(work.size());
  for (size_t i = 0; i < work.size(); ++i) items[i] = work[i].second;
  int rc = SSV_OK;
  if (bp->nitems > 0) rc = bp->dfloat ? batch_config_df(bp) : batch_config_any<false>(bp);
  cudaError_t e = cudaSuccess;
  if (rc == SSV_OK && bp->nitems > 0) {
    if (bp->stream_ordered) {
      // stream-ordered: no device-wide synchronisation, so concurrent batches on
      // other streams keep running; pageable sources are consumed before return
      cudaStream_t st = bp->stream;
      e = pool_alloc((void**)&bp->systems, sizeof(FpSys) * nsys, st);
      if (e == cudaSuccess)
        e = pool_alloc((void**)&bp->items, sizeof(unsigned long long) * items.size(), st);
      if (e == cudaSuccess)
        e = pool_alloc((void**)&bp->scratch, sizeof(cd) * bp->slot * bp->grid, st);
      if (e == cudaSuccess)
        e = cudaMemcpyAsync(bp->systems, sys.data(), sizeof(FpSys) * nsys, cudaMemcpyHostToDevice, st);
      if (e == cudaSuccess)
        e = cudaMemcpyAsync(bp->items, items.data(), sizeof(unsigned long long) * items.size(),
                            cudaMemcpyHostToDevice, st);
    } else {
      e = cudaMalloc((void**)&bp->systems, sizeof(FpSys) * nsys);
      if (e == cudaSuccess) e = cudaMalloc((void**)&bp->items, sizeof(unsigned long long) * items.size());
      if (e == cudaSuccess) e = cudaMalloc((void**)&bp->scratch, sizeof(cd) * bp->slot * bp->grid);
      if (e == cudaSuccess)
        e = cudaMemcpy(bp->systems, sys.data(), sizeof(FpSys) * nsys, cudaMemcpyHostToDevice);
      if (e == cudaSuccess)
        e = cudaMemcpy(bp->items, items.data(), sizeof(unsigned long long) * items.size(),
                       cudaMemcpyHostToDevice);
    }
    if (e != cudaSuccess) {
      set_cuda_error(e);
      rc = e == cudaErrorMemoryAllocation ? SSV_ENOMEM : SSV_ECUDA;
    }
  }
  if (rc != SSV_OK) {
    batch_destroy(bp);
    return rc;
  }
  *out = bp;
  return SSV_OK;
}

int batch_run(const BatchPlan* bp, cudaStream_t st) {
  if (bp->nitems == 0) return SSV_OK;
  if (bp->dfloat) batch_launch_df(bp, st);
  else batch_launch_any<false>(bp, st);
  SSV_CUDA_TRY(cudaGetLastError());
  return SSV_OK;
}

void batch_destroy(BatchPlan* bp) {
  if (!bp) return;
  if (bp->stream_ordered) {
    if (bp->systems) cudaFreeAsync(bp->systems, bp->stream);
    if (bp->items) cudaFreeAsync(bp->items, bp->stream);
    if (bp->scratch) cudaFreeAsync(bp->scratch, bp->stream);
  } else {
    cudaFree(bp->systems);
    cudaFree(bp->items);
    cudaFree(bp->scratch);
  }
  delete bp;
}

}  // namespace ssv
