// The many-systems launch: kernel, configuration and launch of one arithmetic
// (solve_batch.cu: FP64 and the plans; solve_batch_df.cu: double-float).
#pragma once
#include "sweep.cuh"

namespace ssv {

struct BatchPlan {
  int dev = 0;
  bool stream_ordered = false;  // buffers from the library pool, ordered on `stream`
  cudaStream_t stream = nullptr;
  int maxm = 1;
  bool dfloat = false;  // SSV_DFLOAT: double-float bulk updates
  int nitems = 0;
  int grid = 0;
  size_t slot = 0;
  size_t smem = 0;
  FpSys* systems = nullptr;
  unsigned long long* items = nullptr;
  cd* scratch = nullptr;
};

// double-float instances (solve_batch_df.cu)
int batch_config_df(BatchPlan* bp);
void batch_launch_df(const BatchPlan* bp, cudaStream_t st);

namespace {

// Many systems in one launch: work item w = (system, shift) from `items`
// (system in the high 32 bits), ordered by decreasing cost.  A system runs in
// the class of its own m (the summation order of ssv_solve), so one wide
// system does not widen the others.
template <int MAXM, bool DF = false>
__global__ void __launch_bounds__(sweep_threads<MAXM>(), sweep_per_sm(MAXM, DF)) solve_fp64_batch_kernel(
    const FpSys* __restrict__ systems, const unsigned long long* __restrict__ items, int nitems,
    cd* __restrict__ scratch, size_t slot_stride) {
  extern __shared__ __align__(16) unsigned char smem_raw[];
  __shared__ int s_piv;
  __shared__ int s_sing;
  constexpr int NT = sweep_threads<MAXM>();
  cd* Z2 = scratch + (size_t)blockIdx.x * slot_stride;
  for (int w = blockIdx.x; w < nitems; w += gridDim.x) {
    const unsigned long long it = items[w];
    const FpSys d = systems[(int)(it >> 32)];
    const int sh = (int)(it & 0xffffffffu);
    if (d.m <= 2) {
      fp64_shift<2, NT, false, false, DF>(d, sh, Z2, smem_raw, &s_piv, &s_sing);
      continue;
    }
    if (d.m <= 4) {
      fp64_shift<4, NT, false, false, DF>(d, sh, Z2, smem_raw, &s_piv, &s_sing);
      continue;
    }
    if (d.m <= 8) {
      fp64_shift<8, NT, false, false, DF>(d, sh, Z2, smem_raw, &s_piv, &s_sing);
      continue;
    }
    if constexpr (MAXM >= 16) {
      if (d.m <= 16) {
        fp64_shift<16, NT, false, false, DF>(d, sh, Z2, smem_raw, &s_piv, &s_sing);
        continue;
      }
    }
    if constexpr (MAXM >= 32) fp64_shift<32, NT, false, false, DF>(d, sh, Z2, smem_raw, &s_piv, &s_sing);
  }
}

template <int MAXM, bool DF>
int batch_config(BatchPlan* bp) {
  using L = Layout<MAXM>;
  auto kern = solve_fp64_batch_kernel<MAXM, DF>;
  SSV_CUDA_TRY(cudaFuncSetAttribute(kern, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)L::bytes));
  int per_sm = 0;
  SSV_CUDA_TRY(cudaOccupancyMaxActiveBlocksPerMultiprocessor(&per_sm, kern, sweep_threads<MAXM>(), L::bytes));
  per_sm = std::max(1, std::min(per_sm, sweep_per_sm(MAXM, DF)));
  bp->grid = std::max(1, std::min(bp->nitems, num_sms() * per_sm));
  bp->smem = L::bytes;
  return SSV_OK;
}

template <int MAXM, bool DF>
void batch_launch(const BatchPlan* bp, cudaStream_t st) {
  solve_fp64_batch_kernel<MAXM, DF><<<bp->grid, sweep_threads<MAXM>(), bp->smem, st>>>(bp->systems, bp->items,
                                                                                      bp->nitems, bp->scratch, bp->slot);
  count_launch();
}

// by the widest system of the plan
template <bool DF>
int batch_config_any(BatchPlan* bp) {
  return bp->maxm <= 8 ? batch_config<8, DF>(bp) : bp->maxm <= 16 ? batch_config<16, DF>(bp) : batch_config<32, DF>(bp);
}
template <bool DF>
void batch_launch_any(const BatchPlan* bp, cudaStream_t st) {
  if (bp->maxm <= 8) batch_launch<8, DF>(bp, st);
  else if (bp->maxm <= 16) batch_launch<16, DF>(bp, st);
  else batch_launch<32, DF>(bp, st);
}

}  // namespace

}  // namespace ssv
