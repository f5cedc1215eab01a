// Thread-block clusters: barrier, distributed shared memory reads, launch.
#pragma once
#include "ssv_internal.cuh"

namespace ssv {

static __device__ __forceinline__ void cluster_sync_all() {
  asm volatile("barrier.cluster.arrive.release.aligned;\n\tbarrier.cluster.wait.acquire.aligned;" ::: "memory");
}
static __device__ __forceinline__ int cluster_rank() {
  uint32_t r;
  asm volatile("mov.u32 %0, %%cluster_ctarank;" : "=r"(r));
  return (int)r;
}
static __device__ __forceinline__ uint32_t cluster_map(const void* p, int rank) {
  const uint32_t a = (uint32_t)__cvta_generic_to_shared(p);
  uint32_t r;
  asm volatile("mapa.shared::cluster.u32 %0, %1, %2;" : "=r"(r) : "r"(a), "r"(rank));
  return r;
}
// shared memory of CTA `rank` of the cluster at the address of the caller's own p
static __device__ __forceinline__ double cluster_ld(const double* p, int rank) {
  double v;
  asm volatile("ld.shared::cluster.f64 %0, [%1];" : "=d"(v) : "r"(cluster_map(p, rank)) : "memory");
  return v;
}
static __device__ __forceinline__ int cluster_ld(const int* p, int rank) {
  int v;
  asm volatile("ld.shared::cluster.s32 %0, [%1];" : "=r"(v) : "r"(cluster_map(p, rank)) : "memory");
  return v;
}

static __device__ __forceinline__ void cluster_st(double* p, int rank, double v) {
  asm volatile("st.shared::cluster.f64 [%0], %1;" ::"r"(cluster_map(p, rank)), "d"(v) : "memory");
}

// The most dynamic shared memory a kernel is ever launched with.  The limit belongs
// to the kernel on the device, not to a launch, and is shared by all host threads:
// set to the size of one launch, it can fall below the size of another thread's
// launch before that one is made.  So always the same value for a kernel.
template <typename... KArgs>
cudaError_t allow_smem(void (*kern)(KArgs...), size_t most) {
  return cudaFuncSetAttribute(kern, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)most);
}

// launch `grid` blocks in clusters of R (grid a multiple of R; R > 8 needs
// cudaFuncAttributeNonPortableClusterSizeAllowed set on the kernel, smem beyond
// 48 KB allow_smem)
template <typename... KArgs, typename... Args>
cudaError_t launch_cluster(void (*kern)(KArgs...), int grid, int threads, int R, size_t smem, cudaStream_t st,
                           Args... args) {
  cudaLaunchConfig_t cfg = {};
  cfg.gridDim = dim3((unsigned)grid);
  cfg.blockDim = dim3((unsigned)threads);
  cfg.dynamicSmemBytes = smem;
  cfg.stream = st;
  cudaLaunchAttribute at[1];
  at[0].id = cudaLaunchAttributeClusterDimension;
  at[0].val.clusterDim.x = (unsigned)R;
  at[0].val.clusterDim.y = 1;
  at[0].val.clusterDim.z = 1;
  cfg.attrs = at;
  cfg.numAttrs = 1;
  const cudaError_t e = cudaLaunchKernelEx(&cfg, kern, args...);
  if (e == cudaSuccess) count_launch();
  return e;
}
// CTAs per item (a power of two up to 8) when `items` items alone leave SMs idle
static inline int cluster_for(long long items) {
  int R = 1;
  while (R < 8 && items * R < num_sms()) R *= 2;
  return R;
}

}  // namespace ssv
