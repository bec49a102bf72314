// cluster_dev.cuh -- one cluster of 16 CTAs that owns bands of rows: barriers,
// stores into a peer's shared memory, the rows of a band.
#pragma once

#include "ehd_dev.cuh"

namespace ehd {

constexpr int kClusterCtas = 16;

__device__ __forceinline__ void cluster_arrive() {
  asm volatile("barrier.cluster.arrive.release.aligned;\n" ::: "memory");
}
__device__ __forceinline__ void cluster_wait() { asm volatile("barrier.cluster.wait.acquire.aligned;\n" ::: "memory"); }
__device__ __forceinline__ void cluster_sync() {
  __syncwarp();
  cluster_arrive();
  cluster_wait();
}
__device__ __forceinline__ unsigned smem_addr(const void* p) { return (unsigned)__cvta_generic_to_shared(p); }
// the address of p's counterpart in CTA `rank` of the cluster
__device__ __forceinline__ unsigned peer_addr(const void* p, int rank) {
  unsigned r;
  asm("mapa.shared::cluster.u32 %0, %1, %2;\n" : "=r"(r) : "r"(smem_addr(p)), "r"(rank));
  return r;
}
__device__ __forceinline__ void st_peer(unsigned a, float v) {
  asm volatile("st.shared::cluster.f32 [%0], %1;\n" ::"r"(a), "f"(v) : "memory");
}
__device__ __forceinline__ void st_peer(unsigned a, float2 v) {
  asm volatile("st.shared::cluster.v2.f32 [%0], {%1, %2};\n" ::"r"(a), "f"(v.x), "f"(v.y) : "memory");
}

// first row of CTA c's band, and the CTA that owns row j
__host__ __device__ __forceinline__ int band_start(int c, int Ny) { return c * Ny / kClusterCtas; }
__device__ __forceinline__ int band_owner(int j, int Ny) { return ((j + 1) * kClusterCtas - 1) / Ny; }

// launch configuration of one such cluster
inline void cluster_launch_config(cudaLaunchConfig_t* c, cudaLaunchAttribute* at, int threads, size_t smem,
                                  cudaStream_t s) {
  at[0].id = cudaLaunchAttributeClusterDimension;
  at[0].val.clusterDim.x = kClusterCtas;
  at[0].val.clusterDim.y = 1;
  at[0].val.clusterDim.z = 1;
  *c = cudaLaunchConfig_t{};
  c->gridDim = dim3(kClusterCtas);
  c->blockDim = dim3(threads);
  c->dynamicSmemBytes = smem;
  c->stream = s;
  c->attrs = at;
  c->numAttrs = 1;
}
// Whether the current device holds a cluster of this kernel with `smem` bytes
// per CTA; sets the kernel's attributes for it.
template <class K>
bool cluster_fits(K kernel, int threads, size_t smem) {
  int dev = 0, optin = 0, n = 0;
  cudaFuncAttributes fa;
  cudaLaunchAttribute at[1];
  cudaLaunchConfig_t c;
  cluster_launch_config(&c, at, threads, smem, nullptr);
  const bool ok = cudaGetDevice(&dev) == cudaSuccess &&
                  cudaDeviceGetAttribute(&optin, cudaDevAttrMaxSharedMemoryPerBlockOptin, dev) == cudaSuccess &&
                  cudaFuncGetAttributes(&fa, kernel) == cudaSuccess && smem + fa.sharedSizeBytes <= (size_t)optin &&
                  cudaFuncSetAttribute(kernel, cudaFuncAttributeMaxDynamicSharedMemorySize,
                                       optin - (int)fa.sharedSizeBytes) == cudaSuccess &&
                  cudaFuncSetAttribute(kernel, cudaFuncAttributeNonPortableClusterSizeAllowed, 1) == cudaSuccess &&
                  cudaOccupancyMaxActiveClusters(&n, kernel, &c) == cudaSuccess && n >= 1;
  if (!ok) (void)cudaGetLastError();
  return ok;
}

}  // namespace ehd
