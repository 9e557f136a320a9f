// cluster.cuh -- thread-block clusters: ranks, barrier, reads of another CTA's
// shared memory, and the launch with a cluster size.
//
// The kernels that use them split the terms of one right-hand side over the
// CTAs of a cluster when the right-hand sides alone leave most SMs idle; the
// CTAs' partial sums then meet through distributed shared memory, in rank
// order, without an intermediate in global memory.  With a cluster size of 1
// (a plain launch) none of these instructions run.
#pragma once

#include <cuda_runtime.h>

namespace pce {

constexpr int kSms = 152;          // SMs of a GB300
constexpr int kMaxCluster = 8;     // portable cluster size

__device__ __forceinline__ int cluster_rank() {
    unsigned r;
    asm("mov.u32 %0, %%cluster_ctarank;\n" : "=r"(r));
    return (int)r;
}
// Every thread of every CTA of the cluster: writes to shared memory before it
// are visible to the cluster's reads after it.
__device__ __forceinline__ void cluster_sync() {
    asm volatile("barrier.cluster.arrive.release.aligned;\nbarrier.cluster.wait.acquire.aligned;\n" ::: "memory");
}
// The object at p (this CTA's shared memory) in CTA `rank` of the cluster.
__device__ __forceinline__ unsigned cluster_map(const void* p, int rank) {
    unsigned a;
    asm("mapa.shared::cluster.u32 %0, %1, %2;\n" : "=r"(a) : "r"((unsigned)__cvta_generic_to_shared(p)), "r"(rank));
    return a;
}
__device__ __forceinline__ float2 cluster_ld2(unsigned a) {
    float2 v;
    asm volatile("ld.shared::cluster.v2.f32 {%0, %1}, [%2];\n" : "=f"(v.x), "=f"(v.y) : "r"(a) : "memory");
    return v;
}
__device__ __forceinline__ float cluster_ld(unsigned a) {
    float v;
    asm volatile("ld.shared::cluster.f32 %0, [%1];\n" : "=f"(v) : "r"(a) : "memory");
    return v;
}

// Launch with clusters of `cluster` CTAs (1: none).
template <class... P, class... A>
cudaError_t launch_cluster(void (*kernel)(P...), dim3 grid, dim3 cluster, int threads, int smem, cudaStream_t s,
                           A... args) {
    cudaLaunchConfig_t cfg = {};
    cfg.gridDim = grid;
    cfg.blockDim = dim3(threads);
    cfg.dynamicSmemBytes = smem;
    cfg.stream = s;
    cudaLaunchAttribute at[1];
    at[0].id = cudaLaunchAttributeClusterDimension;
    at[0].val.clusterDim.x = cluster.x;
    at[0].val.clusterDim.y = cluster.y;
    at[0].val.clusterDim.z = cluster.z;
    cfg.attrs = at;
    cfg.numAttrs = cluster.x * cluster.y * cluster.z > 1 ? 1 : 0;
    return cudaLaunchKernelEx(&cfg, kernel, static_cast<P>(args)...);
}

}  // namespace pce
