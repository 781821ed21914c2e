// Thread-block clusters: rank, barrier, a value of another block's shared
// memory, and the launch with a cluster of a size chosen at run time.
#pragma once

#include "bem_internal.cuh"

namespace bem {

__device__ __forceinline__ unsigned cluster_rank() {
    unsigned r;
    asm volatile("mov.u32 %0, %%cluster_ctarank;" : "=r"(r));
    return r;
}
__device__ __forceinline__ void cluster_sync() {
    asm volatile("barrier.cluster.arrive;\n\tbarrier.cluster.wait;" ::: "memory");
}
// a double of another block's shared memory, at the address p has here
__device__ __forceinline__ double peer_double(const double *p, unsigned rank) {
    const unsigned a = (unsigned)__cvta_generic_to_shared(p);
    unsigned r;
    double v;
    asm volatile("mapa.shared::cluster.u32 %0, %1, %2;" : "=r"(r) : "r"(a), "r"(rank));
    asm volatile("ld.shared::cluster.f64 %0, [%1];" : "=d"(v) : "r"(r));
    return v;
}

__device__ __forceinline__ double peer_load(const double *p, unsigned rank) { return peer_double(p, rank); }
__device__ __forceinline__ float peer_load(const float *p, unsigned rank) {
    const unsigned a = (unsigned)__cvta_generic_to_shared(p);
    unsigned r;
    float v;
    asm volatile("mapa.shared::cluster.u32 %0, %1, %2;" : "=r"(r) : "r"(a), "r"(rank));
    asm volatile("ld.shared::cluster.f32 %0, [%1];" : "=f"(v) : "r"(r));
    return v;
}

template <class... P, class... A>
int launch_cluster(void (*kernel)(P...), unsigned blocks, int threads, size_t smem, int cluster, cudaStream_t s, A... args) {
    cudaLaunchAttribute at[1];
    at[0].id = cudaLaunchAttributeClusterDimension;
    at[0].val.clusterDim.x = cluster;
    at[0].val.clusterDim.y = at[0].val.clusterDim.z = 1;
    cudaLaunchConfig_t cfg{};
    cfg.gridDim = dim3(blocks);
    cfg.blockDim = dim3(threads);
    cfg.dynamicSmemBytes = smem;
    cfg.stream = s;
    cfg.attrs = at;
    cfg.numAttrs = cluster > 1 ? 1 : 0;
    BEM_CUDA(cudaLaunchKernelEx(&cfg, kernel, static_cast<P>(args)...));
    count_launch();
    return BEM_OK;
}

}  // namespace bem
