// Thread-block cluster primitives of the 256 x 256 kernels, whose surfaces and
// images lie in the distributed shared memory of a few CTAs.
#pragma once
#include <atomic>

#include "common.cuh"

__device__ __forceinline__ uint32_t cluster_rank() {
    uint32_t r;
    asm volatile("mov.u32 %0, %%cluster_ctarank;" : "=r"(r));
    return r;
}
// releases every access before it.  The form for a thread that has read another
// CTA's shared memory, whose owner overwrites it after the wait: only a release
// orders those loads before the owner's stores
__device__ __forceinline__ void cluster_arrive() { asm volatile("barrier.cluster.arrive.release.aligned;" ::: "memory"); }
// releases accesses to this CTA's own shared memory only, for values that the others
// read after the wait: does not wait for global stores in flight, and orders no read of
// another CTA's shared memory
__device__ __forceinline__ void cluster_arrive_shared() {
    asm volatile("fence.release.sync_restrict::shared::cta.cluster;\nbarrier.cluster.arrive.relaxed.aligned;" ::: "memory");
}
__device__ __forceinline__ void cluster_wait() { asm volatile("barrier.cluster.wait.acquire.aligned;" ::: "memory"); }
__device__ __forceinline__ uint32_t map_to_rank(const void *p, uint32_t rank) {
    const uint32_t local = (uint32_t)__cvta_generic_to_shared(p);
    uint32_t r;
    asm volatile("mapa.shared::cluster.u32 %0, %1, %2;" : "=r"(r) : "r"(local), "r"(rank));
    return r;
}
__device__ __forceinline__ float2 ld_cluster(uint32_t addr) {
    float2 v;
    asm volatile("ld.shared::cluster.v2.f32 {%0, %1}, [%2];" : "=f"(v.x), "=f"(v.y) : "r"(addr) : "memory");
    return v;
}
__device__ __forceinline__ float ld_cluster_f(uint32_t addr) {
    float v;
    asm volatile("ld.shared::cluster.f32 %0, [%1];" : "=f"(v) : "r"(addr) : "memory");
    return v;
}

// launch of `clusters` clusters of nc CTAs of nt threads
template <class... Params, class... Args>
cudaError_t launch_clusters(void (*kern)(Params...), int nc, int nt, size_t smem, long clusters, cudaStream_t st,
                            Args... args) {
    cudaError_t e = cudaFuncSetAttribute(kern, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem);
    if (e != cudaSuccess) return e;
    cudaLaunchAttribute attr[1];
    attr[0].id = cudaLaunchAttributeClusterDimension;
    attr[0].val.clusterDim.x = nc;
    attr[0].val.clusterDim.y = 1;
    attr[0].val.clusterDim.z = 1;
    cudaLaunchConfig_t cfg = {};
    cfg.gridDim = dim3((unsigned)(nc * clusters));
    cfg.blockDim = dim3(nt);
    cfg.dynamicSmemBytes = smem;
    cfg.stream = st;
    cfg.attrs = attr;
    cfg.numAttrs = 1;
    return cudaLaunchKernelEx(&cfg, kern, static_cast<Params>(args)...);
}
// how many such clusters are resident together; `resident` keeps it between calls
template <class K>
cudaError_t resident_clusters(K *kern, int nc, int nt, size_t smem, std::atomic<int> &resident, int *most) {
    *most = resident.load(std::memory_order_relaxed);
    if (*most > 0) return cudaSuccess;
    cudaError_t e = cudaFuncSetAttribute(kern, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem);
    if (e != cudaSuccess) return e;
    cudaLaunchAttribute attr[1];
    attr[0].id = cudaLaunchAttributeClusterDimension;
    attr[0].val.clusterDim.x = nc;
    attr[0].val.clusterDim.y = 1;
    attr[0].val.clusterDim.z = 1;
    cudaLaunchConfig_t cfg = {};
    cfg.gridDim = dim3((unsigned)(nc * 64));
    cfg.blockDim = dim3(nt);
    cfg.dynamicSmemBytes = smem;
    cfg.attrs = attr;
    cfg.numAttrs = 1;
    e = cudaOccupancyMaxActiveClusters(most, kern, &cfg);
    if (e != cudaSuccess) return e;
    if (*most <= 0) return cudaErrorInvalidConfiguration;
    resident.store(*most, std::memory_order_relaxed);
    return cudaSuccess;
}
