// Thread-block clusters: rank, size, barrier and launch configuration of the kernels that give one system or path to
// several blocks.
#pragma once

#include <cuda_runtime.h>

namespace wpccc {

static __device__ __forceinline__ int cluster_rank() {
    int r;
    asm volatile("mov.u32 %0, %%cluster_ctarank;\n" : "=r"(r));
    return r;
}
static __device__ __forceinline__ int cluster_size() {
    int r;
    asm volatile("mov.u32 %0, %%cluster_nctarank;\n" : "=r"(r));
    return r;
}
// Barrier over all threads of the cluster; global- and shared-memory writes made before it are visible after it
// (release / acquire at cluster scope), by plain loads too.  __ldcg marks reads of what other blocks wrote where the line
// would not be read again from L1.
static __device__ __forceinline__ void cluster_sync_all() {
    asm volatile("barrier.cluster.arrive.release.aligned;\nbarrier.cluster.wait.acquire.aligned;\n" ::: "memory");
}

// Launch of `systems` clusters of `size` blocks (size 1 to 8).
struct ClusterLaunch {
    cudaLaunchConfig_t cfg = {};
    cudaLaunchAttribute attr[1];
    ClusterLaunch(int systems, int size, int threads, size_t smem, cudaStream_t st) {
        cfg.gridDim = dim3((unsigned)(systems * size));
        cfg.blockDim = dim3((unsigned)threads);
        cfg.dynamicSmemBytes = smem;
        cfg.stream = st;
        attr[0].id = cudaLaunchAttributeClusterDimension;
        attr[0].val.clusterDim.x = (unsigned)size;
        attr[0].val.clusterDim.y = attr[0].val.clusterDim.z = 1;
        cfg.attrs = attr;
        cfg.numAttrs = 1;
    }
};

}  // namespace wpccc
