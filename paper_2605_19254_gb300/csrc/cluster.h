// Thread-block clusters: a launch of one cluster, its barrier, and stores into
// the shared memory of its blocks (the panel kernels of the eliminations, whose
// columns are a serial chain: a cluster barrier costs a fraction of a launch).
#pragma once

#include <cuda_runtime.h>
#include <stdint.h>

#include <utility>

namespace smf {

#ifdef __CUDACC__
// Every thread of every block of the cluster; remote stores before it are
// visible after it.
__device__ __forceinline__ void cluster_sync() {
    asm volatile("barrier.cluster.arrive.release.aligned;\n\tbarrier.cluster.wait.acquire.aligned;" ::: "memory");
}
// *p = v in the shared memory of block `rank` of the cluster (p: this block's address of the variable)
__device__ __forceinline__ void cluster_store(uint32_t* p, int rank, uint32_t v) {
    const uint32_t a = (uint32_t)__cvta_generic_to_shared(p);
    asm volatile("{\n .reg .u32 r;\n mapa.shared::cluster.u32 r, %0, %1;\n st.shared::cluster.u32 [r], %2;\n}\n" ::"r"(a),
                 "r"(rank), "r"(v)
                 : "memory");
}
#endif

// One cluster of C blocks (up to 16), as a programmatic dependent of the kernel
// before it.  smem_limit: the most dynamic shared memory any launch of the kernel
// takes (the attribute is the kernel's, not the launch's, and other threads may
// launch it at the same time with other sizes).
template <typename... KArgs, typename... Args>
cudaError_t launch_cluster(void (*kernel)(KArgs...), int C, int threads, size_t smem, size_t smem_limit, cudaStream_t s,
                           Args&&... args) {
    if (smem > smem_limit) return cudaErrorInvalidValue;
    cudaError_t e = cudaFuncSetAttribute(kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem_limit);
    if (e == cudaSuccess && C > 8) e = cudaFuncSetAttribute(kernel, cudaFuncAttributeNonPortableClusterSizeAllowed, 1);
    if (e != cudaSuccess) return e;
    cudaLaunchConfig_t cfg{};
    cfg.gridDim = dim3((unsigned)C);
    cfg.blockDim = dim3((unsigned)threads);
    cfg.dynamicSmemBytes = smem;
    cfg.stream = s;
    cudaLaunchAttribute attr[2];
    attr[0].id = cudaLaunchAttributeClusterDimension;
    attr[0].val.clusterDim.x = (unsigned)C;
    attr[0].val.clusterDim.y = 1;
    attr[0].val.clusterDim.z = 1;
    attr[1].id = cudaLaunchAttributeProgrammaticStreamSerialization;
    attr[1].val.programmaticStreamSerializationAllowed = 1;
    cfg.attrs = attr;
    cfg.numAttrs = 2;
    return cudaLaunchKernelEx(&cfg, kernel, std::forward<Args>(args)...);
}

}  // namespace smf
