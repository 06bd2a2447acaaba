// Launch of one instantiation of the cluster-resident solver: n clusters of C blocks.
#pragma once

#include "launch.h"
#include "resident.cuh"

namespace dl {

struct ResConfig {
    cudaLaunchConfig_t cfg;
    cudaLaunchAttribute attr[1];
    ResConfig(int C, int n, size_t smem, cudaStream_t s) {
        cfg = {};
        cfg.gridDim = dim3((unsigned)(C * n));
        cfg.blockDim = dim3(RES_THREADS);
        cfg.dynamicSmemBytes = smem;
        cfg.stream = s;
        attr[0].id = cudaLaunchAttributeClusterDimension;
        attr[0].val.clusterDim.x = (unsigned)C;
        attr[0].val.clusterDim.y = attr[0].val.clusterDim.z = 1;
        cfg.attrs = attr;
        cfg.numAttrs = 1;
    }
};

// Clusters of more than 8 blocks and more than 48 KiB of shared memory are opt-ins of the kernel.
template <typename K>
inline cudaError_t resident_opt_in(K kernel, size_t smem) {
    const cudaError_t e = cudaFuncSetAttribute(kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem);
    if (e != cudaSuccess) return e;
    return cudaFuncSetAttribute(kernel, cudaFuncAttributeNonPortableClusterSizeAllowed, 1);
}

// Clusters of C blocks that can be resident at once (0: size not available).
template <typename K>
inline int resident_max_clusters(K kernel, size_t smem, int C) {
    ResConfig c(C, 1, smem, 0);
    int n = 0;
    if (resident_opt_in(kernel, smem) != cudaSuccess || cudaOccupancyMaxActiveClusters(&n, kernel, &c.cfg) != cudaSuccess) {
        cudaGetLastError();  // (an answer, not a failure: the solve goes step by step)
        return 0;
    }
    return n;
}

template <typename S>
inline cudaError_t resident_go(const ResArgs &a, int C, int n, int cg, cudaStream_t s) {
    auto kernel = cg ? resident_kernel<S, 1> : resident_kernel<S, 0>;
    constexpr size_t smem = sizeof(ResShared<typename Real<S>::type>);
    cudaError_t e = resident_opt_in(kernel, smem);
    if (e != cudaSuccess) return e;
    ResConfig c(C, n, smem, s);
    return cudaLaunchKernelEx(&c.cfg, kernel, a);
}

}  // namespace dl
