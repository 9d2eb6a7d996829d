// Which thread-block cluster a launch takes.  A cluster's CTAs start together
// on SMs of one GPC, so a GPU with fewer SMs to give (a partition) may not hold
// one; the kernels give the same bits at any size and run alone as well.
#pragma once

namespace img {

// The largest of want, want / 2, ... CTAs (want a power of two) of which the
// GPU can hold a cluster: active(ctas) is how many such clusters fit at once,
// 0 or negative when none does or the query fails.  1: no cluster.
template <class Active>
int cluster_that_fits(int want, Active active) {
    for (int c = want; c > 1; c /= 2)
        if (active(c) > 0) return c;
    return 1;
}

}  // namespace img

#ifdef __CUDACC__
#include <cuda_runtime.h>

namespace img {

// Clusters of `ctas` CTAs of kernel func that the device holds at once; func's
// shared-memory limit is set.
inline int active_clusters(const void *func, int ctas, int threads, size_t smem) {
    cudaLaunchAttribute attr{};
    attr.id = cudaLaunchAttributeClusterDimension;
    attr.val.clusterDim = {(unsigned)ctas, 1, 1};
    cudaLaunchConfig_t cfg{};
    cfg.gridDim = dim3(ctas);
    cfg.blockDim = dim3(threads);
    cfg.dynamicSmemBytes = smem;
    cfg.attrs = &attr;
    cfg.numAttrs = 1;
    int n = 0;
    if (cudaOccupancyMaxActiveClusters(&n, func, &cfg) != cudaSuccess) {
        cudaGetLastError();
        return -1;
    }
    return n;
}

}  // namespace img
#endif
