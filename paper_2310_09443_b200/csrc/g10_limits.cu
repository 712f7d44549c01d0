// What the current device lets a kernel have.
#include <cstdlib>

#include "g10_internal.h"

namespace g10 {

// Can the current device place a cluster of so many blocks of `kernel` with so much dynamic shared memory each?
static bool places_cluster(const void *kernel, int blocks, int threads, size_t smem)
{
    cudaLaunchConfig_t cfg = {};
    cudaLaunchAttribute at[1];
    at[0].id = cudaLaunchAttributeClusterDimension;
    at[0].val.clusterDim.x = (unsigned)blocks; at[0].val.clusterDim.y = 1; at[0].val.clusterDim.z = 1;
    cfg.gridDim = dim3((unsigned)blocks); cfg.blockDim = dim3((unsigned)threads); cfg.dynamicSmemBytes = smem; cfg.attrs = at; cfg.numAttrs = 1;
    int n = 0;
    if (cudaOccupancyMaxActiveClusters(&n, kernel, &cfg) == cudaSuccess && n >= 1) return true;
    cudaGetLastError();
    return false;
}

// Blocks of the largest cluster (16, 8, 4, 2 or 1; 0: none) that the current device can place: of kernels[0] for any size, or of
// kernels[j] for 16 >> j blocks.  A whole B200 has room for 16 blocks that fill their SMs, a part of one need not.  `known`
// [kMaxDevices] remembers the answers (plus one).
int largest_cluster(const void *const *kernels, bool one_each, int threads, size_t smem, int *known)
{
    int dev = 0, most = -1;
    if (cudaGetDevice(&dev) != cudaSuccess || dev < 0) return 0;
    if (dev < kMaxDevices) most = __atomic_load_n(&known[dev], __ATOMIC_ACQUIRE) - 1;
    if (most < 0) {
        most = kChipMaxCluster;
        for (int j = 0; most >= 1 && !places_cluster(kernels[one_each ? j : 0], most, threads, smem); ++j) most >>= 1;
        if (dev < kMaxDevices) __atomic_store_n(&known[dev], most + 1, __ATOMIC_RELEASE);
    }
#ifdef G10_TEST_HOOKS
    // test build: a device that cannot place more than so many
    if (const char *h = getenv("G10_TEST_MAX_CLUSTER")) { const int cap = atoi(h); most = most < cap ? most : cap; }
#endif
    return most;
}

}  // namespace g10
