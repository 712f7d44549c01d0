// What the current device lets a kernel have.
#include <cuda.h>

#include <cstdlib>

#include "g10_internal.h"

namespace g10 {

// Dynamic shared memory that a block of `kernel` can be given on the current device (the most a block can opt in to, minus the kernel's
// static part; 0 if a query fails).  `known` [kMaxDevices] remembers it.
int dynamic_smem_room(const void *kernel, int *known)
{
    int dev = 0, optin = 0;
    cudaFuncAttributes fa;
    if (cudaGetDevice(&dev) != cudaSuccess || dev < 0) return 0;
    if (dev < kMaxDevices) if (const int b = __atomic_load_n(&known[dev], __ATOMIC_ACQUIRE)) return b;
    if (cudaDeviceGetAttribute(&optin, cudaDevAttrMaxSharedMemoryPerBlockOptin, dev) != cudaSuccess) return 0;
    if (cudaFuncGetAttributes(&fa, kernel) != cudaSuccess) return 0;
    const int room = optin - (int)fa.sharedSizeBytes;
    if (room <= 0) return 0;
    if (dev < kMaxDevices) __atomic_store_n(&known[dev], room, __ATOMIC_RELEASE);
    return room;
}

// Allows `kernel` so much dynamic shared memory, and clusters of so many blocks, on the current device.  For every launch: what was
// allowed once is gone after cudaDeviceReset.  (The same amount each time, not what one launch needs: threads may launch side by side.)
cudaError_t allow_launch(const void *kernel, size_t smem, int cluster)
{
    cudaError_t e = cudaSuccess;
    if (smem != 0) e = cudaFuncSetAttribute(kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem);
    if (e == cudaSuccess && cluster > 8) e = cudaFuncSetAttribute(kernel, cudaFuncAttributeNonPortableClusterSizeAllowed, 1);
    return e;
}

// Can the current device place a cluster of so many blocks of `kernel` with so much dynamic shared memory each?
static bool places_cluster(const void *kernel, int blocks, int threads, size_t smem)
{
    cudaLaunchConfig_t cfg = {};
    cudaLaunchAttribute at[1];
    at[0].id = cudaLaunchAttributeClusterDimension;
    at[0].val.clusterDim.x = (unsigned)blocks; at[0].val.clusterDim.y = 1; at[0].val.clusterDim.z = 1;
    cfg.gridDim = dim3((unsigned)blocks); cfg.blockDim = dim3((unsigned)threads); cfg.dynamicSmemBytes = smem; cfg.attrs = at; cfg.numAttrs = 1;
    int n = 0;
    if (allow_launch(kernel, smem, blocks) == cudaSuccess && cudaOccupancyMaxActiveClusters(&n, kernel, &cfg) == cudaSuccess && n >= 1) return true;
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

// The device's address of pinned host memory if all `bytes` from p on lie in ONE pinned range, else null: memory may be registered in
// pieces, and a kernel that reads past one faults where a copy returns an error.
void *pinned_address(const void *p, size_t bytes)
{
    typedef CUresult (*Query)(unsigned, CUpointer_attribute *, void **, CUdeviceptr);
    static void *known = nullptr;                    // (the driver's function: the same in every thread)
    void *f = __atomic_load_n(&known, __ATOMIC_ACQUIRE);
    if (f == nullptr) {
        cudaDriverEntryPointQueryResult found;
        if (cudaGetDriverEntryPoint("cuPointerGetAttributes", &f, cudaEnableDefault, &found) != cudaSuccess || found != cudaDriverEntryPointSuccess) {
            cudaGetLastError();
            return nullptr;
        }
        __atomic_store_n(&known, f, __ATOMIC_RELEASE);
    }
    CUmemorytype type = (CUmemorytype)0;
    CUdeviceptr start = 0;
    void *device = nullptr;
    size_t size = 0;
    int managed = 0;
    CUpointer_attribute what[] = {CU_POINTER_ATTRIBUTE_MEMORY_TYPE, CU_POINTER_ATTRIBUTE_DEVICE_POINTER, CU_POINTER_ATTRIBUTE_RANGE_START_ADDR,
                                  CU_POINTER_ATTRIBUTE_RANGE_SIZE, CU_POINTER_ATTRIBUTE_IS_MANAGED};
    void *to[] = {&type, &device, &start, &size, &managed};
    if (((Query)f)(5, what, to, (CUdeviceptr)(uintptr_t)p) != CUDA_SUCCESS || type != CU_MEMORYTYPE_HOST || managed) return nullptr;
    const uintptr_t at = (uintptr_t)p;
    if ((uintptr_t)device != at || start == 0 || at < start || bytes > size || at - start > size - bytes) return nullptr;
    return device;
}

#ifdef G10_TEST_HOOKS
extern "C" int32_t g10_test_reads_in_place(const void *p, size_t bytes) { return pinned_address(p, bytes) != nullptr; }
// For a test that resets the device under the library: the reset, and device memory of the library's own runtime.
extern "C" int32_t g10_test_device_reset(void) { return (int32_t)cudaDeviceReset(); }
extern "C" void *g10_test_upload(const void *src, size_t bytes)
{
    void *p = nullptr;
    if (cudaMalloc(&p, bytes) != cudaSuccess || (src != nullptr && cudaMemcpy(p, src, bytes, cudaMemcpyHostToDevice) != cudaSuccess)) return nullptr;
    return p;
}
extern "C" int32_t g10_test_download(void *dst, const void *src, size_t bytes) { return (int32_t)cudaMemcpy(dst, src, bytes, cudaMemcpyDeviceToHost); }
#endif

}  // namespace g10
