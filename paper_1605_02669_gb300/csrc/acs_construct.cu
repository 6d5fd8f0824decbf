// acs_construct.cu -- choice and launch of the construct kernel's variants.
#include <cstdint>
#include <mutex>

#include <cuda_runtime.h>

#include "acs_internal.cuh"

namespace acs {

template <int MODE, bool ALONE>
void* construct_variant(int tpa);   // acs_construct_variant.cu

// mode 0 matrix, 1 SPM with its working copies in global memory, 2 in shared memory
static void* select_kernel(int tpa, int mode, int csize)
{
    const bool alone = csize == 1;
    switch (mode) {
    case 0: return alone ? construct_variant<0, true>(tpa) : construct_variant<0, false>(tpa);
    case 1: return alone ? construct_variant<1, true>(tpa) : construct_variant<1, false>(tpa);
    case 2: return alone ? construct_variant<2, true>(tpa) : construct_variant<2, false>(tpa);
    default: return nullptr;
    }
}

// Raises the kernel's dynamic shared-memory limit to at least `smem` and
// allows clusters above 8 CTAs (outside any stream capture). The limit is a
// per-function setting shared by every context in the process, so it is only
// ever raised: lowering it would make the launches of an existing context
// with a larger layout fail.
cudaError_t prepare_construct(int tpa, int mode, int csize, size_t smem)
{
    static std::mutex mu;
    void* k = select_kernel(tpa, mode, csize);
    if (!k) return cudaErrorInvalidValue;
    std::lock_guard<std::mutex> lock(mu);
    cudaError_t e = cudaFuncSetAttribute(k, cudaFuncAttributeNonPortableClusterSizeAllowed, 1);
    if (e != cudaSuccess) return e;
    cudaFuncAttributes fa;
    e = cudaFuncGetAttributes(&fa, k);
    if (e != cudaSuccess) return e;
    if ((size_t)fa.maxDynamicSharedSizeBytes >= smem) return cudaSuccess;
    return cudaFuncSetAttribute(k, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem);
}

// Clusters of `csize` CTAs that can be resident at once (0 if none fits).
int construct_occupancy(int tpa, int mode, int block, size_t smem, int csize)
{
    void* k = select_kernel(tpa, mode, csize);
    if (!k) return 0;
    cudaLaunchConfig_t cfg = {};
    cfg.gridDim = dim3(csize);
    cfg.blockDim = dim3(block);
    cfg.dynamicSmemBytes = smem;
    cudaLaunchAttribute attr;
    attr.id = cudaLaunchAttributeClusterDimension;
    attr.val.clusterDim.x = csize;
    attr.val.clusterDim.y = 1;
    attr.val.clusterDim.z = 1;
    cfg.attrs = &attr;
    cfg.numAttrs = 1;
    int nclusters = 0;
    if (cudaOccupancyMaxActiveClusters(&nclusters, k, &cfg) != cudaSuccess) {
        cudaGetLastError();
        return 0;
    }
    return nclusters;
}

// Stream-ordered launch of one iteration on clusters of `csize` CTAs; safe
// inside a stream capture (the counter reset becomes a memset node). grid
// must be a multiple of csize.
cudaError_t launch_construct(const ConstructArgs& A, int tpa, int mode, int grid, int block,
                             size_t smem, int csize, cudaStream_t stream)
{
    void* k = select_kernel(tpa, mode, csize);
    if (!k) return cudaErrorInvalidValue;
    if (A.sched) {
        const cudaError_t e = cudaMemsetAsync(A.sched, 0, sizeof(int32_t), stream);
        if (e != cudaSuccess) return e;
    }
    cudaLaunchConfig_t cfg = {};
    cfg.gridDim = dim3(grid);
    cfg.blockDim = dim3(block);
    cfg.dynamicSmemBytes = smem;
    cfg.stream = stream;
    cudaLaunchAttribute attr;
    attr.id = cudaLaunchAttributeClusterDimension;
    attr.val.clusterDim.x = csize;
    attr.val.clusterDim.y = 1;
    attr.val.clusterDim.z = 1;
    cfg.attrs = &attr;
    cfg.numAttrs = 1;
    void* args[] = {const_cast<ConstructArgs*>(&A)};
    return cudaLaunchKernelExC(&cfg, k, args);
}

}  // namespace acs
