// acs_construct.cu -- choice and launch of the construct kernel's variants.
#include <cstdint>
#include <mutex>

#include <cuda_runtime.h>

#include "acs_internal.cuh"

namespace acs {

template <int MODE, bool ALONE, int KIND>
void* construct_variant(int lanes);   // acs_construct_variant.cu

template <int MODE>
static void* select_mode(int lanes, bool alone, int kind)
{
    switch (kind) {
    case kShort: return alone ? construct_variant<MODE, true, kShort>(lanes) : construct_variant<MODE, false, kShort>(lanes);
    case kLong: return alone ? nullptr : construct_variant<MODE, false, kLong>(lanes);
    case kTurns: return alone ? construct_variant<MODE, true, kTurns>(lanes) : construct_variant<MODE, false, kTurns>(lanes);
    default: return nullptr;
    }
}

// mode 0 matrix, 1 SPM with its working copies in global memory, 2 in shared memory
static void* select_kernel(int lanes, int mode, int csize, int kind)
{
    switch (mode) {
    case 0: return select_mode<0>(lanes, csize == 1, kind);
    case 1: return select_mode<1>(lanes, csize == 1, kind);
    case 2: return select_mode<2>(lanes, csize == 1, kind);
    default: return nullptr;
    }
}

// Raises the kernel's dynamic shared-memory limit to at least `smem` and
// allows clusters above 8 CTAs (outside any stream capture). The limit is a
// per-function setting shared by every context in the process, so it is only
// ever raised: lowering it would make the launches of an existing context
// with a larger layout fail.
cudaError_t prepare_construct(int lanes, int mode, int csize, int kind, size_t smem)
{
    static std::mutex mu;
    void* k = select_kernel(lanes, mode, csize, kind);
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
int construct_occupancy(int lanes, int mode, int block, size_t smem, int csize, int kind)
{
    void* k = select_kernel(lanes, mode, csize, kind);
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
cudaError_t launch_construct(const ConstructArgs& A, int lanes, int mode, int kind, int grid, int block,
                             size_t smem, int csize, cudaStream_t stream)
{
    void* k = select_kernel(lanes, mode, csize, kind);
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
