// Host side of the tensor maps (TMA descriptors) and of the launches the tcgen05 kernels share.
#pragma once
#include <cuda.h>
#include <cuda_runtime.h>

namespace slimspec {

typedef CUresult (*EncodeTiledFn)(CUtensorMap*, CUtensorMapDataType, cuuint32_t, void*, const cuuint64_t*,
                                  const cuuint64_t*, const cuuint32_t*, const cuuint32_t*, CUtensorMapInterleave,
                                  CUtensorMapSwizzle, CUtensorMapL2promotion, CUtensorMapFloatOOBfill);

inline EncodeTiledFn encode_fn()
{
    static const EncodeTiledFn fn = [] {
        void* ptr = nullptr;
        cudaDriverEntryPointQueryResult qr;
        if (cudaGetDriverEntryPoint("cuTensorMapEncodeTiled", &ptr, cudaEnableDefault, &qr) != cudaSuccess ||
            qr != cudaDriverEntryPointSuccess)
            ptr = nullptr;
        return (EncodeTiledFn)ptr;
    }();
    return fn;
}

// bf16 matrix [rows][cols], rows `pitch` elements apart (a multiple of 8), cols contiguous; box = box_cols x box_rows.
// The swizzle follows from the box's row: 64 columns are a 128-byte row, 32 columns a 64-byte row.  Reads
// outside the matrix give zeros.
inline bool make_map_pitched(CUtensorMap* map, const void* base, int rows, int cols, long long pitch, int box_cols, int box_rows)
{
    EncodeTiledFn fn = encode_fn();
    if (!fn) return false;
    cuuint64_t dims[2] = {(cuuint64_t)cols, (cuuint64_t)rows};
    cuuint64_t strides[1] = {(cuuint64_t)pitch * 2};
    cuuint32_t box[2] = {(cuuint32_t)box_cols, (cuuint32_t)box_rows};
    cuuint32_t es[2] = {1, 1};
    return fn(map, CU_TENSOR_MAP_DATA_TYPE_BFLOAT16, 2, const_cast<void*>(base), dims, strides, box, es,
              CU_TENSOR_MAP_INTERLEAVE_NONE, box_cols == 32 ? CU_TENSOR_MAP_SWIZZLE_64B : CU_TENSOR_MAP_SWIZZLE_128B,
              CU_TENSOR_MAP_L2_PROMOTION_L2_256B, CU_TENSOR_MAP_FLOAT_OOB_FILL_NONE) == CUDA_SUCCESS;
}

inline bool make_map(CUtensorMap* map, const void* base, int rows, int cols, int box_cols, int box_rows)
{
    return make_map_pitched(map, base, rows, cols, cols, box_cols, box_rows);
}

// Launch with (or without) the programmatic-dependent-launch attribute: the kernel may start while
// the one before it in the stream is still running and meets it at griddepcontrol.wait.  cluster: CTAs of a cluster.
template <typename... KArgs, typename... Args>
static cudaError_t launch_chain_cluster(void (*kern)(KArgs...), int grid, int cluster, int block, size_t smem, bool pdl, cudaStream_t st,
                                        Args... args)
{
    cudaLaunchConfig_t cfg = {};
    cfg.gridDim = dim3(grid);
    cfg.blockDim = dim3(block);
    cfg.dynamicSmemBytes = smem;
    cfg.stream = st;
    cudaLaunchAttribute attr[2];
    int n = 0;
    if (pdl) {
        attr[n].id = cudaLaunchAttributeProgrammaticStreamSerialization;
        attr[n++].val.programmaticStreamSerializationAllowed = 1;
    }
    if (cluster > 1) {
        attr[n].id = cudaLaunchAttributeClusterDimension;
        attr[n].val.clusterDim.x = (unsigned)cluster;
        attr[n].val.clusterDim.y = 1;
        attr[n++].val.clusterDim.z = 1;
    }
    cfg.attrs = attr;
    cfg.numAttrs = n;
    return cudaLaunchKernelEx(&cfg, kern, args...);
}

template <typename... KArgs, typename... Args>
static cudaError_t launch_chain(void (*kern)(KArgs...), int grid, int block, size_t smem, bool pdl, cudaStream_t st,
                                Args... args)
{
    return launch_chain_cluster(kern, grid, 1, block, smem, pdl, st, args...);
}

}  // namespace slimspec
