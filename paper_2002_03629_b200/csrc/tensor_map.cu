// Tensor maps (cuTensorMapEncodeTiled, reached through the runtime's entry-point query: the library does not link libcuda).
#include <cuda.h>

#include "js_common.cuh"
#include "js_model.h"

typedef CUresult (*EncodeTiledFn)(CUtensorMap *, CUtensorMapDataType, cuuint32_t, void *, const cuuint64_t *,
                                  const cuuint64_t *, const cuuint32_t *, const cuuint32_t *, CUtensorMapInterleave,
                                  CUtensorMapSwizzle, CUtensorMapL2promotion, CUtensorMapFloatOOBfill);

static EncodeTiledFn encode_fn()
{
    static EncodeTiledFn fn = nullptr;
    if (fn) return fn;
    void *p = nullptr;
    cudaDriverEntryPointQueryResult q;
    if (cudaGetDriverEntryPoint("cuTensorMapEncodeTiled", &p, cudaEnableDefault, &q) != cudaSuccess ||
        q != cudaDriverEntryPointSuccess)
        return nullptr;
    fn = (EncodeTiledFn)p;
    return fn;
}

bool js_tensor_maps() { return encode_fn() != nullptr; }

// up to four dimensions, innermost first; 128-byte swizzle, zeros outside the tensor
bool js_encode_map(CUtensorMap *out, CUtensorMapDataType type, const void *base, int rank, const cuuint64_t *dims,
                   const cuuint64_t *strides, const cuuint32_t *box)
{
    EncodeTiledFn fn = encode_fn();
    if (!fn) return false;
    const cuuint32_t estr[4] = {1, 1, 1, 1};
    return fn(out, type, rank, const_cast<void *>(base), dims, strides, box, estr, CU_TENSOR_MAP_INTERLEAVE_NONE,
              CU_TENSOR_MAP_SWIZZLE_128B, CU_TENSOR_MAP_L2_PROMOTION_L2_256B, CU_TENSOR_MAP_FLOAT_OOB_FILL_NONE) == CUDA_SUCCESS;
}

// row-major [rows][cols], rows row_stride values apart (0: cols), box = box_cols columns (128 bytes) x box_rows rows
bool js_encode_map_2d(CUtensorMap *out, CUtensorMapDataType type, const void *base, int rows, int cols, int box_cols, int box_rows,
                      int row_stride)
{
    const cuuint64_t dims[2] = {(cuuint64_t)cols, (cuuint64_t)rows};
    const cuuint64_t strides[1] = {(cuuint64_t)(row_stride ? row_stride : cols) * (type == CU_TENSOR_MAP_DATA_TYPE_FLOAT32 ? 4 : 2)};
    const cuuint32_t box[2] = {(cuuint32_t)box_cols, (cuuint32_t)box_rows};
    return js_encode_map(out, type, base, 2, dims, strides, box);
}
