// Host side of the TMA loads: tensor maps of packed [rows, heads x head_dim] bf16 tensors.
#pragma once
#include <cuda.h>

#include "common.cuh"

namespace sp {

typedef CUresult (*EncodeTiledFn)(CUtensorMap *, CUtensorMapDataType, cuuint32_t, void *, const cuuint64_t *,
                                  const cuuint64_t *, const cuuint32_t *, const cuuint32_t *, CUtensorMapInterleave,
                                  CUtensorMapSwizzle, CUtensorMapL2promotion, CUtensorMapFloatOOBfill);

// [rows, cols] bf16 row-major seen as 3-D (64 columns, rows, cols / 64): a box of box_rows rows and one or all
// 64-column halves of a head lands as [half][row][64 columns] with the 128-byte swizzle, the layout the MMA
// descriptors expect.
inline int encode_rows_map(CUtensorMap *m, const void *base, int64_t rows, int64_t cols, int box_rows, int halves)
{
    static EncodeTiledFn enc = nullptr;
    if (!enc) {
        void *fn = nullptr;
        cudaDriverEntryPointQueryResult qres;
        SP_CUDA(cudaGetDriverEntryPoint("cuTensorMapEncodeTiled", &fn, cudaEnableDefault, &qres));
        SP_REQUIRE(fn != nullptr && qres == cudaDriverEntryPointSuccess, SP_ERR_CUDA,
                   "cuTensorMapEncodeTiled is not available from this driver");
        enc = reinterpret_cast<EncodeTiledFn>(fn);
    }
    cuuint64_t dims[3] = {64, (cuuint64_t)rows, (cuuint64_t)(cols / 64)};
    cuuint64_t strides[2] = {(cuuint64_t)cols * 2, 128};
    cuuint32_t box[3] = {64, (cuuint32_t)box_rows, (cuuint32_t)halves};
    cuuint32_t estr[3] = {1, 1, 1};
    const CUresult r = enc(m, CU_TENSOR_MAP_DATA_TYPE_BFLOAT16, 3, const_cast<void *>(base), dims, strides, box, estr,
                           CU_TENSOR_MAP_INTERLEAVE_NONE, CU_TENSOR_MAP_SWIZZLE_128B, CU_TENSOR_MAP_L2_PROMOTION_L2_128B,
                           CU_TENSOR_MAP_FLOAT_OOB_FILL_NONE);
    SP_REQUIRE(r == CUDA_SUCCESS, SP_ERR_CUDA, "cuTensorMapEncodeTiled failed with code %d", (int)r);
    return SP_OK;
}

}  // namespace sp
