// Host-side encoding of TMA tensor maps (128-byte swizzle, zero fill outside the tensor).
#pragma once

#include <cuda.h>
#include <cuda_runtime.h>
#include <stdint.h>

namespace eql {

typedef CUresult (*EncodeTiledFn)(CUtensorMap*, CUtensorMapDataType, cuuint32_t, void*, const cuuint64_t*,
                                  const cuuint64_t*, const cuuint32_t*, const cuuint32_t*, CUtensorMapInterleave,
                                  CUtensorMapSwizzle, CUtensorMapL2promotion, CUtensorMapFloatOOBfill);

inline EncodeTiledFn tensor_map_encoder() {
    static const EncodeTiledFn fn = [] {
        void* p = nullptr;
        cudaDriverEntryPointQueryResult q;
        if (cudaGetDriverEntryPoint("cuTensorMapEncodeTiled", &p, cudaEnableDefault, &q) != cudaSuccess ||
            q != cudaDriverEntryPointSuccess)
            p = nullptr;
        return reinterpret_cast<EncodeTiledFn>(p);
    }();
    return fn;
}

inline bool encode_map(CUtensorMap* map, const void* base, int rank, const cuuint64_t* dim, const cuuint64_t* stride_bytes,
                       const cuuint32_t* box, int elem_bytes) {
    const EncodeTiledFn enc = tensor_map_encoder();
    if (enc == nullptr) return false;
    const cuuint32_t ones[4] = {1, 1, 1, 1};
    return enc(map, elem_bytes == 4 ? CU_TENSOR_MAP_DATA_TYPE_FLOAT32 : CU_TENSOR_MAP_DATA_TYPE_FLOAT16, (cuuint32_t)rank,
               const_cast<void*>(base), dim, stride_bytes, box, ones, CU_TENSOR_MAP_INTERLEAVE_NONE,
               CU_TENSOR_MAP_SWIZZLE_128B, CU_TENSOR_MAP_L2_PROMOTION_L2_128B, CU_TENSOR_MAP_FLOAT_OOB_FILL_NONE) == CUDA_SUCCESS;
}
// [rows][cols] elements with a row pitch, box [box_rows][box_cols]
inline bool encode_map_2d(CUtensorMap* map, const void* base, int64_t cols, int64_t rows, int64_t pitch, int box_cols,
                          int box_rows, int elem_bytes) {
    const cuuint64_t dim[2] = {(cuuint64_t)cols, (cuuint64_t)rows};
    const cuuint64_t stride[1] = {(cuuint64_t)(pitch * elem_bytes)};
    const cuuint32_t box[2] = {(cuuint32_t)box_cols, (cuuint32_t)box_rows};
    return encode_map(map, base, 2, dim, stride, box, elem_bytes);
}
// [rows][slabs of 128 bytes] of a matrix whose rows are whole slabs (or padded to them), box [box_slabs][box_rows][128 bytes]:
// one copy brings several slabs, one behind the other.
// The plane form: two matrices plane_pitch elements apart, both in every box.
inline bool encode_map_slabs(CUtensorMap* map, const void* base, int64_t slabs, int64_t rows, int64_t pitch, int box_slabs,
                             int box_rows, int elem_bytes) {
    const cuuint64_t dim[3] = {(cuuint64_t)(128 / elem_bytes), (cuuint64_t)rows, (cuuint64_t)slabs};
    const cuuint64_t stride[2] = {(cuuint64_t)(pitch * elem_bytes), 128};
    const cuuint32_t box[3] = {(cuuint32_t)(128 / elem_bytes), (cuuint32_t)box_rows, (cuuint32_t)box_slabs};
    return encode_map(map, base, 3, dim, stride, box, elem_bytes);
}
inline bool encode_map_plane_slabs(CUtensorMap* map, const void* base, int64_t slabs, int64_t rows, int64_t pitch,
                                   int64_t plane_pitch, int box_slabs, int box_rows, int elem_bytes) {
    const cuuint64_t dim[4] = {(cuuint64_t)(128 / elem_bytes), (cuuint64_t)rows, 2, (cuuint64_t)slabs};
    const cuuint64_t stride[3] = {(cuuint64_t)(pitch * elem_bytes), (cuuint64_t)(plane_pitch * elem_bytes), 128};
    const cuuint32_t box[4] = {(cuuint32_t)(128 / elem_bytes), (cuuint32_t)box_rows, 2, (cuuint32_t)box_slabs};
    return encode_map(map, base, 4, dim, stride, box, elem_bytes);
}

}  // namespace eql
