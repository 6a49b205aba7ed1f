// ppf_tmap.h -- host side: tensor maps for the boxes that TMA loads.
#pragma once

#include <cuda.h>
#include <cuda_runtime.h>

namespace ppf {

// Element type of a tensor map for items of `bytes` (box edges count items).
inline CUtensorMapDataType tmap_type(int bytes) {
    return bytes == 2 ? CU_TENSOR_MAP_DATA_TYPE_UINT16
         : bytes == 4 ? CU_TENSOR_MAP_DATA_TYPE_UINT32 : CU_TENSOR_MAP_DATA_TYPE_INT64;
}

// Rows of `cols` items of `bytes`, `rows` of them (row_bytes apart) in each of
// `planes` planes (plane_bytes apart), in boxes of box_cols x box_rows of one
// plane; planes = 0 makes the map two-dimensional.  Loads outside give zeros.
// base and the strides are multiples of 16 bytes, plane_bytes of row_bytes.
inline cudaError_t make_tmap(CUtensorMap* map, const void* base, int bytes, unsigned long long cols,
                             unsigned long long rows, unsigned long long row_bytes, unsigned long long planes,
                             unsigned long long plane_bytes, unsigned box_cols, unsigned box_rows) {
    using Encode = decltype(&cuTensorMapEncodeTiled);
    static const Encode encode = [] {
        void* fn = nullptr;
        cudaDriverEntryPointQueryResult found;
        if (cudaGetDriverEntryPointByVersion("cuTensorMapEncodeTiled", &fn, 12000, cudaEnableDefault, &found) != cudaSuccess ||
            found != cudaDriverEntryPointSuccess)
            fn = nullptr;
        return reinterpret_cast<Encode>(fn);
    }();
    if (encode == nullptr) return cudaErrorNotSupported;
    if (row_bytes % 16 != 0 || (planes > 0 && plane_bytes % row_bytes != 0)) return cudaErrorInvalidValue;
    const cuuint64_t dims[3] = {cols, rows, planes}, strides[2] = {row_bytes, plane_bytes};
    const cuuint32_t box[3] = {box_cols, box_rows, 1}, one[3] = {1, 1, 1};
    return encode(map, tmap_type(bytes), planes > 0 ? 3 : 2, const_cast<void*>(base), dims, strides, box, one,
                  CU_TENSOR_MAP_INTERLEAVE_NONE, CU_TENSOR_MAP_SWIZZLE_NONE, CU_TENSOR_MAP_L2_PROMOTION_L2_256B,
                  CU_TENSOR_MAP_FLOAT_OOB_FILL_NONE) == CUDA_SUCCESS
               ? cudaSuccess : cudaErrorInvalidValue;
}

}  // namespace ppf
