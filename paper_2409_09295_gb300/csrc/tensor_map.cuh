// Tensor maps for the TMA copies of the convolution kernels (host side).
#pragma once
#include <cudaTypedefs.h>

#include "gevo_internal.cuh"

namespace gevo {

// A five-dimensional BF16 map, zeros outside the tensor.  strides: bytes of
// dimensions 1 to 4.
inline bool encode_map_bf16(CUtensorMap& map, const void* p, const uint64_t dims[5],
                            const uint64_t strides[4], const uint32_t box[5])
{
    static const PFN_cuTensorMapEncodeTiled_v12000 encode = [] {
        void* f = nullptr;
        cudaDriverEntryPointQueryResult q;
        if (cudaGetDriverEntryPointByVersion("cuTensorMapEncodeTiled", &f, 12000, cudaEnableDefault, &q) !=
                cudaSuccess ||
            q != cudaDriverEntryPointSuccess)
            f = nullptr;
        return reinterpret_cast<PFN_cuTensorMapEncodeTiled_v12000>(f);
    }();
    if (!encode) return false;
    cuuint64_t d[5], s[4];
    cuuint32_t b[5], one[5];
    for (int i = 0; i < 5; i++) {
        d[i] = dims[i];
        b[i] = box[i];
        one[i] = 1;
        if (i < 4) s[i] = strides[i];
    }
    return encode(&map, CU_TENSOR_MAP_DATA_TYPE_BFLOAT16, 5, const_cast<void*>(p), d, s, b, one,
                  CU_TENSOR_MAP_INTERLEAVE_NONE, CU_TENSOR_MAP_SWIZZLE_NONE,
                  CU_TENSOR_MAP_L2_PROMOTION_L2_128B, CU_TENSOR_MAP_FLOAT_OOB_FILL_NONE) == CUDA_SUCCESS;
}

// NHWC activations as (8 channels, x, y, channel group, image): a box of bx x by pixels
// and bg groups lands as planes of eight channels, 16 bytes a pixel.  The innermost
// coordinate is always 0, so every copy starts on a 16-byte boundary.
inline bool nhwc_planes_map(CUtensorMap& map, const void* X, int nb, int H, int W, int C, int bx, int by,
                            int bg)
{
    const uint64_t row = (uint64_t)C * 2;
    const uint64_t dims[5] = {8, (uint64_t)W, (uint64_t)H, (uint64_t)(C / 8), (uint64_t)nb};
    const uint64_t strides[4] = {row, row * W, 16, row * W * H};
    const uint32_t box[5] = {8, (uint32_t)bx, (uint32_t)by, (uint32_t)bg, 1};
    return encode_map_bf16(map, X, dims, strides, box);
}

}  // namespace gevo
