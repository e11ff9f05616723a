// Host-side construction of TMA tensor maps for the KV pools (used by the tile and the streaming kernel).
// cuTensorMapEncodeTiled is fetched through the runtime's driver entry point, so nothing links against libcuda.
#pragma once
#include <cuda.h>
#include <cuda_runtime.h>
#include <stdint.h>

namespace hat {

typedef CUresult (*EncodeTiledFn)(CUtensorMap*, CUtensorMapDataType, cuuint32_t, void*, const cuuint64_t*,
                                  const cuuint64_t*, const cuuint32_t*, const cuuint32_t*, CUtensorMapInterleave,
                                  CUtensorMapSwizzle, CUtensorMapL2promotion, CUtensorMapFloatOOBfill);

inline EncodeTiledFn tma_encode_fn() {
    static EncodeTiledFn fn = [] {
        void* p = nullptr;
        cudaDriverEntryPointQueryResult q;
        if (cudaGetDriverEntryPoint("cuTensorMapEncodeTiled", &p, cudaEnableDefault, &q) != cudaSuccess ||
            q != cudaDriverEntryPointSuccess)
            p = nullptr;
        return reinterpret_cast<EncodeTiledFn>(p);
    }();
    return fn;
}

// A K or V pool as a 4-D tensor (column, slot, head, page) read in boxes of 64 columns x 16 slots (one page of one
// head, one 128-byte column half) with the 128-byte shared-memory swizzle.  Strides are in elements.
inline bool tma_encode_pool_map(CUtensorMap* map, bool bf16, const void* pool, int head_dim, int num_pages, int H,
                                int64_t stride_page, int64_t stride_token, int64_t stride_head) {
    EncodeTiledFn fn = tma_encode_fn();
    if (!fn || num_pages <= 0) return false;
    const cuuint64_t dims[4] = {(cuuint64_t)head_dim, 16, (cuuint64_t)H, (cuuint64_t)num_pages};
    const cuuint64_t strides[3] = {(cuuint64_t)stride_token * 2, (cuuint64_t)stride_head * 2, (cuuint64_t)stride_page * 2};
    const cuuint32_t box[4] = {64, 16, 1, 1};
    const cuuint32_t estr[4] = {1, 1, 1, 1};
    return fn(map, bf16 ? CU_TENSOR_MAP_DATA_TYPE_BFLOAT16 : CU_TENSOR_MAP_DATA_TYPE_FLOAT16, 4, const_cast<void*>(pool),
              dims, strides, box, estr, CU_TENSOR_MAP_INTERLEAVE_NONE, CU_TENSOR_MAP_SWIZZLE_128B,
              CU_TENSOR_MAP_L2_PROMOTION_L2_256B, CU_TENSOR_MAP_FLOAT_OOB_FILL_NONE) == CUDA_SUCCESS;
}

// The same pool with the column halves as a dimension, (column of a half, slot, half, head, page), read in boxes that hold
// one whole page of one head: the halves land one after the other, 2 KiB each, as two boxes of the map above would.
inline bool tma_encode_page_map(CUtensorMap* map, bool bf16, const void* pool, int head_dim, int num_pages, int H,
                                int64_t stride_page, int64_t stride_token, int64_t stride_head) {
    EncodeTiledFn fn = tma_encode_fn();
    if (!fn || num_pages <= 0) return false;
    const cuuint64_t dims[5] = {64, 16, (cuuint64_t)head_dim / 64, (cuuint64_t)H, (cuuint64_t)num_pages};
    const cuuint64_t strides[4] = {(cuuint64_t)stride_token * 2, 128, (cuuint64_t)stride_head * 2, (cuuint64_t)stride_page * 2};
    const cuuint32_t box[5] = {64, 16, (cuuint32_t)head_dim / 64, 1, 1};
    const cuuint32_t estr[5] = {1, 1, 1, 1, 1};
    return fn(map, bf16 ? CU_TENSOR_MAP_DATA_TYPE_BFLOAT16 : CU_TENSOR_MAP_DATA_TYPE_FLOAT16, 5, const_cast<void*>(pool),
              dims, strides, box, estr, CU_TENSOR_MAP_INTERLEAVE_NONE, CU_TENSOR_MAP_SWIZZLE_128B,
              CU_TENSOR_MAP_L2_PROMOTION_L2_256B, CU_TENSOR_MAP_FLOAT_OOB_FILL_NONE) == CUDA_SUCCESS;
}

// The same pool for the tile kernels: boxes that hold a whole page of one head as the tensor core's 8-row groups, i.e.
// (column of a half, slot of a group, half, group): 1 KiB blocks, so that a tile of several pages is one operand with a uniform
// distance of head_dim * 16 bytes between groups.  The group is a dimension beside head or page, whichever stride it
// divides evenly (*fold = 1: the head coordinate is 2 h; 2: the page coordinate is 2 page); other strides take two boxes per
// page, by the slot coordinate (*fold = 0).
inline bool tma_encode_tile_map(CUtensorMap* map, bool bf16, const void* pool, int head_dim, int num_pages, int H,
                                int64_t stride_page, int64_t stride_token, int64_t stride_head, int* fold) {
    EncodeTiledFn fn = tma_encode_fn();
    if (!fn || num_pages <= 0) return false;
    const cuuint32_t halves = (cuuint32_t)head_dim / 64;
    *fold = stride_head == 16 * stride_token ? 1 : stride_page == 16 * stride_token ? 2 : 0;
    const cuuint64_t tok = (cuuint64_t)stride_token * 2, hd = (cuuint64_t)stride_head * 2, pg = (cuuint64_t)stride_page * 2;
    const cuuint64_t dims[5] = {64, *fold ? 8u : 16u, halves, (cuuint64_t)H * (*fold == 1 ? 2 : 1), (cuuint64_t)num_pages * (*fold == 2 ? 2 : 1)};
    const cuuint64_t strides[4] = {tok, 128, *fold == 1 ? 8 * tok : hd, *fold == 2 ? 8 * tok : pg};
    const cuuint32_t box[5] = {64, 8, halves, *fold == 1 ? 2u : 1u, *fold == 2 ? 2u : 1u};
    const cuuint32_t estr[5] = {1, 1, 1, 1, 1};
    return fn(map, bf16 ? CU_TENSOR_MAP_DATA_TYPE_BFLOAT16 : CU_TENSOR_MAP_DATA_TYPE_FLOAT16, 5, const_cast<void*>(pool),
              dims, strides, box, estr, CU_TENSOR_MAP_INTERLEAVE_NONE, CU_TENSOR_MAP_SWIZZLE_128B,
              CU_TENSOR_MAP_L2_PROMOTION_L2_256B, CU_TENSOR_MAP_FLOAT_OOB_FILL_NONE) == CUDA_SUCCESS;
}

// Packed rows k_new / v_new [T][H][d] as (column of a half, row, half, head), read in boxes of box_rows rows and box_halves
// column halves of one head.
inline bool tma_encode_new_map(CUtensorMap* map, bool bf16, const void* base, int T, int H, int head_dim, int box_rows, int box_halves) {
    EncodeTiledFn fn = tma_encode_fn();
    if (!fn) return false;
    const cuuint64_t dims[4] = {64, (cuuint64_t)T, (cuuint64_t)head_dim / 64, (cuuint64_t)H};
    const cuuint64_t strides[3] = {(cuuint64_t)H * head_dim * 2, 128, (cuuint64_t)head_dim * 2};
    const cuuint32_t box[4] = {64, (cuuint32_t)box_rows, (cuuint32_t)box_halves, 1};
    const cuuint32_t estr[4] = {1, 1, 1, 1};
    return fn(map, bf16 ? CU_TENSOR_MAP_DATA_TYPE_BFLOAT16 : CU_TENSOR_MAP_DATA_TYPE_FLOAT16, 4, const_cast<void*>(base),
              dims, strides, box, estr, CU_TENSOR_MAP_INTERLEAVE_NONE, CU_TENSOR_MAP_SWIZZLE_128B,
              CU_TENSOR_MAP_L2_PROMOTION_L2_256B, CU_TENSOR_MAP_FLOAT_OOB_FILL_NONE) == CUDA_SUCCESS;
}

// The query rows [T][H][d] as a 3-D tensor (column, head, row) read in boxes of 64 columns x 128 rows of one head.
inline bool tma_encode_q_map(CUtensorMap* map, bool bf16, const void* q, int T, int H, int head_dim) {
    EncodeTiledFn fn = tma_encode_fn();
    if (!fn) return false;
    const cuuint64_t dims[3] = {(cuuint64_t)head_dim, (cuuint64_t)H, (cuuint64_t)T};
    const cuuint64_t strides[2] = {(cuuint64_t)head_dim * 2, (cuuint64_t)H * head_dim * 2};
    const cuuint32_t box[3] = {64, 1, 128};
    const cuuint32_t estr[3] = {1, 1, 1};
    return fn(map, bf16 ? CU_TENSOR_MAP_DATA_TYPE_BFLOAT16 : CU_TENSOR_MAP_DATA_TYPE_FLOAT16, 3, const_cast<void*>(q), dims,
              strides, box, estr, CU_TENSOR_MAP_INTERLEAVE_NONE, CU_TENSOR_MAP_SWIZZLE_128B,
              CU_TENSOR_MAP_L2_PROMOTION_L2_256B, CU_TENSOR_MAP_FLOAT_OOB_FILL_NONE) == CUDA_SUCCESS;
}

// A row-major 16-bit matrix [rows][cols] as a 2-D tensor (column, row) read in boxes of 64 columns x box_rows rows.
inline bool tma_encode_matrix_map(CUtensorMap* map, bool bf16, const void* base, int64_t rows, int64_t cols, int box_rows) {
    EncodeTiledFn fn = tma_encode_fn();
    if (!fn || rows <= 0 || cols <= 0) return false;
    const cuuint64_t dims[2] = {(cuuint64_t)cols, (cuuint64_t)rows};
    const cuuint64_t strides[1] = {(cuuint64_t)cols * 2};
    const cuuint32_t box[2] = {64, (cuuint32_t)box_rows};
    const cuuint32_t estr[2] = {1, 1};
    return fn(map, bf16 ? CU_TENSOR_MAP_DATA_TYPE_BFLOAT16 : CU_TENSOR_MAP_DATA_TYPE_FLOAT16, 2, const_cast<void*>(base), dims,
              strides, box, estr, CU_TENSOR_MAP_INTERLEAVE_NONE, CU_TENSOR_MAP_SWIZZLE_128B,
              CU_TENSOR_MAP_L2_PROMOTION_L2_256B, CU_TENSOR_MAP_FLOAT_OOB_FILL_NONE) == CUDA_SUCCESS;
}

}  // namespace hat
