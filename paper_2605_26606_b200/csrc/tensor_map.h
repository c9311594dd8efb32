// Host-side construction of TMA descriptors for row-major bf16 matrices [rows, cols] read as
// 128-byte-swizzled boxes of 64 columns x box_rows rows.  The driver entry point is looked up at run time
// so that the library loads on machines without a CUDA driver.
#pragma once

#include <cuda.h>
#include <cuda_runtime.h>

#include <cstdint>
#include <cstring>

namespace pc {

typedef CUresult (*EncodeTiledFn)(CUtensorMap*, CUtensorMapDataType, cuuint32_t, void*, const cuuint64_t*, const cuuint64_t*,
                                  const cuuint32_t*, const cuuint32_t*, CUtensorMapInterleave, CUtensorMapSwizzle,
                                  CUtensorMapL2promotion, CUtensorMapFloatOOBfill);

inline EncodeTiledFn encode_tiled_fn() {
    static EncodeTiledFn fn = nullptr;
    if (fn == nullptr) {
        void* p = nullptr;
        cudaDriverEntryPointQueryResult q;
        if (cudaGetDriverEntryPoint("cuTensorMapEncodeTiled", &p, cudaEnableDefault, &q) == cudaSuccess &&
            q == cudaDriverEntryPointSuccess)
            fn = reinterpret_cast<EncodeTiledFn>(p);
    }
    return fn;
}

// Returns false when the descriptor cannot be built (no driver, bad alignment, ...).
inline bool make_bf16_map(CUtensorMap* map, const void* base, uint64_t rows, uint64_t cols, uint32_t box_rows) {
    EncodeTiledFn fn = encode_tiled_fn();
    if (fn == nullptr) return false;
    const cuuint64_t gdim[2] = {cols, rows};
    const cuuint64_t gstride[1] = {cols * 2};
    const cuuint32_t box[2] = {64, box_rows};
    const cuuint32_t estride[2] = {1, 1};
    std::memset(map, 0, sizeof(*map));
    return fn(map, CU_TENSOR_MAP_DATA_TYPE_BFLOAT16, 2, const_cast<void*>(base), gdim, gstride, box, estride,
              CU_TENSOR_MAP_INTERLEAVE_NONE, CU_TENSOR_MAP_SWIZZLE_128B, CU_TENSOR_MAP_L2_PROMOTION_L2_256B,
              CU_TENSOR_MAP_FLOAT_OOB_FILL_NONE) == CUDA_SUCCESS;
}

// A KV arena [planes][n_slots][head_dim] of 16-bit elements, planes = layer x (K | V) x KV head, read as tiles of box_rows
// consecutive slots that hold K and V of one (layer, KV head): coordinates (0, row of the K plane, 0, 0), the third dimension
// being the 64-element halves of head_dim and the fourth K | V.  In shared memory a tile is [K|V][half][slot][64], swizzled.
inline bool make_kv_tile_map(CUtensorMap* map, const void* base, uint64_t planes, uint64_t n_slots, uint64_t n_kv_heads, uint64_t head_dim,
                             uint32_t box_rows) {
    EncodeTiledFn fn = encode_tiled_fn();
    if (fn == nullptr) return false;
    const cuuint64_t gdim[4] = {64, planes * n_slots - n_kv_heads * n_slots, head_dim / 64, 2};
    const cuuint64_t gstride[3] = {head_dim * 2, 128, n_kv_heads * n_slots * head_dim * 2};
    const cuuint32_t box[4] = {64, box_rows, (cuuint32_t)(head_dim / 64), 2};
    const cuuint32_t estride[4] = {1, 1, 1, 1};
    std::memset(map, 0, sizeof(*map));
    return fn(map, CU_TENSOR_MAP_DATA_TYPE_BFLOAT16, 4, const_cast<void*>(base), gdim, gstride, box, estride,
              CU_TENSOR_MAP_INTERLEAVE_NONE, CU_TENSOR_MAP_SWIZZLE_128B, CU_TENSOR_MAP_L2_PROMOTION_L2_256B,
              CU_TENSOR_MAP_FLOAT_OOB_FILL_NONE) == CUDA_SUCCESS;
}

}  // namespace pc
