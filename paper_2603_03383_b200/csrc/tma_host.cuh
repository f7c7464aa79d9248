// Host side of the 2-D TMA loads: a tensor map over a row-major bf16 matrix whose box is 64 columns
// (one 128-byte swizzle span) by box_rows rows, from the table of those already encoded.
#pragma once
#include "attn_common.cuh"

namespace mtv {

static inline bool tma_map_2d_bf16(CUtensorMap *map, const void *base, int rows, int H, int box_rows) {
    const cuuint64_t dims[2] = {(cuuint64_t)H, (cuuint64_t)rows};
    const cuuint64_t str[1] = {(cuuint64_t)H * 2};
    const cuuint32_t box[2] = {64, (cuuint32_t)box_rows};
    return tensor_map_bf16(map, base, 2, dims, str, box);
}

}  // namespace mtv
