// Host helper: tensor maps for TMA copies (128-byte swizzle, out-of-range elements read as 0).
#pragma once
#include <cuda.h>
#include <stdint.h>

namespace obc {

// `planes` dense matrices of rows x inner elements one after the other; box_inner * elem_bytes must be 128, the base 16-byte
// aligned and inner * elem_bytes a multiple of 16.
bool make_tensor_map_3d(CUtensorMap* map, CUtensorMapDataType type, int elem_bytes, const void* base, int64_t inner, int64_t rows,
                        int64_t planes, int box_inner, int box_rows, int box_planes);

}  // namespace obc
