// 2-D TMA tensor maps, encoded by the driver on the host.
#pragma once

#include <cstdint>

#include <cuda.h>

namespace pvs {

// Row-major matrix of `elem`-byte elements, boxes of box_cols x box_rows, 128-byte
// swizzle, elements past the matrix read as zero; false when the driver refuses it.
bool tensor_map_2d(CUtensorMap* m, CUtensorMapDataType type, int elem, const void* base,
                   uint64_t rows, uint64_t cols, uint32_t box_cols, uint32_t box_rows);

}  // namespace pvs
