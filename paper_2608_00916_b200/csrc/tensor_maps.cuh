// Tensor maps (copy-engine descriptors) of the operands, all bf16 with the 128-byte swizzle.
#pragma once
#include <cuda.h>
#include <stdint.h>

namespace moe {

typedef CUresult (*EncodeTiledFn)(CUtensorMap*, CUtensorMapDataType, cuuint32_t, void*, const cuuint64_t*,
                                  const cuuint64_t*, const cuuint32_t*, const cuuint32_t*, CUtensorMapInterleave,
                                  CUtensorMapSwizzle, CUtensorMapL2promotion, CUtensorMapFloatOOBfill);

// bf16 row-major [rows, width] -> 2D map with box {64, box_rows}
inline bool map_2d(void* fn, CUtensorMap* m, const void* base, int64_t rows, int64_t width, int box_rows) {
  cuuint64_t dims[2] = {static_cast<cuuint64_t>(width), static_cast<cuuint64_t>(rows)};
  cuuint64_t strides[1] = {static_cast<cuuint64_t>(width) * 2};
  cuuint32_t box[2] = {64, static_cast<cuuint32_t>(box_rows)};
  cuuint32_t es[2] = {1, 1};
  return reinterpret_cast<EncodeTiledFn>(fn)(m, CU_TENSOR_MAP_DATA_TYPE_BFLOAT16, 2, const_cast<void*>(base), dims,
                                             strides, box, es, CU_TENSOR_MAP_INTERLEAVE_NONE,
                                             CU_TENSOR_MAP_SWIZZLE_128B, CU_TENSOR_MAP_L2_PROMOTION_L2_256B,
                                             CU_TENSOR_MAP_FLOAT_OOB_FILL_NONE) == CUDA_SUCCESS;
}
// bf16 [E, rows, width] -> 3D map with box {64, box_rows, 1}
inline bool map_3d(void* fn, CUtensorMap* m, const void* base, int64_t E, int64_t rows, int64_t width,
                   int box_rows) {
  cuuint64_t dims[3] = {static_cast<cuuint64_t>(width), static_cast<cuuint64_t>(rows), static_cast<cuuint64_t>(E)};
  cuuint64_t strides[2] = {static_cast<cuuint64_t>(width) * 2, static_cast<cuuint64_t>(width) * rows * 2};
  cuuint32_t box[3] = {64, static_cast<cuuint32_t>(box_rows), 1};
  cuuint32_t es[3] = {1, 1, 1};
  return reinterpret_cast<EncodeTiledFn>(fn)(m, CU_TENSOR_MAP_DATA_TYPE_BFLOAT16, 3, const_cast<void*>(base), dims,
                                             strides, box, es, CU_TENSOR_MAP_INTERLEAVE_NONE,
                                             CU_TENSOR_MAP_SWIZZLE_128B, CU_TENSOR_MAP_L2_PROMOTION_L2_256B,
                                             CU_TENSOR_MAP_FLOAT_OOB_FILL_NONE) == CUDA_SUCCESS;
}

// MN-major operands, `chunks` 64-column chunks of 64 K rows in one box that lands in shared memory chunk by chunk.  The
// chunk is a dimension of the map (64 columns apart), so the width has to be a multiple of 64, or at most 64 with one
// chunk in use (columns beyond the width read as zeros).
inline bool map_chunks(void* fn, CUtensorMap* m, const void* base, int64_t E, int64_t rows, int64_t width, int chunks,
                       int rank) {
  cuuint64_t dims[4] = {static_cast<cuuint64_t>(width < 64 ? width : 64), static_cast<cuuint64_t>(rows),
                        static_cast<cuuint64_t>((width + 63) / 64), static_cast<cuuint64_t>(E)};
  cuuint64_t strides[3] = {static_cast<cuuint64_t>(width) * 2, 128, static_cast<cuuint64_t>(width) * rows * 2};
  cuuint32_t box[4] = {64, 64, static_cast<cuuint32_t>(chunks), 1};
  cuuint32_t es[4] = {1, 1, 1, 1};
  return reinterpret_cast<EncodeTiledFn>(fn)(m, CU_TENSOR_MAP_DATA_TYPE_BFLOAT16, rank, const_cast<void*>(base), dims,
                                             strides, box, es, CU_TENSOR_MAP_INTERLEAVE_NONE,
                                             CU_TENSOR_MAP_SWIZZLE_128B, CU_TENSOR_MAP_L2_PROMOTION_L2_256B,
                                             CU_TENSOR_MAP_FLOAT_OOB_FILL_NONE) == CUDA_SUCCESS;
}
// bf16 weights [E, rows, width]: coordinates (0, row, chunk, expert)
inline bool map_mn(void* fn, CUtensorMap* m, const void* base, int64_t E, int64_t rows, int64_t width, int chunks) {
  return map_chunks(fn, m, base, E, rows, width, chunks, 4);
}
// bf16 rows [rows, width]: coordinates (0, row, chunk)
inline bool map_mn_rows(void* fn, CUtensorMap* m, const void* base, int64_t rows, int64_t width, int chunks) {
  return map_chunks(fn, m, base, 1, rows, width, chunks, 3);
}

}  // namespace moe
