// Host-side helpers shared by the attention kernels' entry points.
#pragma once
#include <cuda.h>

#include "common.cuh"
#include "host.h"

namespace us {

constexpr int kAttnD = 64;                 // head width
constexpr int kAttnMaxKeys = 512;

// 4-d map (column, row, inner problem index, outer problem index) over elements of es bytes (2, or 1 for FP8); box of
// box_bytes (128 or 64, the swizzle of that width) x box_rows rows of one problem; columns of a box beyond the matrix read as zeros.
inline bool attn_tmap(CUtensorMap* tm, const us_mat* m, const int64_t* stride, const int64_t* count, int box_rows, int es = 2,
                      int box_bytes = 128) {
  host::EncodeTiledFn fn = host::encode_tiled_fn();
  if (!fn) return false;
  cuuint64_t dims[4] = {(cuuint64_t)m->cols, (cuuint64_t)m->rows, (cuuint64_t)count[1], (cuuint64_t)count[0]};
  // a dimension of extent 1 still needs a valid (multiple of 16 bytes) stride
  const cuuint64_t s1 = count[1] > 1 ? (cuuint64_t)stride[1] * es : 16, s0 = count[0] > 1 ? (cuuint64_t)stride[0] * es : 16;
  cuuint64_t strides[3] = {(cuuint64_t)m->ld * es, s1, s0};
  cuuint32_t box[4] = {(cuuint32_t)(box_bytes / es), (cuuint32_t)box_rows, 1, 1};
  cuuint32_t estr[4] = {1, 1, 1, 1};
  return fn(tm, es == 1 ? CU_TENSOR_MAP_DATA_TYPE_UINT8 : CU_TENSOR_MAP_DATA_TYPE_UINT16, 4, m->ptr, dims, strides, box, estr, CU_TENSOR_MAP_INTERLEAVE_NONE,
            box_bytes == 64 ? CU_TENSOR_MAP_SWIZZLE_64B : CU_TENSOR_MAP_SWIZZLE_128B, CU_TENSOR_MAP_L2_PROMOTION_L2_128B,
            CU_TENSOR_MAP_FLOAT_OOB_FILL_NONE) == CUDA_SUCCESS;
}

inline bool attn_aligned(const us_mat* m, const int64_t* stride, const int64_t* count, int es) {
  if (reinterpret_cast<uintptr_t>(m->ptr) % 16 || (m->ld * es) % 16) return false;
  for (int i = 0; i < 2; ++i)
    if (count[i] > 1 && (stride[i] * es) % 16) return false;
  return true;
}

}  // namespace us
