// Host side of the TMA tile loads: the tensor-map encoder (a driver entry point
// fetched through the runtime, so that the library does not link the driver
// library) and the one tensor shape every tensor-core kernel of this library
// reads.
#pragma once
#include <cuda.h>
#include <cuda_runtime.h>

namespace spiffy {
namespace {

typedef CUresult (*EncodeTiledFn)(CUtensorMap*, CUtensorMapDataType, cuuint32_t, void*,
                                  const cuuint64_t*, const cuuint64_t*, const cuuint32_t*,
                                  const cuuint32_t*, CUtensorMapInterleave, CUtensorMapSwizzle,
                                  CUtensorMapL2promotion, CUtensorMapFloatOOBfill);

EncodeTiledFn encode_fn() {
  static EncodeTiledFn fn = [] {
    void* f = nullptr;
    cudaDriverEntryPointQueryResult q;
    if (cudaGetDriverEntryPoint("cuTensorMapEncodeTiled", &f, cudaEnableDefault, &q) != cudaSuccess)
      f = nullptr;
    return reinterpret_cast<EncodeTiledFn>(f);
  }();
  return fn;
}

// Tensor [outer][rows][heads][inner] of bf16, inner = 64 or 128 (equally: a [rows][heads * 128]
// matrix), seen as a 4-D TMA tensor with a 64-element half of a head row innermost (the whole of
// it when inner = 64); box = 64 x box_heads x box_rows x 1.
// `outer_stride_rows`: rows between consecutive outer slices (0 = densely packed, i.e. `rows`);
// larger when the tensor is a window of `rows` rows into a longer one.
bool make_map(CUtensorMap* m, const void* base, int heads, int64_t rows, int outer, int box_heads,
              int box_rows, int64_t outer_stride_rows = 0, int inner = 128) {
  EncodeTiledFn enc = encode_fn();
  if (!enc) return false;
  if (outer_stride_rows <= 0) outer_stride_rows = rows;
  const cuuint64_t dims[4] = {(cuuint64_t)inner, (cuuint64_t)heads, (cuuint64_t)rows, (cuuint64_t)outer};
  const cuuint64_t strides[3] = {(cuuint64_t)inner * 2, (cuuint64_t)heads * inner * 2,
                                 (cuuint64_t)outer_stride_rows * heads * inner * 2};
  const cuuint32_t box[4] = {64, (cuuint32_t)box_heads, (cuuint32_t)box_rows, 1};
  const cuuint32_t es[4] = {1, 1, 1, 1};
  return enc(m, CU_TENSOR_MAP_DATA_TYPE_BFLOAT16, 4, const_cast<void*>(base), dims, strides, box,
             es, CU_TENSOR_MAP_INTERLEAVE_NONE, CU_TENSOR_MAP_SWIZZLE_128B,
             CU_TENSOR_MAP_L2_PROMOTION_L2_256B, CU_TENSOR_MAP_FLOAT_OOB_FILL_NONE) == CUDA_SUCCESS;
}

// Tensor [outer][rows][heads][64 * halves] of bf16 as a 5-D TMA tensor {64 elements, head, row, half,
// outer}; box = 64 x box_heads x box_rows x box_halves x 1.  The half of a head row comes behind the
// rows, so that one instruction brings a tile's halves as they lie in shared memory, one 64-element
// swizzled block behind the other (`block`: or 32-element ones): an instruction takes its warp 85 to 105
// cycles to issue, some 200 among others, whatever its size.
bool make_tile_map(CUtensorMap* m, const void* base, int heads, int64_t rows, int outer, int box_heads, int box_rows,
                   int box_halves, int64_t outer_stride_rows, int halves, int block = 64) {
  EncodeTiledFn enc = encode_fn();
  if (!enc) return false;
  if (outer_stride_rows <= 0) outer_stride_rows = rows;
  const cuuint64_t row_bytes = (cuuint64_t)halves * block * 2;
  const cuuint64_t dims[5] = {(cuuint64_t)block, (cuuint64_t)heads, (cuuint64_t)rows, (cuuint64_t)halves, (cuuint64_t)outer};
  const cuuint64_t strides[4] = {row_bytes, heads * row_bytes, (cuuint64_t)block * 2, (cuuint64_t)outer_stride_rows * heads * row_bytes};
  const cuuint32_t box[5] = {(cuuint32_t)block, (cuuint32_t)box_heads, (cuuint32_t)box_rows, (cuuint32_t)box_halves, 1};
  const cuuint32_t es[5] = {1, 1, 1, 1, 1};
  return enc(m, CU_TENSOR_MAP_DATA_TYPE_BFLOAT16, 5, const_cast<void*>(base), dims, strides, box, es,
             CU_TENSOR_MAP_INTERLEAVE_NONE, block == 64 ? CU_TENSOR_MAP_SWIZZLE_128B : CU_TENSOR_MAP_SWIZZLE_64B, CU_TENSOR_MAP_L2_PROMOTION_L2_256B,
             CU_TENSOR_MAP_FLOAT_OOB_FILL_NONE) == CUDA_SUCCESS;
}

}  // namespace
}  // namespace spiffy
