// Tensor maps of the (slabs x n x d) tensors for the TMA copies of the tensor-core kernels.
#pragma once
#include <cuda.h>
#include <cuda_runtime.h>

#include "common.cuh"

namespace wersa {

typedef CUresult (*EncodeTiledFn)(CUtensorMap*, CUtensorMapDataType, cuuint32_t, void*, const cuuint64_t*,
                                  const cuuint64_t*, const cuuint32_t*, const cuuint32_t*, CUtensorMapInterleave,
                                  CUtensorMapSwizzle, CUtensorMapL2promotion, CUtensorMapFloatOOBfill);

inline EncodeTiledFn encode_fn() {
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

inline cudaError_t make_map(const void* base, CUtensorMapDataType type, int elem, int slabs, int n, int d, int box_cols,
                            int box_rows, CUtensorMap* out) {
  EncodeTiledFn fn = encode_fn();
  if (fn == nullptr) return cudaErrorNotSupported;
  const cuuint64_t dims[3] = {(cuuint64_t)d, (cuuint64_t)n, (cuuint64_t)slabs};
  const cuuint64_t strides[2] = {(cuuint64_t)d * elem, (cuuint64_t)n * d * elem};
  const cuuint32_t box[3] = {(cuuint32_t)box_cols, (cuuint32_t)box_rows, 1};
  const cuuint32_t estr[3] = {1, 1, 1};
  const CUresult r = fn(out, type, 3, const_cast<void*>(base), dims, strides, box, estr, CU_TENSOR_MAP_INTERLEAVE_NONE,
                        CU_TENSOR_MAP_SWIZZLE_128B, CU_TENSOR_MAP_L2_PROMOTION_L2_128B, CU_TENSOR_MAP_FLOAT_OOB_FILL_NONE);
  return r == CUDA_SUCCESS ? cudaSuccess : cudaErrorInvalidValue;
}

// (slabs x n x d) bf16 row-major tensor, boxes of 128 rows x 64 columns of one slab, 128-byte swizzle.  Rows are d values
// (a multiple of 8: row pitches are multiples of 16 bytes) and the box is always 64 columns wide, so that a narrower tensor
// arrives zero-filled up to column 63 and is stored clipped; rows past the end of a slab read as zeros and are not written.
inline cudaError_t make_tile_map(const void* base, int slabs, int n, CUtensorMap* out, int d = kD) {
  return make_map(base, CU_TENSOR_MAP_DATA_TYPE_BFLOAT16, 2, slabs, n, d, kD, 128, out);
}

// Store map of a result tensor: fp32 in boxes of 128 rows x 32 columns (128 bytes, the widest a 128-byte swizzle takes),
// bf16 in boxes of 128 rows x 64 columns; rows past n are not written.
inline cudaError_t make_out_map(void* base, int slabs, int n, int d, bool bf16, CUtensorMap* out) {
  if (bf16) return make_tile_map(base, slabs, n, out, d);
  return make_map(base, CU_TENSOR_MAP_DATA_TYPE_FLOAT32, 4, slabs, n, d, 32, 128, out);
}

}  // namespace wersa
