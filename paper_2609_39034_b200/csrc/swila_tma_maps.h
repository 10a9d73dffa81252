// Host side of the tensor copies (TMA): one tiled tensor map.
#pragma once

#include <cuda.h>  // CUtensorMap and its enums (types only; the encoder is fetched through the runtime)
#include <cuda_runtime.h>

namespace swila {

// cuTensorMapEncodeTiled, fetched through the runtime so that the library does not link against the driver.
typedef CUresult (*TmaEncodeTiledFn)(CUtensorMap *, CUtensorMapDataType, cuuint32_t, void *, const cuuint64_t *,
                                     const cuuint64_t *, const cuuint32_t *, const cuuint32_t *, CUtensorMapInterleave,
                                     CUtensorMapSwizzle, CUtensorMapL2promotion, CUtensorMapFloatOOBfill);
inline TmaEncodeTiledFn tma_encode_fn() {
  static TmaEncodeTiledFn fn = [] {
    void *sym = nullptr;
    cudaDriverEntryPointQueryResult res;
    if (cudaGetDriverEntryPoint("cuTensorMapEncodeTiled", &sym, cudaEnableDefault, &res) != cudaSuccess ||
        res != cudaDriverEntryPointSuccess)
      sym = nullptr;
    return (TmaEncodeTiledFn)sym;
  }();
  return fn;
}

// One tensor map: `rank` dimensions (innermost first) of sizes `dims` with byte strides `strides` (for dimensions
// 1 .. rank-1) and a copy box of `box` elements; out-of-range elements read as zero.
inline bool tma_encode(CUtensorMap *map, const void *base, int rank, const cuuint64_t *dims, const cuuint64_t *strides,
                       const cuuint32_t *box, CUtensorMapSwizzle swizzle = CU_TENSOR_MAP_SWIZZLE_NONE,
                       CUtensorMapDataType type = CU_TENSOR_MAP_DATA_TYPE_BFLOAT16) {
  TmaEncodeTiledFn fn = tma_encode_fn();
  if (!fn) return false;
  const cuuint32_t ones[4] = {1, 1, 1, 1};
  return fn(map, type, (cuuint32_t)rank, const_cast<void *>(base), dims, strides, box, ones, CU_TENSOR_MAP_INTERLEAVE_NONE, swizzle,
            CU_TENSOR_MAP_L2_PROMOTION_L2_128B, CU_TENSOR_MAP_FLOAT_OOB_FILL_NONE) == CUDA_SUCCESS;
}

}  // namespace swila
