// Tensor maps of bf16 planes (K-major rows) for TMA.
#pragma once
#include <cuda.h>

#include <mutex>

#include "common.cuh"

namespace chase {

typedef CUresult (*EncodeFn)(CUtensorMap*, CUtensorMapDataType, cuuint32_t, void*, const cuuint64_t*, const cuuint64_t*,
                             const cuuint32_t*, const cuuint32_t*, CUtensorMapInterleave, CUtensorMapSwizzle,
                             CUtensorMapL2promotion, CUtensorMapFloatOOBfill);

inline EncodeFn encode_fn() {
  static EncodeFn fn = nullptr;
  static std::once_flag once;
  std::call_once(once, []() {
    void* p = nullptr;
    cudaDriverEntryPointQueryResult q;
    if (cudaGetDriverEntryPoint("cuTensorMapEncodeTiled", &p, cudaEnableDefault, &q) == cudaSuccess &&
        q == cudaDriverEntryPointSuccess)
      fn = (EncodeFn)p;
  });
  return fn;
}

// `planes` planes of `rows` rows of K values (row pitch Kpad); box: box_k x box_rows x box_planes, landing
// plane-major in shared memory; values outside the extents read as zero
inline CUtensorMap make_tmap_bf16(const void* base, int64_t K, int64_t Kpad, int64_t rows, int planes, int box_k,
                                  int box_rows, int box_planes, CUtensorMapSwizzle swizzle) {
  CUtensorMap m;
  cuuint64_t dims[3] = {(cuuint64_t)K, (cuuint64_t)rows, (cuuint64_t)planes};
  cuuint64_t strides[2] = {(cuuint64_t)(Kpad * 2), (cuuint64_t)(Kpad * 2 * rows)};
  cuuint32_t box[3] = {(cuuint32_t)box_k, (cuuint32_t)box_rows, (cuuint32_t)box_planes};
  cuuint32_t es[3] = {1, 1, 1};
  EncodeFn fn = encode_fn();
  CHASE_REQUIRE(fn != nullptr, 9, "cuTensorMapEncodeTiled unavailable");
  CUresult r = fn(&m, CU_TENSOR_MAP_DATA_TYPE_BFLOAT16, 3, const_cast<void*>(base), dims, strides, box, es,
                  CU_TENSOR_MAP_INTERLEAVE_NONE, swizzle, CU_TENSOR_MAP_L2_PROMOTION_L2_256B,
                  CU_TENSOR_MAP_FLOAT_OOB_FILL_NONE);
  CHASE_REQUIRE(r == CUDA_SUCCESS, 6, "cuTensorMapEncodeTiled failed");
  return m;
}

}  // namespace chase
