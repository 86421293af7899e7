// Host-side tensor maps (cuTensorMapEncodeTiled through the runtime's driver
// entry point; the library does not link libcuda).
#pragma once
#include <cuda.h>
#include <cudaTypedefs.h>
#include <cuda_bf16.h>
#include <cuda_runtime.h>

#include <mutex>

namespace rc {

inline PFN_cuTensorMapEncodeTiled_v12000 tma_encode_fn() {
  static PFN_cuTensorMapEncodeTiled_v12000 fn = nullptr;
  static std::once_flag once;
  std::call_once(once, [] {
    void* p = nullptr;
    cudaDriverEntryPointQueryResult q;
    if (cudaGetDriverEntryPointByVersion("cuTensorMapEncodeTiled", &p, 12000, cudaEnableDefault,
                                         &q) == cudaSuccess &&
        q == cudaDriverEntryPointSuccess)
      fn = reinterpret_cast<PFN_cuTensorMapEncodeTiled_v12000>(p);
  });
  return fn;
}

// bf16 tensor of `rank` dimensions (innermost first), strides in elements of
// dimensions 1 .. rank - 1; boxes with a 64-wide innermost extent use the
// 128-byte swizzle, 16-wide ones the 32-byte swizzle; reads outside the
// tensor give zero.
inline cudaError_t tma_map(const __nv_bfloat16* p, int rank, const cuuint64_t* dims,
                           const cuuint64_t* strides, const cuuint32_t* box, CUtensorMap* out) {
  auto fn = tma_encode_fn();
  if (!fn) return cudaErrorNotSupported;
  cuuint64_t st[4] = {};
  cuuint32_t es[5] = {1, 1, 1, 1, 1};
  for (int i = 0; i + 1 < rank; ++i) st[i] = strides[i] * sizeof(__nv_bfloat16);
  const CUresult r =
      fn(out, CU_TENSOR_MAP_DATA_TYPE_BFLOAT16, cuuint32_t(rank),
         const_cast<__nv_bfloat16*>(p), dims, st, box, es, CU_TENSOR_MAP_INTERLEAVE_NONE,
         box[0] == 64 ? CU_TENSOR_MAP_SWIZZLE_128B : CU_TENSOR_MAP_SWIZZLE_32B,
         CU_TENSOR_MAP_L2_PROMOTION_L2_128B, CU_TENSOR_MAP_FLOAT_OOB_FILL_NONE);
  return r == CUDA_SUCCESS ? cudaSuccess : cudaErrorInvalidValue;
}

}  // namespace rc
