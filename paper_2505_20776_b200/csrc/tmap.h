// Host side: encoding of the TMA tensor maps the attention kernels use.
#ifndef SPECEXT_TMAP_H_
#define SPECEXT_TMAP_H_

#include <atomic>

#include <cuda.h>
#include <cuda_runtime.h>

typedef CUresult (*SpxEncodeTiledFn)(CUtensorMap*, CUtensorMapDataType, cuuint32_t, void*, const cuuint64_t*,
                                     const cuuint64_t*, const cuuint32_t*, const cuuint32_t*, CUtensorMapInterleave,
                                     CUtensorMapSwizzle, CUtensorMapL2promotion, CUtensorMapFloatOOBfill);

// The driver's encoder, looked up until it is found (several threads may do so at once); null when there is no driver.
inline SpxEncodeTiledFn spx_encode_fn() {
  static std::atomic<SpxEncodeTiledFn> known{nullptr};
  SpxEncodeTiledFn fn = known.load();
  if (fn) return fn;
  void* ptr = nullptr;
  cudaDriverEntryPointQueryResult qres;
  if (cudaGetDriverEntryPoint("cuTensorMapEncodeTiled", &ptr, cudaEnableDefault, &qres) != cudaSuccess ||
      qres != cudaDriverEntryPointSuccess)
    return nullptr;
  fn = reinterpret_cast<SpxEncodeTiledFn>(ptr);
  known.store(fn);
  return fn;
}

// bf16 tensor [n2][n1][n0] with element strides (s2, s1, 1); box = 64 x b1 x b2, 128-byte swizzle, out-of-range
// elements read as zero.
inline bool spx_encode_map(CUtensorMap* m, const void* ptr, int n0, long long n1, long long s1, long long n2,
                           long long s2, int b1, int b2) {
  const SpxEncodeTiledFn fn = spx_encode_fn();
  if (!fn) return false;
  const cuuint64_t dims[3] = {(cuuint64_t)n0, (cuuint64_t)n1, (cuuint64_t)n2};
  const cuuint64_t strides[2] = {(cuuint64_t)s1 * 2, (cuuint64_t)s2 * 2};
  const cuuint32_t box[3] = {64, (cuuint32_t)b1, (cuuint32_t)b2};
  const cuuint32_t es[3] = {1, 1, 1};
  return fn(m, CU_TENSOR_MAP_DATA_TYPE_BFLOAT16, 3, const_cast<void*>(ptr), dims, strides, box, es,
            CU_TENSOR_MAP_INTERLEAVE_NONE, CU_TENSOR_MAP_SWIZZLE_128B, CU_TENSOR_MAP_L2_PROMOTION_L2_256B,
            CU_TENSOR_MAP_FLOAT_OOB_FILL_NONE) == CUDA_SUCCESS;
}

#endif  // SPECEXT_TMAP_H_
