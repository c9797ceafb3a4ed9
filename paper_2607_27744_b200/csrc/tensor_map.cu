// Host helpers on the driver API: TMA tensor maps with cuTensorMapEncodeTiled, the id of the current context with
// cuCtxGetId, both resolved at run time through cudaGetDriverEntryPoint so that librocs.so has no link-time dependency
// on libcuda.
#include "rocs_internal.h"
#include "sm100_ptx.cuh"

namespace rocs {
namespace {

using EncodeTiledFn = CUresult (*)(CUtensorMap*, CUtensorMapDataType, cuuint32_t, void*, const cuuint64_t*,
                                   const cuuint64_t*, const cuuint32_t*, const cuuint32_t*, CUtensorMapInterleave,
                                   CUtensorMapSwizzle, CUtensorMapL2promotion, CUtensorMapFloatOOBfill);

using GetContextIdFn = CUresult (*)(CUcontext, unsigned long long*);

template <typename F>
F driver_function(const char* name) {
  void* p = nullptr;
  cudaDriverEntryPointQueryResult q;
  if (cudaGetDriverEntryPoint(name, &p, cudaEnableDefault, &q) != cudaSuccess || q != cudaDriverEntryPointSuccess) return nullptr;
  return reinterpret_cast<F>(p);
}

EncodeTiledFn encode_tiled() {
  static const EncodeTiledFn fn = driver_function<EncodeTiledFn>("cuTensorMapEncodeTiled");
  return fn;
}

}  // namespace

unsigned long long context_id() {
  static const GetContextIdFn fn = driver_function<GetContextIdFn>("cuCtxGetId");
  unsigned long long id = 0;
  return fn != nullptr && fn(nullptr, &id) == CUDA_SUCCESS ? id : 0;
}

bool make_tensor_map_2d(CUtensorMap* map, const void* base, CUtensorMapDataType dtype, uint32_t elem_bytes,
                        uint64_t rows, uint64_t cols, uint64_t ld, uint32_t box_rows, uint32_t box_cols,
                        bool swizzle128, bool swizzle64) {
  EncodeTiledFn fn = encode_tiled();
  if (!fn || rows == 0 || cols == 0) return false;
  const cuuint64_t dims[2] = {cols, rows};
  const cuuint64_t strides[1] = {ld * elem_bytes};  // byte stride of dimension 1
  const cuuint32_t box[2] = {box_cols, box_rows};
  const cuuint32_t elem_strides[2] = {1, 1};
  return fn(map, dtype, 2, const_cast<void*>(base), dims, strides, box, elem_strides, CU_TENSOR_MAP_INTERLEAVE_NONE,
            swizzle64 ? CU_TENSOR_MAP_SWIZZLE_64B : swizzle128 ? CU_TENSOR_MAP_SWIZZLE_128B : CU_TENSOR_MAP_SWIZZLE_NONE,
            CU_TENSOR_MAP_L2_PROMOTION_L2_256B,
            CU_TENSOR_MAP_FLOAT_OOB_FILL_NONE) == CUDA_SUCCESS;
}

bool make_tensor_map_3d(CUtensorMap* map, const void* base, uint64_t cols, uint64_t rows, uint64_t n, uint32_t box_cols,
                        uint32_t box_rows, uint32_t box_n) {
  EncodeTiledFn fn = encode_tiled();
  if (!fn || n == 0 || rows == 0 || cols == 0) return false;
  const cuuint64_t dims[3] = {cols, rows, n};
  const cuuint64_t strides[2] = {cols * 2, rows * cols * 2};
  const cuuint32_t box[3] = {box_cols, box_rows, box_n};
  const cuuint32_t elem_strides[3] = {1, 1, 1};
  return fn(map, CU_TENSOR_MAP_DATA_TYPE_BFLOAT16, 3, const_cast<void*>(base), dims, strides, box, elem_strides,
            CU_TENSOR_MAP_INTERLEAVE_NONE, CU_TENSOR_MAP_SWIZZLE_128B, CU_TENSOR_MAP_L2_PROMOTION_L2_256B,
            CU_TENSOR_MAP_FLOAT_OOB_FILL_NONE) == CUDA_SUCCESS;
}

}  // namespace rocs
