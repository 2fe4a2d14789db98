// What the host side asks the driver itself: tensor-map (TMA descriptor) encoding, and how far an address's allocation
// reaches.  The entry points are resolved at run time so the library carries no link-time dependency on libcuda.
#include <cudaTypedefs.h>

#include "runtime.h"

namespace lv {

static bool resolve(const char* name, void** fn) {
  void* p = nullptr;
  cudaDriverEntryPointQueryResult q;
  cudaError_t e = cudaGetDriverEntryPoint(name, &p, cudaEnableDefault, &q);
  if (e != cudaSuccess || q != cudaDriverEntryPointSuccess || p == nullptr) {
    (void)cudaGetLastError();
    return false;
  }
  *fn = p;
  return true;
}

bool resolve_encode_tiled(void** fn) { return resolve("cuTensorMapEncodeTiled", fn); }

bool allocation_of(const void* device_ptr, const uint8_t** begin, size_t* bytes) {
  static std::atomic<void*> resolved{nullptr};
  void* fn = resolved.load(std::memory_order_acquire);
  if (fn == nullptr) {
    if (!resolve("cuPointerGetAttribute", &fn)) return false;
    resolved.store(fn, std::memory_order_release);
  }
  auto attribute = reinterpret_cast<PFN_cuPointerGetAttribute_v4000>(fn);
  const CUdeviceptr p = reinterpret_cast<CUdeviceptr>(device_ptr);
  CUdeviceptr start = 0;
  if (attribute(&start, CU_POINTER_ATTRIBUTE_RANGE_START_ADDR, p) != CUDA_SUCCESS ||
      attribute(bytes, CU_POINTER_ATTRIBUTE_RANGE_SIZE, p) != CUDA_SUCCESS)
    return false;
  *begin = reinterpret_cast<const uint8_t*>(start);
  return true;
}

bool make_tmap_bf16_2d(void* encode_fn, CUtensorMap* out, const void* base, uint64_t inner, uint64_t outer,
                       uint64_t pitch_elems, uint32_t box_inner, uint32_t box_outer, bool box_alone) {
  auto encode = reinterpret_cast<PFN_cuTensorMapEncodeTiled_v12000>(encode_fn);
  const cuuint64_t dims[2] = {inner, outer};
  const cuuint64_t strides[1] = {pitch_elems * 2};  // bytes, dimension 1
  const cuuint32_t box[2] = {box_inner, box_outer};
  const cuuint32_t elem_strides[2] = {1, 1};
  const CUresult r = encode(out, CU_TENSOR_MAP_DATA_TYPE_BFLOAT16, 2, const_cast<void*>(base), dims, strides, box,
                            elem_strides, CU_TENSOR_MAP_INTERLEAVE_NONE, CU_TENSOR_MAP_SWIZZLE_128B,
                            box_alone ? CU_TENSOR_MAP_L2_PROMOTION_L2_128B : CU_TENSOR_MAP_L2_PROMOTION_L2_256B,
                            CU_TENSOR_MAP_FLOAT_OOB_FILL_NONE);
  return r == CUDA_SUCCESS;
}

// 2-D tensor of bytes [outer, inner] with row pitch `pitch_bytes`; box [box_outer, box_inner bytes];
// 64-byte swizzle for boxes whose rows are 64 bytes, 128-byte swizzle otherwise; zero fill outside.
bool make_tmap_u8_2d(void* encode_fn, CUtensorMap* out, const void* base, uint64_t inner, uint64_t outer,
                     uint64_t pitch_bytes, uint32_t box_inner, uint32_t box_outer) {
  auto encode = reinterpret_cast<PFN_cuTensorMapEncodeTiled_v12000>(encode_fn);
  const cuuint64_t dims[2] = {inner, outer};
  const cuuint64_t strides[1] = {pitch_bytes};
  const cuuint32_t box[2] = {box_inner, box_outer};
  const cuuint32_t elem_strides[2] = {1, 1};
  const CUtensorMapSwizzle swizzle = box_inner == 64 ? CU_TENSOR_MAP_SWIZZLE_64B : CU_TENSOR_MAP_SWIZZLE_128B;
  CUresult r = encode(out, CU_TENSOR_MAP_DATA_TYPE_UINT8, 2, const_cast<void*>(base), dims, strides, box, elem_strides,
                      CU_TENSOR_MAP_INTERLEAVE_NONE, swizzle, CU_TENSOR_MAP_L2_PROMOTION_L2_256B,
                      CU_TENSOR_MAP_FLOAT_OOB_FILL_NONE);
  return r == CUDA_SUCCESS;
}

}  // namespace lv
