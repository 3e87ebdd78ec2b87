// Host-side TMA tensor-map encoding (cuTensorMapEncodeTiled through the
// runtime's driver entry point, so the library needs no -lcuda).
#include <cuda.h>
#include <cudaTypedefs.h>
#include <cuda_runtime.h>

#include "tmap.cuh"

namespace xs {
namespace {

// The driver's encoder, looked up once (a function-local static is
// initialised exactly once even when host threads race on the first call).
PFN_cuTensorMapEncodeTiled_v12000 encode_fn() {
  static const PFN_cuTensorMapEncodeTiled_v12000 fn = []() -> PFN_cuTensorMapEncodeTiled_v12000 {
    void *ptr = nullptr;
    cudaDriverEntryPointQueryResult q;
    if (cudaGetDriverEntryPointByVersion("cuTensorMapEncodeTiled", &ptr, 12000, cudaEnableDefault,
                                         &q) == cudaSuccess &&
        q == cudaDriverEntryPointSuccess)
      return reinterpret_cast<PFN_cuTensorMapEncodeTiled_v12000>(ptr);
    return nullptr;
  }();
  return fn;
}

}  // namespace

bool encode_tmap(CUtensorMap *m, CUtensorMapDataType dtype, const void *base, int rank,
                 const uint64_t *dims, const uint64_t *strides, const uint32_t *box,
                 CUtensorMapSwizzle swizzle) {
  auto fn = encode_fn();
  if (fn == nullptr || rank < 1 || rank > 5) return false;
  cuuint64_t d[5], st[5];
  cuuint32_t bx[5], one[5];
  for (int i = 0; i < rank; ++i) {
    d[i] = dims[i];
    st[i] = i + 1 < rank ? strides[i] : 0;
    bx[i] = box[i];
    one[i] = 1;
  }
  return fn(m, dtype, static_cast<cuuint32_t>(rank), const_cast<void *>(base), d, st, bx, one,
            CU_TENSOR_MAP_INTERLEAVE_NONE, swizzle, CU_TENSOR_MAP_L2_PROMOTION_L2_256B,
            CU_TENSOR_MAP_FLOAT_OOB_FILL_NONE) == CUDA_SUCCESS;
}

bool encode_tmap_2d(CUtensorMap *m, CUtensorMapDataType dtype, uint32_t elem_bytes,
                    const void *base, uint64_t inner, uint64_t outer, uint32_t box_inner,
                    uint32_t box_outer, CUtensorMapSwizzle swizzle) {
  const uint64_t dims[2] = {inner, outer}, strides[1] = {inner * elem_bytes};
  const uint32_t box[2] = {box_inner, box_outer};
  return encode_tmap(m, dtype, base, 2, dims, strides, box, swizzle);
}

}  // namespace xs
