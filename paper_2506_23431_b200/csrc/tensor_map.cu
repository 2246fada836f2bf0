// Tensor maps for the TMA kernels: the driver's encoder behind one call.
#include "pd_internal.h"

namespace pd {

// Row-major tiles of `rank` dimensions (innermost first), 128-byte swizzle, reads beyond the tensor filled with zeros.
// gdim, box: `rank` extents in elements; gstride: rank - 1 strides in bytes.  *driver_code gets the CUresult when the encode itself
// fails.  The encoder's address is looked up once per process: a look-up costs more than an encode, and the stand-alone
// operators encode their maps on every call.
cudaError_t encode_tensor_map(CUtensorMap *out, CUtensorMapDataType type, int rank, const void *base, const uint64_t *gdim,
                              const uint64_t *gstride, const uint32_t *box, int *driver_code) {
  typedef CUresult (*EncodeFn)(CUtensorMap *, CUtensorMapDataType, cuuint32_t, void *, const cuuint64_t *, const cuuint64_t *,
                               const cuuint32_t *, const cuuint32_t *, CUtensorMapInterleave, CUtensorMapSwizzle,
                               CUtensorMapL2promotion, CUtensorMapFloatOOBfill);
  struct Entry { EncodeFn fn; cudaError_t err; };
  static const Entry entry = [] {
    void *fn = nullptr;
    cudaDriverEntryPointQueryResult qres;
    cudaError_t e = cudaGetDriverEntryPoint("cuTensorMapEncodeTiled", &fn, cudaEnableDefault, &qres);
    if (e == cudaSuccess && (fn == nullptr || qres != cudaDriverEntryPointSuccess)) e = cudaErrorNotSupported;
    return Entry{(EncodeFn)fn, e};
  }();
  if (driver_code) *driver_code = 0;
  if (entry.err != cudaSuccess) return entry.err;
  cuuint64_t gd[3], gs[2];
  const cuuint32_t estr[3] = {1u, 1u, 1u};
  for (int i = 0; i < rank; ++i) gd[i] = gdim[i];
  for (int i = 0; i + 1 < rank; ++i) gs[i] = gstride[i];
  CUresult r = entry.fn(out, type, (cuuint32_t)rank, const_cast<void *>(base), gd, gs, box, estr, CU_TENSOR_MAP_INTERLEAVE_NONE,
                        CU_TENSOR_MAP_SWIZZLE_128B, CU_TENSOR_MAP_L2_PROMOTION_L2_256B, CU_TENSOR_MAP_FLOAT_OOB_FILL_NONE);
  if (r != CUDA_SUCCESS) { if (driver_code) *driver_code = (int)r; return cudaErrorInvalidValue; }
  return cudaSuccess;
}

}  // namespace pd
