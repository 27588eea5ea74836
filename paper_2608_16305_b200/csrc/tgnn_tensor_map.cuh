// The driver's tensor-map encoder for the tensor-core kernels.
#pragma once
#include <cuda.h>
#include <cuda_runtime.h>

namespace tgnn {

typedef CUresult (*TensorMapEncodeFn)(CUtensorMap*, CUtensorMapDataType, cuuint32_t, void*, const cuuint64_t*,
                                      const cuuint64_t*, const cuuint32_t*, const cuuint32_t*, CUtensorMapInterleave,
                                      CUtensorMapSwizzle, CUtensorMapL2promotion, CUtensorMapFloatOOBfill);

// Looked up once through the runtime (no link against the driver library), by whichever thread comes first, while the others
// wait for it; nullptr if it is unavailable.
inline TensorMapEncodeFn tensor_map_encoder() {
  static const TensorMapEncodeFn enc = [] {
    void* fn = nullptr;
    cudaDriverEntryPointQueryResult q;
    const bool ok = cudaGetDriverEntryPoint("cuTensorMapEncodeTiled", &fn, cudaEnableDefault, &q) == cudaSuccess &&
                    q == cudaDriverEntryPointSuccess;
    (void)cudaGetLastError();
    return ok ? reinterpret_cast<TensorMapEncodeFn>(fn) : nullptr;
  }();
  return enc;
}

}  // namespace tgnn
