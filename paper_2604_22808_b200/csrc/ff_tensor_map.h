// The driver's tensor-map calls, looked up once, and the one kind of map the kernels use: tiled, densely packed elements,
// zeros outside the tensor.
#pragma once
#include <cuda.h>
#include <cudaTypedefs.h>
#include <cuda_runtime.h>

struct FFTensorMapDriver {
  PFN_cuTensorMapEncodeTiled encode;
};
inline const FFTensorMapDriver& ff_tensor_map_driver() {
  static const FFTensorMapDriver driver = [] {
    auto find = [](const char* name) -> void* {
      void* fn = nullptr;
      cudaDriverEntryPointQueryResult qr;
      return cudaGetDriverEntryPoint(name, &fn, cudaEnableDefault, &qr) == cudaSuccess ? fn : nullptr;
    };
    return FFTensorMapDriver{(PFN_cuTensorMapEncodeTiled)find("cuTensorMapEncodeTiled")};
  }();
  return driver;
}
inline bool ff_encode_map(CUtensorMap* map, CUtensorMapDataType type, int rank, const void* base, const cuuint64_t* dims,
                          const cuuint64_t* strides, const cuuint32_t* box, CUtensorMapSwizzle swizzle, CUtensorMapL2promotion l2) {
  const auto encode = ff_tensor_map_driver().encode;
  const cuuint32_t steps[5] = {1, 1, 1, 1, 1};
  return encode && encode(map, type, (cuuint32_t)rank, const_cast<void*>(base), dims, strides, box, steps, CU_TENSOR_MAP_INTERLEAVE_NONE,
                          swizzle, l2, CU_TENSOR_MAP_FLOAT_OOB_FILL_NONE) == CUDA_SUCCESS;
}
