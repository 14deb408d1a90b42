// The driver's tensor-map calls, looked up once, and the one kind of map the kernels use: tiled, densely packed elements,
// zeros outside the tensor.
#pragma once
#include <cuda.h>
#include <cudaTypedefs.h>
#include <cuda_runtime.h>

struct FFTensorMapDriver {
  PFN_cuTensorMapEncodeTiled encode;
  PFN_cuTensorMapReplaceAddress replace_address;
};
inline const FFTensorMapDriver& ff_tensor_map_driver() {
  static const FFTensorMapDriver driver = [] {
    auto find = [](const char* name) -> void* {
      void* fn = nullptr;
      cudaDriverEntryPointQueryResult qr;
      return cudaGetDriverEntryPoint(name, &fn, cudaEnableDefault, &qr) == cudaSuccess ? fn : nullptr;
    };
    return FFTensorMapDriver{(PFN_cuTensorMapEncodeTiled)find("cuTensorMapEncodeTiled"),
                             (PFN_cuTensorMapReplaceAddress)find("cuTensorMapReplaceAddress")};
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

// Tensor maps kept between calls: encoding the two dozen of a forward took longer on the host than the launches they are
// for.  An entry is known by what the plan's configuration makes of it (the encoder's own code and the number of slices),
// never by an address: every use puts in the address it is for, so new tensors cost what old ones do.
struct FFMapCache {
  static constexpr int N = 48;             // (a plan has at most 40 kinds; with more, the last ones are encoded every time)
  CUtensorMap map[N];
  int code[N], slices[N];
  int used;
  template <class Encode>
  bool get(CUtensorMap* out, const void* base, int c, int s, Encode encode) {
    const auto replace = ff_tensor_map_driver().replace_address;
    for (int i = 0; replace && i < used; ++i)
      if (code[i] == c && slices[i] == s) { *out = map[i]; return replace(out, const_cast<void*>(base)) == CUDA_SUCCESS; }
    if (!encode()) return false;
    if (used < N) { map[used] = *out; code[used] = c; slices[used] = s; ++used; }
    return true;
  }
};
