// Small device helpers of the kernels that read band token lists.
#pragma once
#include "ff_internal.h"

template <typename T> __device__ __forceinline__ float ldf(const T* p);
template <> __device__ __forceinline__ float ldf<float>(const float* p) { return *p; }
template <> __device__ __forceinline__ float ldf<__nv_bfloat16>(const __nv_bfloat16* p) { return __bfloat162float(*p); }
template <typename T> __device__ __forceinline__ void stf(T* p, float v);
template <> __device__ __forceinline__ void stf<float>(float* p, float v) { *p = v; }
template <> __device__ __forceinline__ void stf<__nv_bfloat16>(__nv_bfloat16* p, float v) { *p = __float2bfloat16_rn(v); }

// four channels
__device__ __forceinline__ float4 ld4(const float* p) { return *(const float4*)p; }
__device__ __forceinline__ float4 ld4(const __nv_bfloat16* p) {
  const uint2 w = *(const uint2*)p;
  return make_float4(__uint_as_float(w.x << 16), __uint_as_float(w.x & 0xffff0000u), __uint_as_float(w.y << 16),
                     __uint_as_float(w.y & 0xffff0000u));
}
__device__ __forceinline__ void st4(float* p, const float4& v) { *(float4*)p = v; }
__device__ __forceinline__ void st4(__nv_bfloat16* p, const float4& v) {
  const __nv_bfloat162 a = __floats2bfloat162_rn(v.x, v.y), b = __floats2bfloat162_rn(v.z, v.w);
  *(uint2*)p = make_uint2(*(const uint32_t*)&a, *(const uint32_t*)&b);
}

__device__ __forceinline__ float warp_sum(float v) {
#pragma unroll
  for (int o = 16; o > 0; o >>= 1) v += __shfl_xor_sync(0xffffffffu, v, o);
  return v;
}

// ------------------------------------------------------------------------------------------------
// Working output of band `band` of head `bh` ("Cross-band residual exchange"): the operator's
// output where the head's mask has the band, the value coefficients V~ otherwise.
// ------------------------------------------------------------------------------------------------
template <typename ST>
struct BandView {
  const float* f32;   // low band rows (pooled output or V~ low)
  const ST* st;       // mid / high rows
  long long n;        // working length
  bool compressed;    // low band executed: row of rank p is p / r
};

template <typename ST>
__device__ __forceinline__ BandView<ST> band_view(const FFBuffers& buf, const FFDims& dm, int bh, int band) {
  BandView<ST> v;
  const bool exec = buf.alloc[bh] & (1 << band);
  const int d = dm.d;
  v.f32 = nullptr; v.st = nullptr; v.compressed = false;
  if (band == 0) {
    if (exec) { v.f32 = buf.y_low + (size_t)bh * dm.Nbar * d; v.n = dm.Nbar; v.compressed = true; }
    else { v.f32 = buf.spec_low + ((size_t)2 * dm.BH + bh) * dm.Nlow * d; v.n = dm.Nlow; }
  } else if (band == 1) {
    v.n = dm.Nmid;
    v.st = exec ? (const ST*)buf.y_mid + (size_t)bh * dm.Nmid * d
                : (const ST*)buf.spec_mid + ((size_t)2 * dm.BH + bh) * dm.Nmid * d;
  } else {
    v.n = dm.Nhigh;
    v.st = exec ? (const ST*)buf.y_high + (size_t)bh * dm.Nhigh * d
                : (const ST*)buf.spec_high + ((size_t)2 * dm.BH + bh) * dm.Nhigh * d;
  }
  return v;
}
