// Three-byte form of an fp32 value: the value rounded to 24 bits, its upper 16 bits (a bf16 by truncation) in one grid
// and the next 8 bits in a byte grid.
#pragma once
#include <cuda_runtime.h>
#include <stdint.h>

// Half of the last of the 24 bits.  Added to the bits of a NaN as arithmetic produces it (0x7fffffff) it would wrap to
// -0: whoever knows a value to be NaN adds nothing, ff_round24 holds such bits back.
constexpr uint32_t FF_HALF24 = 0x80u;

__device__ __forceinline__ uint32_t ff_round24(uint32_t bits) { return (uint32_t)min((int)bits, 0x7fffff7f) + FF_HALF24; }
__device__ __forceinline__ uint32_t ff_round24(float v) { return ff_round24(__float_as_uint(v)); }

// Upper halves of two rounded values, bytes of four.
__device__ __forceinline__ uint32_t ff_hi2(uint32_t u0, uint32_t u1) { return __byte_perm(u0, u1, 0x7632); }
__device__ __forceinline__ uint32_t ff_lo4(uint32_t u0, uint32_t u1, uint32_t u2, uint32_t u3) {
  return __byte_perm(__byte_perm(u0, u1, 0x0051), __byte_perm(u2, u3, 0x0051), 0x5410);
}
