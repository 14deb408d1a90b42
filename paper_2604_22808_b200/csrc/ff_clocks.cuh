// Cycle sums of what a kernel's warps wait for and work on: `python -m paper_2604_22808_b200.clocks` builds the library
// with them (-DFF_CLOCKS) and prints them; every other build compiles them away.  One thread of a role adds; a kernel with
// clocks is slower than one without, so the shares count, not the sums.
#pragma once
#include <cuda_runtime.h>
#include <stdint.h>

#ifdef FF_CLOCKS
constexpr int FF_CLOCK_SLOTS = 64;
namespace {
__device__ unsigned long long ff_clock_sum[FF_CLOCK_SLOTS];     // times added in the upper 24 bits, cycles below
__device__ __forceinline__ void ff_clock_add(int slot, unsigned since) {
  atomicAdd(&ff_clock_sum[slot], (1ull << 40) + (unsigned)((unsigned)clock() - since));
}
}  // namespace
#define FF_CLOCK(t) const unsigned t = (unsigned)clock()
#define FF_CLOCK_ADD(on, slot, t) do { if (on) ff_clock_add((slot), (t)); } while (0)
// Reads and clears the sums of the translation unit's kernels.
#define FF_CLOCKS_READ(name)                                                                                       \
  extern "C" int32_t ff_clocks_##name(unsigned long long* sums) {                                                  \
    const unsigned long long zero[FF_CLOCK_SLOTS] = {};                                                            \
    cudaError_t e = cudaDeviceSynchronize();                                                                       \
    if (e == cudaSuccess) e = cudaMemcpyFromSymbol(sums, ff_clock_sum, sizeof(zero));                              \
    if (e == cudaSuccess) e = cudaMemcpyToSymbol(ff_clock_sum, zero, sizeof(zero));                                \
    return e == cudaSuccess ? 0 : 1;                                                                               \
  }
#else
#define FF_CLOCK(t)
#define FF_CLOCK_ADD(on, slot, t)
#define FF_CLOCKS_READ(name)
#endif
