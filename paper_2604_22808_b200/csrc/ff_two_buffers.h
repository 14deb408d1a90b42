// Hand-over of two staging buffers that several warps fill together, step by step, and one of them (the issuer) sends out:
//   1  (from step 2 on) the issuer waits until the stores of step - 2 have read the buffer, and frees it; all wait for that
//   2  every warp writes its part of the buffer and arrives at full(step)
//   3  the issuer waits for full(step) and issues the stores
// A full barrier per buffer: the first two steps wait for no free buffer, and only the issuer waits for a full one, so a warp
// may arrive for step 1 before another has arrived for step 0.  On one barrier its second arrival would stand in for the
// missing first one, and the issuer would send out a part that nobody has written yet.  On its own barrier a warp's second
// arrival comes after the free barrier of that step, hence after the issuer has passed the full one of step - 1 and step - 2.
// One free barrier does: the issuer arrives there for step + 1 only after full(step), which every warp arrives at behind its
// own wait for free(step), so no phase ends unseen.
// No CUDA in here: tests/test_two_buffers.py runs these functions through every order of the warps.
#pragma once

#if defined(__CUDACC__)
#define FF_TB __host__ __device__ __forceinline__
#else
#define FF_TB inline
#endif

struct FFTwoBuffers {
  static constexpr int BUFFERS = 2, FULL = 2;                                 // buffers, full barriers
  FF_TB static int buffer(unsigned step) { return (int)(step & 1); }
  FF_TB static int full(unsigned step) { return buffer(step); }
  FF_TB static unsigned full_parity(unsigned step) { return (step >> 1) & 1; }
  FF_TB static bool waits_free(unsigned step) { return step >= BUFFERS; }
  FF_TB static unsigned free_parity(unsigned step) { return step & 1; }       // (its first phase ends at step 2)
};
#undef FF_TB
