// The first launch of the forward and the last one of the inverse transform ("Separable spectral decomposition",
// "Reconstruction") where the t axis has 16 positions: the w axis on the tensor cores, t in fp32 registers.  bf16 storage, DCT-II.
//
// A 16 x 16 matrix is too small for the tensor core: as Mat kron I it fills an eighth of the 128 x 128 operand that
// ff_dct2_tc.cu multiplies with, three times over for the hi/lo parts, and its input has to go from the accumulators through
// registers and shared memory to become an operand.  Here a thread takes all 16 t coefficients of a (h, w) position from the
// accumulators of the w axis and folds them (C[k][15 - i] = (-1)^k C[k][i]: even and odd k apart), eight
// FMA and one addition a value, in fp32.  On long runs every launch of this path meets the board's power limit; three of six
// tensor products and the plane's way through shared memory are energy, too.
//
// A work item is 16 t x 128 (h, w) positions (128/W neighbouring h) x 16 channels of a head.  A tile of 128 positions at
// one t is the MN-major B operand (32-byte rows, 32-byte swizzle), the matrix I kron C_w the A operand in tensor memory
// (hi and lo bf16 parts); eight tiles share one instruction (N = 128).  D holds a position per lane and (t, channel) in its
// columns, so that nothing crosses lanes; 256 columns an item and 128 more for the first half of the next.
//   warp 0       TMA producer (ring of twelve slots: two tiles as a hi/lo pair)
//   warp 1       tcgen05.mma issuer; owns the tensor-memory allocation
//   warps 2..17  epilogue: four warps per 32 lanes; a warp makes four of the 16 t positions (two pairs i, 15 - i) for all
//                channels, stages its rows and sends two t positions at a time out with a tensor store
// Every wait is bounded.
//
// Bound by its epilogue and the loads: six heads of 64K tokens alone 62 us, 0.3 GB at 4.9 TB/s, issue slots 50%.  The four
// warps of 32 lanes share a scheduler; when each made all t positions of four channels and they staged whole rows together, the
// scheduler stood still at every hand-over: 69 us, six heads of 16K tokens 193 -> 190 for the whole layer.  With ff_dct2_tc.cu in
// this launch's place it took 334 us for 24 heads of 64K tokens at 1.6 GHz, with the shared staging 254.  The forward launch has a kernel of its own, below.
#include <cuda.h>

#include <vector>

#include "ff_clocks.cuh"
#include "ff_internal.h"
#include "ff_sm100.cuh"

using namespace sm100;

namespace {

constexpr int T = 16, C = 16;                  // t positions, channels of an item
constexpr int ROWS = 128;                      // positions of a tile
constexpr int TILE_B = ROWS * C * 2;           // 4 KB as bf16
constexpr int SLOT_B = 2 * TILE_B;             // two t positions
constexpr int BATCH = 4;                       // slots of an instruction batch: N = 8 tiles of 16 channels
constexpr int NSLOT = 12, LO_OFF = NSLOT * SLOT_B;     // ring: three batches, the hi parts, behind them their lo parts (192 KB)
constexpr int NACC = 3;                        // accumulator buffers of 128 columns, behind the matrix (2 x 64)
constexpr int EPI = 4;                         // epilogue warps per 32 lanes
constexpr int THREADS = 64 + 4 * EPI * 32;
constexpr int BOX_B = 2 * 32 * C * 2;          // 2 KB: 32 positions at two t, staged for a store (an area per epilogue warp)

struct T16Params {
  FFDims dm;
  const uint32_t* img;     // matrix of the w axis: hi [128][64] cells, then lo
  alignas(16) float mat[T][T / 2];     // mat[k][i] = C[k][i], i < 8
  int group, group_start;  // heads of the launch, the first one's place in the caller's tensor
  int nchunk, nh, hpt;     // channel chunks, groups of h positions, h positions of a group (128 / W; forward: 64 / W)
  double* clear;           // (forward) band energies to clear for the sums that follow (first launch of a routed forward), or NULL
  int* status;
};

// Nobody arrives twice in one phase of any of these: a second arrival always lies behind a wait for the first one's phase.
//   full       the producer, again for a slot behind empty, which the issuer commits behind its wait for full
//   empty      the issuer's commit, again behind full, which the producer arms behind its wait for empty
//   acc_full   the issuer's commit, again for a buffer behind acc_empty, where all epilogue threads arrive behind acc_full
//   acc_empty  an epilogue thread, again behind acc_full, which the issuer commits behind its wait for acc_empty
struct T16Shared {
  uint64_t full[NSLOT], empty[NSLOT], acc_full[NACC], acc_empty[NACC];
  uint32_t tmem_base;
  int abort_flag;
};

// Shared-memory descriptor of an MN-major operand stored as rows of 16 bf16 with the 32-byte swizzle: 8-row groups 256 bytes
// apart, tiles of 16 channels (along N) TILE_B apart.
__device__ __forceinline__ uint64_t smem_desc_sw32(uint32_t smem_addr) {
  return (uint64_t)((smem_addr & 0x3FFFF) >> 4) | (uint64_t)(TILE_B >> 4) << 16 | (uint64_t)(256 >> 4) << 32 | (uint64_t)1 << 46 | (uint64_t)6 << 61;
}

// The matrix (hi, then lo part) into tensor memory by four warps: a thread loads the row of its lane.
__device__ __forceinline__ void matrix_to_tmem(const uint32_t* img, uint32_t tm, int quarter, int lane) {
  const int row = quarter * 32 + lane;
  const uint32_t lane_addr = (uint32_t)(quarter * 32) << 16;
#pragma unroll 1
  for (int c0 = 0; c0 < 128; c0 += 32) {
    const uint32_t* src = img + (size_t)(c0 >> 6) * FF_IMAGE_PART + (size_t)row * 64 + (c0 & 63);
    uint32_t r[32];
#pragma unroll
    for (int i = 0; i < 8; ++i) {
      const uint4 v = *(const uint4*)(src + 4 * i);
      r[4 * i] = v.x; r[4 * i + 1] = v.y; r[4 * i + 2] = v.z; r[4 * i + 3] = v.w;
    }
    tmem_st32(tm + lane_addr + c0, r);
  }
  tmem_wait_st();
}

// map_hi, map_lo: the pair of grids; map_out: the caller's tensor, box = 32 positions at two t.
__global__ void __launch_bounds__(THREADS, 1)
dct_t16_kernel(const __grid_constant__ CUtensorMap map_hi, const __grid_constant__ CUtensorMap map_lo,
               const __grid_constant__ CUtensorMap map_out, const __grid_constant__ T16Params P) {
  extern __shared__ uint8_t smem_raw[];
  uint8_t* smem = (uint8_t*)(((uintptr_t)smem_raw + 1023) & ~(uintptr_t)1023);
  const FFDims& dm = P.dm;
  constexpr uint32_t COL_ACC = 128;
  uint8_t* sIn = smem;
  uint8_t* sStage = smem + 2 * LO_OFF;                      // an area per epilogue warp
  T16Shared& sh = *(T16Shared*)(sStage + 4 * EPI * BOX_B);
  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
  const int total = P.group * P.nh * P.nchunk;

  if (threadIdx.x == 0) {
    for (int i = 0; i < NSLOT; ++i) { mbar_init(&sh.full[i], 1); mbar_init(&sh.empty[i], 1); }
    for (int i = 0; i < NACC; ++i) { mbar_init(&sh.acc_full[i], 1); mbar_init(&sh.acc_empty[i], 4 * EPI * 32); }
    sh.abort_flag = 0;
    fence_mbar_init();
  }
  if (warp == 1) { tmem_alloc(&sh.tmem_base, 512); tmem_relinquish(); }
  tc_fence_before();
  __syncthreads();
  tc_fence_after();
  const uint32_t tm = sh.tmem_base;
  volatile int* abort_flag = &sh.abort_flag;
  if (warp >= 2 && warp < 6) matrix_to_tmem(P.img, tm, warp & 3, lane);
  // (the next launch comes in when this one's blocks end: let in earlier, its blocks slowed the last third of this
  // launch down, 16K tokens, six heads: 30.6 us instead of 22.3)
  ff_pdl_join();
  tc_fence_before();
  __syncthreads();
  tc_fence_after();

  FF_CLOCK(t_all);
  // Item: chunk fastest (CTAs that run side by side read neighbouring pieces of the same rows), then h, then the head.
  if (warp == 0) {
    if (lane == 0) {
      tma_prefetch_desc(&map_hi); tma_prefetch_desc(&map_lo);
      unsigned n = 0;
      bool ok = true;
      for (int it = blockIdx.x; it < total && ok; it += gridDim.x) {
        const int chunk = it % P.nchunk, rest = it / P.nchunk, h0 = rest % P.nh * P.hpt, gi = rest / P.nh;
        for (int k = 0; k < T / 2 && ok; ++k, ++n) {
          const int slot = n % NSLOT;
          FF_CLOCK(tp);
          if (n >= (unsigned)NSLOT) ok = mbar_wait(&sh.empty[slot], ((n / NSLOT) - 1) & 1, abort_flag);
          FF_CLOCK_ADD(true, 0, tp);
          if (!ok) break;
          // (debug build) the box lies inside the grid; a refused item ends in the bounded wait of its consumer
          if (!FF_DBG_OK((chunk + 1) * C <= dm.d && h0 + P.hpt <= dm.H && gi < P.group, P.status, 7)) continue;
          uint8_t* dst = sIn + slot * SLOT_B;
          mbar_arrive_expect_tx(&sh.full[slot], 2 * SLOT_B);
          tma_load_5d(dst, &map_hi, &sh.full[slot], chunk * C, 0, h0, 2 * k, gi);
          tma_load_5d(dst + LO_OFF, &map_lo, &sh.full[slot], chunk * C, 0, h0, 2 * k, gi);
        }
      }
    }
  } else if (warp == 1) {
    const uint32_t idesc = idesc_bf16_f32(ROWS, 128, /*a_mn_major=*/false, /*b_mn_major=*/true);
    const uint32_t in_base = smem_u32(sIn);
    unsigned nb = 0;
    bool ok = true;
    for (int it = blockIdx.x; it < total && ok; it += gridDim.x) {
      for (int half = 0; half < 2 && ok; ++half, ++nb) {
        const int ab = nb % NACC, s0 = nb * BATCH % NSLOT;
        FF_CLOCK(ti);
        for (int i = 0; i < BATCH && ok; ++i) ok = mbar_wait_warp(&sh.full[s0 + i], (nb * BATCH / NSLOT) & 1, abort_flag);
        FF_CLOCK_ADD(lane == 0, 1, ti);
        FF_CLOCK(ta);
        if (ok && nb >= NACC) ok = mbar_wait_warp(&sh.acc_empty[ab], ((nb / NACC) - 1) & 1, abort_flag);
        FF_CLOCK_ADD(lane == 0, 2, ta);
        if (!ok) break;
        tc_fence_after();
        const uint64_t xh = smem_desc_sw32(in_base + s0 * SLOT_B), xl = smem_desc_sw32(in_base + s0 * SLOT_B + LO_OFF);
        const uint32_t d_tm = tm + COL_ACC + ab * 128;
#pragma unroll
        for (int ks = 0; ks < ROWS / 16; ++ks) {           // (16 rows of K: 512 bytes, 32 in a descriptor's address field)
          umma_ts(d_tm, tm + ks * 8, xh + (uint64_t)(ks * 32), idesc, ks > 0 ? 1u : 0u);
          umma_ts(d_tm, tm + 64 + ks * 8, xh + (uint64_t)(ks * 32), idesc, 1u);
          umma_ts(d_tm, tm + ks * 8, xl + (uint64_t)(ks * 32), idesc, 1u);
        }
        for (int i = 0; i < BATCH; ++i) umma_commit(&sh.empty[s0 + i]);
        umma_commit(&sh.acc_full[ab]);
      }
    }
  } else {
    const int quarter = warp & 3, part = (warp - 2) >> 2;  // TMEM lanes; which t: 2 part, 2 part + 1 and 14 - 2 part, 15 - 2 part
    const uint32_t lane_addr = (uint32_t)(quarter * 32) << 16;
    const int p0 = quarter * 32;                           // the warp's first position: w fastest, then h
    const int w0 = p0 % dm.W, hq = p0 / dm.W;
    const int i0 = __shfl_sync(0xffffffffu, 2 * part, 0);
    uint8_t* stage = sStage + (warp - 2) * BOX_B;
    unsigned nb = 0;
    bool ok = true;
    for (int it = blockIdx.x; it < total && ok; it += gridDim.x) {
      const int chunk = it % P.nchunk, rest = it / P.nchunk, h0 = rest % P.nh * P.hpt + hq, gi = rest / P.nh;
      float e[2][C] = {}, o[2][C] = {};
#pragma unroll 1
      for (int b = 0; b < 2; ++b, ++nb) {
        const int ab = nb % NACC;
        FF_CLOCK(te);
        ok = mbar_wait_warp(&sh.acc_full[ab], (nb / NACC) & 1, abort_flag);
        FF_CLOCK_ADD(threadIdx.x == 64, 3, te);
        if (!ok) break;
        tc_fence_after();
#pragma unroll 1
        for (int k2 = 0; k2 < T / 2; k2 += 2)
#pragma unroll
          for (int odd = 0; odd < 2; ++odd) {
            const int k = k2 + odd;
            uint32_t x[C];
            tmem_ld16(tm + lane_addr + COL_ACC + ab * 128 + k * C, x);
            const float2 m = *(const float2*)(P.mat[b * 8 + k] + i0);
            tmem_wait_ld();
#pragma unroll
            for (int c = 0; c < C; ++c) {
              float& f0 = odd ? o[0][c] : e[0][c];
              float& f1 = odd ? o[1][c] : e[1][c];
              f0 = fmaf(m.x, __uint_as_float(x[c]), f0);
              f1 = fmaf(m.y, __uint_as_float(x[c]), f1);
            }
          }
        tc_fence_before();
        mbar_arrive(&sh.acc_empty[ab]);
      }
      if (!ok) break;
      FF_CLOCK(tw);
#pragma unroll
      for (int back = 0; back < 2; ++back) {               // the two t of one end, then those of the other
        uint32_t v[2][C / 2];
#pragma unroll
        for (int j = 0; j < 2; ++j)
#pragma unroll
          for (int c = 0; c < C; c += 2)
            v[j][c / 2] = back ? bf16_pair(__float_as_uint(e[1 - j][c] - o[1 - j][c]), __float_as_uint(e[1 - j][c + 1] - o[1 - j][c + 1]))
                               : bf16_pair(__float_as_uint(e[j][c] + o[j][c]), __float_as_uint(e[j][c + 1] + o[j][c + 1]));
        FF_CLOCK(tb);
        if (lane == 0) bulk_wait_read0();                  // the warp's previous store has read the area
        __syncwarp();
        FF_CLOCK_ADD(threadIdx.x == 64, 4, tb);
#pragma unroll
        for (int j = 0; j < 2; ++j)
#pragma unroll
          for (int c = 0; c < 2; ++c)                      // (32-byte swizzle)
            *(uint4*)(stage + j * (BOX_B / 2) + lane * 32 + ((c ^ ((lane >> 2) & 1)) << 4)) = make_uint4(v[j][4 * c], v[j][4 * c + 1], v[j][4 * c + 2], v[j][4 * c + 3]);
        fence_proxy_async();
        __syncwarp();
        // (debug build) its 32 positions are whole lines of the plane, or lie in one
        if (lane == 0 && FF_DBG_OK((chunk + 1) * C <= dm.d && w0 + (dm.W < 32 ? dm.W : 32) <= dm.W &&
                                       h0 + (dm.W < 32 ? 32 / dm.W : 1) <= dm.H && P.group_start + gi < dm.BH, P.status, 7)) {
          tma_store_5d(stage, &map_out, chunk * C, w0, h0, back ? 14 - i0 : i0, P.group_start + gi);
          bulk_commit();
        }
      }
      FF_CLOCK_ADD(threadIdx.x == 64, 6, tw);
    }
    if (lane == 0) bulk_wait0();
    FF_CLOCK_ADD(threadIdx.x == 64, 7, t_all);
  }

  tc_fence_before();
  __syncthreads();
  if (sh.abort_flag) {
    if (threadIdx.x == 0) atomicExch(P.status, FF_ERR_TIMEOUT | 0x700);   // low byte: status, next byte: which kernel
    const long long t0 = clock64();
    while (clock64() - t0 < 2000000) { }
    __syncthreads();
  }
  if (warp == 1) {
    tc_fence_after();
    tmem_dealloc(tm, 512);
  }
}

// ------------------------------------------------------------------------------------------------------------------
// Forward.  w on the tensor cores, t in fp32 registers, and the fold of t on the tensor cores, too: a tile is 64 positions at
// t = i over the same 64 at t = 15 - i, the operand [[M, M], [M, -M]] with M = I kron C_w.  Lanes 0..63 then hold the w transform
// of x[i] + x[15 - i], lanes 64..127 that of x[i] - x[15 - i], and a thread makes the eight even or the eight odd t coefficients
// of its position from eight numbers a channel: an item of 32 channels takes the 256 accumulator columns that one of 16 would
// take unfolded, and rows of 64 bytes go in and out.
//   warp 0       TMA producer (ring of five batches of four tiles)
//   warp 1       tcgen05.mma issuer; owns the tensor-memory allocation
//   warps 2..17  epilogue: four warps per 32 lanes, two coefficients each; a warp stages and sends its rows by itself.  (The
//                four warps of 32 lanes share a scheduler: when they shared the staging area, too, eight channels each, it stood
//                still at every hand-over.)
// Every wait is bounded.
//
// Bound by HBM and, close behind, by the epilogue: six heads of 64K tokens alone 163 us, 0.9 GB at 5.6 TB/s, issue slots 62%.
// ff_dct2_tc.cu sends the intermediate through shared memory as a bf16 pair and multiplies t with a 128 x 128 operand that is
// seven eighths zeros.  Layers before and after (us, 24 heads of 64K tokens at 1.6 GHz 2850 / 2711; all bands 3575 / 3417; 16 heads
// with head_dim 64 1025 / 967; six heads of 16K 206 / 193, four of 8K 126 / 118, six of 128K 1581 / 1501).  A line of 128
// positions does not fit twice into the operand: that grid keeps the two-axis launch.  Variants (six heads of 64K): eight channels a
// thread, staged by four warps together, coefficients as constants of unrolled code 201 us (instruction cache), in a loop 177; packed
// FMA 181; without its stores that form took 155, without its FMA 163.
constexpr int FC = 32, FPOS = 64;                          // channels, positions of an item
constexpr int F_TILE_B = 2 * FPOS * FC * 2;                // 8 KB
constexpr int F_NSLOT = 5, F_SLOT_B = 4 * F_TILE_B;        // ring
constexpr int F_BOX_B = 32 * FC * 2;                       // 2 KB: 32 positions at one t, hi or lo
constexpr int F_STAGE_B = 2 * F_BOX_B;                     // staging area of an epilogue warp

struct T16ForwardShared {
  uint64_t full[F_NSLOT], empty[F_NSLOT], acc_full[NACC], acc_empty[NACC];
  uint32_t tmem_base;
  int abort_flag;
};

// Descriptor of an MN-major operand stored as rows of 32 bf16 with the 64-byte swizzle, tiles F_TILE_B apart along N.
__device__ __forceinline__ uint64_t smem_desc_sw64(uint32_t smem_addr) {
  return (uint64_t)((smem_addr & 0x3FFFF) >> 4) | (uint64_t)(F_TILE_B >> 4) << 16 | (uint64_t)(512 >> 4) << 32 | (uint64_t)1 << 46 | (uint64_t)4 << 61;
}
// map0..map2: Q, K, V; map_oh, map_ol: the pair of grids, box = 32 positions at one t.
__global__ void __launch_bounds__(THREADS, 1)
dct_t16_forward_kernel(const __grid_constant__ CUtensorMap map0, const __grid_constant__ CUtensorMap map1,
                       const __grid_constant__ CUtensorMap map2, const __grid_constant__ CUtensorMap map_oh,
                       const __grid_constant__ CUtensorMap map_ol, const __grid_constant__ T16Params P) {
  extern __shared__ uint8_t smem_raw[];
  uint8_t* smem = (uint8_t*)(((uintptr_t)smem_raw + 1023) & ~(uintptr_t)1023);
  const FFDims& dm = P.dm;
  constexpr uint32_t COL_ACC = 128;
  uint8_t* sIn = smem;
  uint8_t* sStage = smem + F_NSLOT * F_SLOT_B;              // an area per epilogue warp
  T16ForwardShared& sh = *(T16ForwardShared*)(sStage + 4 * EPI * F_STAGE_B);
  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
  const int total = P.group * P.nh * P.nchunk;

  if (threadIdx.x == 0) {
    for (int i = 0; i < F_NSLOT; ++i) { mbar_init(&sh.full[i], 1); mbar_init(&sh.empty[i], 1); }
    for (int i = 0; i < NACC; ++i) { mbar_init(&sh.acc_full[i], 1); mbar_init(&sh.acc_empty[i], 4 * EPI * 32); }
    sh.abort_flag = 0;
    fence_mbar_init();
  }
  if (warp == 1) { tmem_alloc(&sh.tmem_base, 512); tmem_relinquish(); }
  tc_fence_before();
  __syncthreads();
  tc_fence_after();
  const uint32_t tm = sh.tmem_base;
  volatile int* abort_flag = &sh.abort_flag;
  if (warp >= 2 && warp < 6) matrix_to_tmem(P.img, tm, warp & 3, lane);
  ff_pdl_wait();
  if (P.clear && blockIdx.x == 0) for (int i = threadIdx.x; i < dm.B * 3 * dm.d; i += THREADS) P.clear[i] = 0.0;
  tc_fence_before();
  __syncthreads();
  tc_fence_after();

  FF_CLOCK(t_all);
  // Item: chunk fastest (CTAs that run side by side read neighbouring pieces of the same rows), then 64 positions, then the tensor-head.
  if (warp == 0) {
    if (lane == 0) {
      tma_prefetch_desc(&map0);
      unsigned n = 0;
      bool ok = true;
      for (int it = blockIdx.x; it < total && ok; it += gridDim.x) {
        const int chunk = it % P.nchunk, rest = it / P.nchunk, p0 = rest % P.nh * FPOS, gi = rest / P.nh;
        const int th = P.group_start + gi, tensor = (th >= dm.BH) + (th >= 2 * dm.BH);
        const CUtensorMap* map = tensor == 0 ? &map0 : (tensor == 1 ? &map1 : &map2);
        for (int b = 0; b < 2 && ok; ++b, ++n) {
          const int slot = n % F_NSLOT;
          FF_CLOCK(tp);
          if (n >= (unsigned)F_NSLOT) ok = mbar_wait(&sh.empty[slot], ((n / F_NSLOT) - 1) & 1, abort_flag);
          FF_CLOCK_ADD(true, 16, tp);
          if (!ok) break;
          uint8_t* dst = sIn + slot * F_SLOT_B;
          mbar_arrive_expect_tx(&sh.full[slot], F_SLOT_B);
#pragma unroll
          for (int k = 0; k < 4; ++k) {
            const int i = b * 4 + k;
            tma_load_5d(dst + k * F_TILE_B, map, &sh.full[slot], chunk * FC, p0, i, th - tensor * dm.BH, 0);
            tma_load_5d(dst + k * F_TILE_B + F_TILE_B / 2, map, &sh.full[slot], chunk * FC, p0, 15 - i, th - tensor * dm.BH, 0);
          }
        }
      }
    }
  } else if (warp == 1) {
    const uint32_t idesc = idesc_bf16_f32(ROWS, 128, /*a_mn_major=*/false, /*b_mn_major=*/true);
    const uint32_t in_base = smem_u32(sIn);
    unsigned nb = 0;
    bool ok = true;
    for (int it = blockIdx.x; it < total && ok; it += gridDim.x) {
      for (int half = 0; half < 2 && ok; ++half, ++nb) {
        const int ab = nb % NACC, slot = nb % F_NSLOT;
        FF_CLOCK(ti);
        ok = mbar_wait_warp(&sh.full[slot], (nb / F_NSLOT) & 1, abort_flag);
        FF_CLOCK_ADD(lane == 0, 17, ti);
        FF_CLOCK(ta);
        if (ok && nb >= NACC) ok = mbar_wait_warp(&sh.acc_empty[ab], ((nb / NACC) - 1) & 1, abort_flag);
        FF_CLOCK_ADD(lane == 0, 18, ta);
        if (!ok) break;
        tc_fence_after();
        const uint64_t x = smem_desc_sw64(in_base + slot * F_SLOT_B);
        const uint32_t d_tm = tm + COL_ACC + ab * 128;
#pragma unroll
        for (int ks = 0; ks < ROWS / 16; ++ks) {           // (16 rows of K: 1024 bytes, 64 in a descriptor's address field)
          umma_ts(d_tm, tm + ks * 8, x + (uint64_t)(ks * 64), idesc, ks > 0 ? 1u : 0u);
          umma_ts(d_tm, tm + 64 + ks * 8, x + (uint64_t)(ks * 64), idesc, 1u);
        }
        umma_commit(&sh.empty[slot]);
        umma_commit(&sh.acc_full[ab]);
      }
    }
  } else {
    const int quarter = warp & 3, part = (warp - 2) >> 2;  // TMEM lanes; which two of the lanes' eight coefficients
    const uint32_t lane_addr = (uint32_t)(quarter * 32) << 16;
    const int k0 = __shfl_sync(0xffffffffu, 4 * part + (quarter >> 1), 0);       // coefficients k0 and k0 + 2
    uint8_t* stage = sStage + (warp - 2) * F_STAGE_B;
    unsigned nb = 0;
    bool ok = true;
    for (int it = blockIdx.x; it < total && ok; it += gridDim.x) {
      const int chunk = it % P.nchunk, rest = it / P.nchunk, p0 = rest % P.nh * FPOS + (quarter & 1) * 32, gi = rest / P.nh;
      float y[2][FC] = {};
#pragma unroll 1
      for (int b = 0; b < 2; ++b, ++nb) {
        const int ab = nb % NACC;
        FF_CLOCK(te);
        ok = mbar_wait_warp(&sh.acc_full[ab], (nb / NACC) & 1, abort_flag);
        FF_CLOCK_ADD(threadIdx.x == 64, 19, te);
        if (!ok) break;
        tc_fence_after();
        const float4 ma = *(const float4*)(P.mat[k0] + 4 * b), mb = *(const float4*)(P.mat[k0 + 2] + 4 * b);
        const float m[2][4] = {{ma.x, ma.y, ma.z, ma.w}, {mb.x, mb.y, mb.z, mb.w}};
#pragma unroll
        for (int i = 0; i < 4; ++i)
#pragma unroll
          for (int h = 0; h < 2; ++h) {
            uint32_t x[16];
            tmem_ld16(tm + lane_addr + COL_ACC + ab * 128 + i * FC + h * 16, x);
            tmem_wait_ld();
#pragma unroll
            for (int j = 0; j < 2; ++j)
#pragma unroll
              for (int c = 0; c < 16; ++c) y[j][h * 16 + c] = fmaf(m[j][i], __uint_as_float(x[c]), y[j][h * 16 + c]);
          }
        tc_fence_before();
        mbar_arrive(&sh.acc_empty[ab]);
      }
      if (!ok) break;
      FF_CLOCK(tw);
#pragma unroll
      for (int j = 0; j < 2; ++j) {
        uint32_t hi[16], lo[16];
#pragma unroll
        for (int c = 0; c < 16; ++c) {
          hi[c] = bf16_pair(__float_as_uint(y[j][2 * c]), __float_as_uint(y[j][2 * c + 1]));
          lo[c] = bf16_pair(__float_as_uint(y[j][2 * c] - __uint_as_float(hi[c] << 16)), __float_as_uint(y[j][2 * c + 1] - __uint_as_float(hi[c] & 0xffff0000u)));
        }
        FF_CLOCK(tb);
        if (lane == 0) bulk_wait_read0();                  // the warp's previous stores have read the area
        __syncwarp();
        FF_CLOCK_ADD(threadIdx.x == 64, 20, tb);
#pragma unroll
        for (int c = 0; c < 4; ++c) {                      // (64-byte swizzle)
          uint8_t* at = stage + lane * 64 + ((c ^ ((lane >> 1) & 3)) << 4);
          *(uint4*)at = make_uint4(hi[4 * c], hi[4 * c + 1], hi[4 * c + 2], hi[4 * c + 3]);
          *(uint4*)(at + F_BOX_B) = make_uint4(lo[4 * c], lo[4 * c + 1], lo[4 * c + 2], lo[4 * c + 3]);
        }
        fence_proxy_async();
        __syncwarp();
        if (lane == 0) {
          // (debug build) the box lies inside the grid
          if (FF_DBG_OK((chunk + 1) * FC <= dm.d && p0 + 32 <= dm.H * dm.W && k0 + 2 * j < T && gi < P.group, P.status, 7)) {
            tma_store_5d(stage, &map_oh, chunk * FC, p0, k0 + 2 * j, gi, 0);
            tma_store_5d(stage + F_BOX_B, &map_ol, chunk * FC, p0, k0 + 2 * j, gi, 0);
          }
          bulk_commit();
        }
      }
      FF_CLOCK_ADD(threadIdx.x == 64, 22, tw);
    }
    if (lane == 0) bulk_wait0();
    FF_CLOCK_ADD(threadIdx.x == 64, 23, t_all);
  }

  tc_fence_before();
  __syncthreads();
  if (sh.abort_flag) {
    if (threadIdx.x == 0) atomicExch(P.status, FF_ERR_TIMEOUT | 0x700);
    const long long t0 = clock64();
    while (clock64() - t0 < 2000000) { }
    __syncthreads();
  }
  if (warp == 1) {
    tc_fence_after();
    tmem_dealloc(tm, 512);
  }
}

// Map over the same grid seen as [slices][t][h w][d]: 32 channels of 64 positions (load) or 32 (store) at one t.
bool forward_map(ff_plan* p, CUtensorMap* map, const void* base, int slices, bool store) {
  const FFDims& dm = p->dm;
  return p->maps.get(map, base, store ? 51 : 50, slices, [&] {
    const cuuint64_t ch = (cuuint64_t)dm.d, hw = (cuuint64_t)dm.H * dm.W, plane = hw * ch * 2;
    const cuuint64_t dims[5] = {ch, hw, T, (cuuint64_t)slices, 1};
    const cuuint64_t strides[4] = {ch * 2, plane, plane * T, plane * T * slices};
    const cuuint32_t box[5] = {FC, (cuuint32_t)(store ? 32 : FPOS), 1, 1, 1};
    return ff_encode_map(map, CU_TENSOR_MAP_DATA_TYPE_BFLOAT16, 5, base, dims, strides, box, CU_TENSOR_MAP_SWIZZLE_64B,
                         store ? CU_TENSOR_MAP_L2_PROMOTION_NONE : CU_TENSOR_MAP_L2_PROMOTION_L2_256B);
  });
}
constexpr size_t F_SMEM = 1024 + (size_t)F_NSLOT * F_SLOT_B + 4 * EPI * F_STAGE_B + sizeof(T16ForwardShared);

// 5-D map over a [slices][T][H][W][d] bf16 grid: the box of 16 channels of two tiles (load), or of 32 positions at two t (store).
bool grid_map(ff_plan* p, CUtensorMap* map, const void* base, int slices, bool store) {
  const FFDims& dm = p->dm;
  return p->maps.get(map, base, store ? 49 : 48, slices, [&] {
    const cuuint64_t ch = (cuuint64_t)dm.d, W = (cuuint64_t)dm.W;
    const cuuint64_t dims[5] = {ch, W, (cuuint64_t)dm.H, (cuuint64_t)dm.T, (cuuint64_t)slices};
    const cuuint64_t strides[4] = {ch * 2, W * ch * 2, dm.H * W * ch * 2, (cuuint64_t)dm.N * ch * 2};
    const cuuint32_t w = (cuuint32_t)(store && dm.W > 32 ? 32 : dm.W);
    const cuuint32_t box[5] = {C, w, (cuuint32_t)(store ? 32 : ROWS) / w, 2, 1};
    return ff_encode_map(map, CU_TENSOR_MAP_DATA_TYPE_BFLOAT16, 5, base, dims, strides, box, CU_TENSOR_MAP_SWIZZLE_32B,
                         store ? CU_TENSOR_MAP_L2_PROMOTION_NONE : CU_TENSOR_MAP_L2_PROMOTION_L2_256B);
  });
}

// (the swizzles are functions of the address: 1024-byte alignment)
constexpr size_t SMEM = 1024 + (size_t)2 * LO_OFF + 4 * EPI * BOX_B + sizeof(T16Shared);

}  // namespace

cudaError_t ffk_dct_t16_init() {
  const cudaError_t e = cudaFuncSetAttribute(dct_t16_kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)SMEM);
  return e != cudaSuccess ? e : cudaFuncSetAttribute(dct_t16_forward_kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)F_SMEM);
}

// Where it takes the place of the two-axis launch: t is that launch's second axis, 16 positions, and folds.
bool ffk_dct_t16_supported(const ff_plan* p) {
  return p->dct2_ok && p->dct2_axis2 == 0 && p->dm.T == T && p->cfg.transform == FF_TRANSFORM_DCT;
}

// Hi/lo grids of heads [h0, h0 + g) -> w and t inverse transform -> out.
cudaError_t ffk_dct_t16_inverse(ff_plan* p, const void* in_hi, const void* in_lo, int h0, int g, void* out, cudaStream_t st) {
  const FFDims& dm = p->dm;
  CUtensorMap mh, ml, mo;
  if (!grid_map(p, &mh, in_hi, p->dct_group, false) || !grid_map(p, &ml, in_lo, p->dct_group, false) || !grid_map(p, &mo, out, dm.BH, true))
    return cudaErrorInvalidValue;
  T16Params P{};
  P.dm = dm; P.status = p->buf.status;
  P.img = p->dct2_images + (size_t)(3 + 2) * FF_IMAGE_CELLS;
  memcpy(P.mat, p->t16_mat, sizeof(P.mat));
  P.group = g; P.group_start = h0;
  P.nchunk = dm.d / C; P.hpt = ROWS / dm.W; P.nh = dm.H / P.hpt;
  const int items = g * P.nh * P.nchunk;
  const cudaError_t e = ff_launch(dct_t16_kernel, dim3((unsigned)(items < p->sm_count ? items : p->sm_count)), dim3(THREADS), SMEM, st, mh, ml, mo, P);
  if (e == cudaSuccess) p->launches += 1;
  return e;
}

// Forward: Q, K, V of tensor-heads [g0, g0 + g) -> w and t transform -> hi/lo grids.
bool ffk_dct_t16_forward_supported(const ff_plan* p) { return ffk_dct_t16_supported(p) && p->dm.W <= FPOS; }

cudaError_t ffk_dct_t16_forward(ff_plan* p, const void* Q, const void* K, const void* V, int g0, int g, void* out_hi, void* out_lo,
                                bool clear_energy, cudaStream_t st) {
  const FFDims& dm = p->dm;
  CUtensorMap mq, mk, mv, oh, ol;
  if (!forward_map(p, &mq, Q, dm.BH, false) || !forward_map(p, &mk, K, dm.BH, false) || !forward_map(p, &mv, V, dm.BH, false) ||
      !forward_map(p, &oh, out_hi, p->dct_group, true) || !forward_map(p, &ol, out_lo, p->dct_group, true))
    return cudaErrorInvalidValue;
  T16Params P{};
  P.dm = dm; P.status = p->buf.status;
  P.img = p->dct2_images + (size_t)6 * FF_IMAGE_CELLS;
  memcpy(P.mat, p->t16_mat, sizeof(P.mat));
  P.group = g; P.group_start = g0;
  P.nchunk = dm.d / FC; P.hpt = FPOS / dm.W; P.nh = dm.H / P.hpt;
  P.clear = clear_energy ? p->buf.energy : nullptr;
  const int items = g * P.nh * P.nchunk;
  const cudaError_t e = ff_launch(dct_t16_forward_kernel, dim3((unsigned)(items < p->sm_count ? items : p->sm_count)), dim3(THREADS), F_SMEM, st,
                                  mq, mk, mv, oh, ol, P);
  if (e == cudaSuccess) p->launches += 1;
  return e;
}

// Its matrix as the tensor-memory A operand, hi and lo parts: [[M, M], [M, -M]], M = I kron C_w over 64 positions.
bool ffk_dct_t16_build_image(ff_plan* p, const float* mat) {
  const int n = p->dm.W;
  std::vector<uint32_t> img(2 * FF_IMAGE_PART);
  for (int j = 0; j < ROWS; ++j)
    for (int r = 0; r < ROWS; ++r) {
      const int a = j % FPOS, b = r % FPOS;
      if (a / n != b / n) continue;
      float v = mat[(a % n) * n + b % n];
      if (j >= FPOS && r >= FPOS) v = -v;
      size_t cell = (size_t)j * 64 + (r >> 1);
      for (int part = 0; part < 2; ++part, cell += FF_IMAGE_PART) {
        const __nv_bfloat16 h = __float2bfloat16_rn(v);
        const uint32_t hb = *(const uint16_t*)&h;
        img[cell] |= (r & 1) ? hb << 16 : hb;
        v -= __bfloat162float(h);
      }
    }
  return cudaMemcpy(p->dct2_images + (size_t)6 * FF_IMAGE_CELLS, img.data(), img.size() * sizeof(uint32_t), cudaMemcpyHostToDevice) == cudaSuccess;
}

FF_CLOCKS_READ(transform_t16)
