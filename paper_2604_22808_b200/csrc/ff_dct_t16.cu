// Two axis passes in one launch with the second axis in fp32 registers instead of on the tensor cores ("Separable spectral
// decomposition", "Reconstruction"): the last launch of the inverse where the t axis has 16 positions, and, below, the first
// launch of the forward where the second axis, t or h, has 16 or 32.  bf16 storage, DCT-II.
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
// warps of 32 lanes share a scheduler; when each made all t positions of four channels and they staged whole rows together in two areas, the
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
  int nchunk, nh, hpt;     // channel chunks, groups of h positions, h positions of a group (128 / W)
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

// The matrix (hi part, the lo part LO cells behind it) into tensor memory by four warps: a thread loads the row of its lane.
template <size_t LO>
__device__ __forceinline__ void matrix_to_tmem(const uint32_t* img, uint32_t tm, int quarter, int lane) {
  const int row = quarter * 32 + lane;
  const uint32_t lane_addr = (uint32_t)(quarter * 32) << 16;
#pragma unroll 1
  for (int c0 = 0; c0 < 128; c0 += 32) {
    const uint32_t* src = img + (size_t)(c0 >> 6) * LO + (size_t)row * 64 + (c0 & 63);
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
  if (warp >= 2 && warp < 6) matrix_to_tmem<FF_IMAGE_PART>(P.img, tm, warp & 3, lane);
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
// Forward.  w on the tensor cores, the second axis (t, or h where h is shorter; n2 = 16 or 32 positions) in fp32 registers, and
// its fold on the tensor cores, too: a tile is 64 positions at i over the same 64 at n2 - 1 - i of the second axis, the operand
// [[M, M], [M, -M]] with M = I kron C_w.  Lanes 0..63 then hold the w transform of x[i] + x[n2 - 1 - i], lanes 64..127 that of the
// difference, and a thread makes the even or the odd coefficients of its position from n2 / 2 numbers a channel.  An item is
// 64 positions at all n2, 32 channels (n2 = 16, rows of 64 bytes) or 16 (n2 = 32, rows of 32): n2 / 2 tiles, 256 accumulator columns.
//   warp 0       TMA producer (ring of five batches: half an item, 32 KB)
//   warp 1       tcgen05.mma issuer; owns the tensor-memory allocation
//   warps 2..17  epilogue: four warps per 32 lanes, two or four coefficients each: 64 sums a thread, to which it adds the
//                accumulators as they come; a warp stages and sends its rows by itself.  (The four warps of 32 lanes share a
//                scheduler: when they shared the staging area, too, a quarter of the channels each, it stood still at every hand-over.)
// Every wait is bounded.
//
// n2 = 16: bound by HBM and, close behind, by the epilogue: six heads of 64K tokens alone 163 us, 0.9 GB at 5.6 TB/s, issue slots
// 62%.  n2 = 32: by its rows of 32 bytes and the epilogue: six heads of 32 x 64 x 64 tokens 365 us, 1.8 GB at 5.0 TB/s, issue slots
// 57% (75% and 384 us without packed FMA, which with n2 = 16 gain nothing: 724 -> 732 us for six heads of 64 x 16 x 64); stores of 32
// bytes from the registers 494.
// ff_dct2_tc.cu sends the intermediate through shared memory as a bf16 pair and multiplies the second axis with a 128 x 128
// operand of which 128 / n2 - 1 parts are zeros.  Layers with that launch / with this one, all else equal, in turn on one box (us,
// under the power limit): 24 heads of 64K tokens 2745 / 2528; all bands 3427 / 3309; 16 heads with head_dim 64 993 / 937; six heads of
// 16K 197 / 185, four of 8K 120 / 116, six of 64 x 16 x 64 765 / 730; n2 = 32: two samples of 24 heads of 32 x 64 x 64 10375 / 9998,
// 12 heads 3059 / 2984, eight with head_dim 64 1197 / 1171, eight of 32 x 64 x 32 979 / 970.  A line of 128 positions does not fit twice
// into the operand: those grids keep the two-axis launch.  Variants (n2 = 16, six heads of 64K): a quarter of the channels a thread, staged by four warps together,
// coefficients as constants of unrolled code 201 us (instruction cache), in a loop 177; packed FMA 181; without its stores that form
// took 155, without its FMA 163.
constexpr int FPOS = 64;                                   // positions of an item
template <int N2> struct Fold {
  static constexpr int C = 512 / N2;                       // channels of an item
  static constexpr int TILE_B = 2 * FPOS * C * 2, BATCH = 128 / C;       // 8 or 4 KB; tiles of a batch
  static constexpr int KPW = N2 / 8;                       // coefficients of an epilogue warp
  static constexpr int BOX_B = 32 * C * 2;                 // 32 positions at one coefficient, hi or lo
  static constexpr int KPS = N2 / 16;                      // coefficients staged at a time
  static constexpr int UNROLL = N2 == 32 ? BATCH : 1;      // (what leaves no register spilled)
};
constexpr size_t FOLD_IMAGE = 2 * FF_IMAGE_PART;           // hi and lo: the third parts of the first two images, which these grids leave unused
constexpr int F_NSLOT = 5, F_SLOT_B = 32 * 1024;           // ring: batches
constexpr int F_STAGE_B = 4 * 1024;                        // staging area of an epilogue warp

struct FoldParams {
  FFDims dm;
  const uint32_t* img;     // [[M, M], [M, -M]]: hi [128][64] cells, lo FF_IMAGE_CELLS behind it
  alignas(16) float mat[2][16][16];      // [parity][i][k / 2]: C[k][i] of the second axis
  int axis2;               // 0 = t, 1 = h
  int group, group_start;  // tensor-heads of the launch, the first one
  int nchunk, n3, lines;   // channel chunks; items along the remaining axis, w lines of an item (64 / W)
  double* clear;           // band energies to clear for the sums that follow (first launch of a routed forward), or NULL
  int* status;
};

struct FoldShared {
  uint64_t full[F_NSLOT], empty[F_NSLOT], acc_full[NACC], acc_empty[NACC];
  uint32_t tmem_base;
  int abort_flag;
};

// Descriptor of an MN-major operand stored as rows of C bf16 with the swizzle of that width, tiles one after the other along N.
template <int C>
__device__ __forceinline__ uint64_t smem_desc_rows(uint32_t smem_addr) {
  return (uint64_t)((smem_addr & 0x3FFFF) >> 4) | (uint64_t)(2 * FPOS * C * 2 >> 4) << 16 | (uint64_t)(8 * C * 2 >> 4) << 32 | (uint64_t)1 << 46 |
         (uint64_t)(C == 32 ? 4 : 6) << 61;
}
__device__ __forceinline__ void st_shared_v4(uint32_t addr, const uint32_t (&v)[4]) {
  asm volatile("st.shared.v4.b32 [%0], {%1, %2, %3, %4};" ::"r"(addr), "r"(v[0]), "r"(v[1]), "r"(v[2]), "r"(v[3]) : "memory");
}
__device__ __forceinline__ float2 fma2(float2 a, float2 b, float2 c) {
  float2 d;
  asm("fma.rn.f32x2 %0, %1, %2, %3;" : "=l"(*(uint64_t*)&d) : "l"(*(uint64_t*)&a), "l"(*(uint64_t*)&b), "l"(*(uint64_t*)&c));
  return d;
}
// map0..map2: Q, K, V; map_oh, map_ol: the pair of grids, box = 32 positions at one coefficient.
template <int N2>
__global__ void __launch_bounds__(THREADS, 1)
dct_fold_kernel(const __grid_constant__ CUtensorMap map0, const __grid_constant__ CUtensorMap map1,
                       const __grid_constant__ CUtensorMap map2, const __grid_constant__ CUtensorMap map_oh,
                       const __grid_constant__ CUtensorMap map_ol, const __grid_constant__ FoldParams P) {
  extern __shared__ uint8_t smem_raw[];
  uint8_t* smem = (uint8_t*)(((uintptr_t)smem_raw + 1023) & ~(uintptr_t)1023);
  const FFDims& dm = P.dm;
  using F = Fold<N2>;
  constexpr int FC = F::C;
  constexpr uint32_t COL_ACC = 128;
  uint8_t* sIn = smem;
  uint8_t* sStage = smem + F_NSLOT * F_SLOT_B;              // an area per epilogue warp
  FoldShared& sh = *(FoldShared*)(sStage + 4 * EPI * F_STAGE_B);
  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
  const int total = P.group * P.n3 * P.nchunk;

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
  if (warp >= 2 && warp < 6) matrix_to_tmem<FF_IMAGE_CELLS>(P.img, tm, warp & 3, lane);
  ff_pdl_wait();
  if (P.clear && blockIdx.x == 0) for (int i = threadIdx.x; i < dm.B * 3 * dm.d; i += THREADS) P.clear[i] = 0.0;
  tc_fence_before();
  __syncthreads();
  tc_fence_after();

  FF_CLOCK(t_all);
  // Item: chunk fastest (CTAs that run side by side read neighbouring pieces of the same rows), then the remaining axis, then the tensor-head.
  if (warp == 0) {
    if (lane == 0) {
      tma_prefetch_desc(&map0);
      unsigned n = 0;
      bool ok = true;
      for (int it = blockIdx.x; it < total && ok; it += gridDim.x) {
        const int chunk = it % P.nchunk, rest = it / P.nchunk, o0 = rest % P.n3 * P.lines, gi = rest / P.n3;
        const int th = P.group_start + gi, tensor = (th >= dm.BH) + (th >= 2 * dm.BH);
        const CUtensorMap* map = tensor == 0 ? &map0 : (tensor == 1 ? &map1 : &map2);
        for (int b = 0; b < 2 && ok; ++b, ++n) {
          const int slot = n % F_NSLOT;
          FF_CLOCK(tp);
          if (n >= (unsigned)F_NSLOT) ok = mbar_wait(&sh.empty[slot], ((n / F_NSLOT) - 1) & 1, abort_flag);
          FF_CLOCK_ADD(true, 16, tp);
          if (!ok) break;
          // (debug build) the boxes lie inside the grid; a refused batch ends in the bounded wait of its consumer
          if (!FF_DBG_OK((chunk + 1) * FC <= dm.d && o0 + P.lines <= (P.axis2 ? dm.T : dm.H) && N2 <= (P.axis2 ? dm.H : dm.T) && th < 3 * dm.BH,
                         P.status, 7)) continue;
          uint8_t* dst = sIn + slot * F_SLOT_B;
          mbar_arrive_expect_tx(&sh.full[slot], F_SLOT_B);
#pragma unroll
          for (int k = 0; k < F::BATCH; ++k) {
            const int i = b * F::BATCH + k, j = N2 - 1 - i;
            tma_load_5d(dst + k * F::TILE_B, map, &sh.full[slot], chunk * FC, 0, P.axis2 ? i : o0, P.axis2 ? o0 : i, th - tensor * dm.BH);
            tma_load_5d(dst + k * F::TILE_B + F::TILE_B / 2, map, &sh.full[slot], chunk * FC, 0, P.axis2 ? j : o0, P.axis2 ? o0 : j, th - tensor * dm.BH);
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
        const uint64_t x = smem_desc_rows<FC>(in_base + slot * F_SLOT_B);
        const uint32_t d_tm = tm + COL_ACC + ab * 128;
#pragma unroll
        for (int ks = 0; ks < ROWS / 16; ++ks) {           // (16 rows of K)
          umma_ts(d_tm, tm + ks * 8, x + (uint64_t)(ks * FC * 2), idesc, ks > 0 ? 1u : 0u);
          umma_ts(d_tm, tm + 64 + ks * 8, x + (uint64_t)(ks * FC * 2), idesc, 1u);
        }
        umma_commit(&sh.empty[slot]);
        umma_commit(&sh.acc_full[ab]);
      }
    }
  } else {
    const int quarter = warp & 3, part = (warp - 2) >> 2;  // TMEM lanes; which of the lanes' coefficients
    const uint32_t lane_addr = (uint32_t)(quarter * 32) << 16;
    const int parity = __shfl_sync(0xffffffffu, quarter >> 1, 0), k0 = __shfl_sync(0xffffffffu, F::KPW * part, 0);
    const uint32_t stage = smem_u32(sStage) + (warp - 2) * F_STAGE_B;
    unsigned nb = 0;
    bool ok = true;
    for (int it = blockIdx.x; it < total && ok; it += gridDim.x) {
      float y[F::KPW][FC] = {};
#pragma unroll 1
      for (int b = 0; b < 2; ++b, ++nb) {
        const int ab = nb % NACC;
        FF_CLOCK(te);
        ok = mbar_wait_warp(&sh.acc_full[ab], (nb / NACC) & 1, abort_flag);
        FF_CLOCK_ADD(threadIdx.x == 64, 19, te);
        if (!ok) break;
        tc_fence_after();
#pragma unroll F::UNROLL
        for (int i = 0; i < F::BATCH; ++i) {
          float m[F::KPW];
          const float* row = P.mat[parity][b * F::BATCH + i] + k0;
          if (F::KPW == 2) { const float2 v = *(const float2*)row; m[0] = v.x; m[1] = v.y; }
          else { const float4 v = *(const float4*)row; m[0] = v.x; m[1] = v.y; m[2] = v.z; m[3] = v.w; }
#pragma unroll
          for (int h = 0; h < FC / 16; ++h) {
            uint32_t x[16];
            tmem_ld16(tm + lane_addr + COL_ACC + ab * 128 + i * FC + h * 16, x);
            tmem_wait_ld();
#pragma unroll
            for (int j = 0; j < F::KPW; ++j)
#pragma unroll
              for (int c = 0; c < 16; c += 2) {
                if (N2 == 32) {
                  const float2 v = fma2(make_float2(m[j], m[j]), make_float2(__uint_as_float(x[c]), __uint_as_float(x[c + 1])),
                                        make_float2(y[j][h * 16 + c], y[j][h * 16 + c + 1]));
                  y[j][h * 16 + c] = v.x; y[j][h * 16 + c + 1] = v.y;
                } else {
                  y[j][h * 16 + c] = fmaf(m[j], __uint_as_float(x[c]), y[j][h * 16 + c]);
                  y[j][h * 16 + c + 1] = fmaf(m[j], __uint_as_float(x[c + 1]), y[j][h * 16 + c + 1]);
                }
              }
          }
        }
        tc_fence_before();
        mbar_arrive(&sh.acc_empty[ab]);
      }
      if (!ok) break;
      FF_CLOCK(tw);
#pragma unroll
      for (int j0 = 0; j0 < F::KPW; j0 += F::KPS) {
        FF_CLOCK(tb);
        if (lane == 0) bulk_wait_read0();                  // the warp's previous stores have read the area
        __syncwarp();
        FF_CLOCK_ADD(threadIdx.x == 64, 20, tb);
#pragma unroll
        for (int j = j0; j < j0 + F::KPS; ++j) {
          const uint32_t box = stage + (j - j0) * 2 * F::BOX_B;
#pragma unroll
          for (int p = 0; p < FC / 8; ++p) {               // 16-byte pieces of the row, under the swizzle
            uint32_t hi[4], lo[4];
#pragma unroll
            for (int c = 0; c < 4; ++c) {
              const float a = y[j][8 * p + 2 * c], e = y[j][8 * p + 2 * c + 1];
              hi[c] = bf16_pair(__float_as_uint(a), __float_as_uint(e));
              lo[c] = bf16_pair(__float_as_uint(a - __uint_as_float(hi[c] << 16)), __float_as_uint(e - __uint_as_float(hi[c] & 0xffff0000u)));
            }
            const uint32_t at = box + lane * FC * 2 + ((FC == 32 ? p ^ ((lane >> 1) & 3) : p ^ ((lane >> 2) & 1)) << 4);
            st_shared_v4(at, hi);
            st_shared_v4(at + F::BOX_B, lo);
          }
        }
        fence_proxy_async();
        __syncwarp();
        if (lane == 0) {
          const int chunk = it % P.nchunk, rest = it / P.nchunk, gi = rest / P.n3;
          const int p0 = (quarter & 1) * 32, w0 = p0 % dm.W, o0 = rest % P.n3 * P.lines + p0 / dm.W;      // the warp's first position
#pragma unroll
          for (int j = j0; j < j0 + F::KPS; ++j) {
            const uint8_t* box = sStage + (warp - 2) * F_STAGE_B + (j - j0) * 2 * F::BOX_B;
            const int k = 2 * (k0 + j) + parity, ch = P.axis2 ? k : o0, ct = P.axis2 ? o0 : k;
            // (debug build) the box lies inside the grid
            if (FF_DBG_OK((chunk + 1) * FC <= dm.d && w0 + (dm.W < 32 ? dm.W : 32) <= dm.W && ch < dm.H && ct < dm.T && gi < P.group, P.status, 7)) {
              tma_store_5d(box, &map_oh, chunk * FC, w0, ch, ct, gi);
              tma_store_5d(box + F::BOX_B, &map_ol, chunk * FC, w0, ch, ct, gi);
            }
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

int fold_length(const FFDims& dm, int axis2) { return axis2 ? dm.H : dm.T; }

// Map over a [slices][T][H][W][d] grid: a chunk's channels of 64 positions (load) or 32 (store) at one position of the second axis.
bool fold_map(ff_plan* p, CUtensorMap* map, const void* base, int slices, bool store) {
  const FFDims& dm = p->dm;
  return p->maps.get(map, base, store ? 51 : 50, slices, [&] {
    const cuuint64_t ch = (cuuint64_t)dm.d, W = (cuuint64_t)dm.W;
    const cuuint64_t dims[5] = {ch, W, (cuuint64_t)dm.H, (cuuint64_t)dm.T, (cuuint64_t)slices};
    const cuuint64_t strides[4] = {ch * 2, W * ch * 2, dm.H * W * ch * 2, (cuuint64_t)dm.N * ch * 2};
    const cuuint32_t C = (cuuint32_t)(512 / fold_length(dm, p->dct2_axis2)), positions = store ? 32 : FPOS, w = (cuuint32_t)dm.W < positions ? (cuuint32_t)dm.W : positions;
    cuuint32_t box[5] = {C, w, 1, 1, 1};
    box[p->dct2_axis2 ? 3 : 2] = positions / w;
    return ff_encode_map(map, CU_TENSOR_MAP_DATA_TYPE_BFLOAT16, 5, base, dims, strides, box, C == 32 ? CU_TENSOR_MAP_SWIZZLE_64B : CU_TENSOR_MAP_SWIZZLE_32B,
                         store ? CU_TENSOR_MAP_L2_PROMOTION_NONE : CU_TENSOR_MAP_L2_PROMOTION_L2_256B);
  });
}
constexpr size_t F_SMEM = 1024 + (size_t)F_NSLOT * F_SLOT_B + 4 * EPI * F_STAGE_B + sizeof(FoldShared);

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
  if (e != cudaSuccess) return e;
  const cudaError_t f = cudaFuncSetAttribute(dct_fold_kernel<16>, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)F_SMEM);
  return f != cudaSuccess ? f : cudaFuncSetAttribute(dct_fold_kernel<32>, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)F_SMEM);
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

// Where it takes the place of the two-axis launch.  With 32 positions from 20 items an SM on, all tensor-heads together: layers, us,
// with that launch / with this one, long runs: four heads of 32 x 64 x 32 tokens (20) 513 / 512, of 32 x 64 x 64 (41) 1050 / 1033, six
// (62) 1529 / 1498; of 32 x 32 x 16 (5) 170 / 179.  In bursts of some ms after a pause, at full clock, the line lies higher: four of
// 32 x 64 x 64 938 / 955, six 1949 / 1962 (all bands), twelve (124) 2735 / 2720.
bool ffk_dct_fold_supported(const ff_plan* p) {
  const FFDims& dm = p->dm;
  const int n2 = fold_length(dm, p->dct2_axis2);
  if (!p->dct2_ok || ff_fp32_grid(dm) || p->cfg.transform != FF_TRANSFORM_DCT || dm.W > FPOS || (n2 != 16 && n2 != 32)) return false;
  return n2 == 16 || 3LL * dm.BH * (dm.N / n2 / FPOS) * (dm.d / Fold<32>::C) >= 20LL * p->sm_count;
}

// Forward: Q, K, V of tensor-heads [g0, g0 + g) -> transform along w and the second axis -> hi/lo grids.
cudaError_t ffk_dct_fold_forward(ff_plan* p, const void* Q, const void* K, const void* V, int g0, int g, void* out_hi, void* out_lo,
                                 bool clear_energy, cudaStream_t st) {
  const FFDims& dm = p->dm;
  CUtensorMap mq, mk, mv, oh, ol;
  if (!fold_map(p, &mq, Q, dm.BH, false) || !fold_map(p, &mk, K, dm.BH, false) || !fold_map(p, &mv, V, dm.BH, false) ||
      !fold_map(p, &oh, out_hi, p->dct_group, true) || !fold_map(p, &ol, out_lo, p->dct_group, true))
    return cudaErrorInvalidValue;
  FoldParams P{};
  const int n2 = fold_length(dm, p->dct2_axis2);
  P.dm = dm; P.status = p->buf.status;
  P.img = p->dct2_images + FOLD_IMAGE;
  for (int k = 0; k < n2; ++k) for (int i = 0; i < n2 / 2; ++i) P.mat[k & 1][i][k >> 1] = p->fold_mat[k * (n2 / 2) + i];
  P.axis2 = p->dct2_axis2; P.group = g; P.group_start = g0;
  P.nchunk = dm.d / (512 / n2); P.lines = FPOS / dm.W; P.n3 = (P.axis2 ? dm.T : dm.H) / P.lines;
  P.clear = clear_energy ? p->buf.energy : nullptr;
  const int items = g * P.n3 * P.nchunk;
  const cudaError_t e = ff_launch(n2 == 16 ? dct_fold_kernel<16> : dct_fold_kernel<32>, dim3((unsigned)(items < p->sm_count ? items : p->sm_count)),
                                  dim3(THREADS), F_SMEM, st, mq, mk, mv, oh, ol, P);
  if (e == cudaSuccess) p->launches += 1;
  return e;
}

// Its matrix as the tensor-memory A operand, hi and lo parts: [[M, M], [M, -M]], M = I kron C_w over 64 positions.
bool ffk_dct_fold_build_image(ff_plan* p, const float* mat) {
  const int n = p->dm.W;
  std::vector<uint32_t> img(2 * FF_IMAGE_PART);
  for (int a = 0; a < n; ++a)
    for (int b = 0; b < n; b += 2) {
      float v[2] = {mat[a * n + b], mat[a * n + b + 1]};
      for (int part = 0; part < 2; ++part) {
        const __nv_bfloat162 h = __floats2bfloat162_rn(v[0], v[1]);
        const uint32_t cell = *(const uint32_t*)&h;
        v[0] -= __low2float(h); v[1] -= __high2float(h);
        for (int l = 0; l < ROWS; l += n)                // the lines of the rows, and the same line in both halves of the columns
          for (int r = l % FPOS; r < ROWS; r += FPOS)
            img[part * FF_IMAGE_PART + (size_t)(l + a) * 64 + ((r + b) >> 1)] = l >= FPOS && r >= FPOS ? cell ^ 0x80008000u : cell;
      }
    }
  const size_t row = FF_IMAGE_PART * sizeof(uint32_t);
  return cudaMemcpy2D(p->dct2_images + FOLD_IMAGE, FF_IMAGE_CELLS * sizeof(uint32_t), img.data(), row, row, 2, cudaMemcpyHostToDevice) == cudaSuccess;
}

FF_CLOCKS_READ(transform_t16)
