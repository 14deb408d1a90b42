// Cross-band residual exchange + recombination on the tensor cores ("Cross-band residual
// exchange", "Reconstruction"), bf16 storage, head_dim 128 or 64 (template parameter XD), for the
// mid and high bands:
//     Y^[p] = Y[p] + softmax(Y[p] Z^T / sqrt(d)) Z,   Z = the 2m summary tokens of the other two bands
// written to the coefficient grid at the position of band rank p (a table built at plan creation).
//
// A CTA owns a contiguous run of (head, band, 128-rank tile) items, so the summary tokens of a head
// are loaded only a few times per CTA.  Two CTAs share an SM (256 tensor-memory columns each).  Per tile:
//   TMA     the 128 band tokens (operator output where the head's mask has the band, V~ otherwise)
//   MMA 1   S[128 x 3m] = Y Z^T against all 3m summaries of the head; with up to 64 keys into one of two buffers, so
//           that the next tile's scores are computed during this tile's softmax
//   softmax one token per thread (row = TMEM lane), 16 keys at a time; chunks that are the band's own summaries are
//           skipped; P (unnormalised) goes back to TMEM as bf16 hi + lo over the 16 scores it comes from, the row sum
//           to the store warps
//   MMA 2   D[128 x 128] = P Z  (A = P from tensor memory, B = the same Z image read MN-major)
//   store   Y + D / row sum in the form the inverse passes read: three bytes (the value rounded to 24 bits: a grid of its
//           upper 16 bits and a grid of the next byte), or fp32 (template parameter F32).  A warp has 32 tokens, one per
//           lane; it turns 32 channels of them in shared memory, so that four lanes write 64 (hi) and 32 (lo) contiguous
//           bytes of a token.  With more than 64 keys a second token tile no longer fits: the tile then goes back to the
//           producer as soon as the scores are done, the update is turned as fp32 and the tokens are read again from
//           global memory, four lanes 64 contiguous bytes.
// Z and P are split into bf16 hi + lo parts (Y is exact bf16), so the logits and the update carry
// about 16 bits: the summary logits of a band with large low-frequency content reach O(100).  (Grids whose values are fp32
// up to here had an fp32 exchange before: the output's error against fp64 is the same to 2e-5 of itself, 1.660e-3.)
// The low band (fp32, a few hundred tokens) has a kernel of its own (ff_summary.cu).
//
// Bound by the store warps (5800 of 9700 cycles a tile; the rest they wait, the softmax takes 1500): 64K tokens, 24 heads
// 248 us = 4.1 TB/s; without the row-scattered stores to global memory 181 us, without all of the store warps' work 105.
// 1M tokens (96 keys): 2.2 -> 1.55 ms per 8 heads since the residual is read four lanes to a token (it was one lane to a
// token) and own-band chunks are skipped.
#include <cuda.h>

#include "ff_clocks.cuh"
#include "ff_internal.h"
#include "ff_sm100.cuh"
#include "ff_three_byte.cuh"

using namespace sm100;

namespace {

constexpr int XT = 128;                 // tokens per tile
constexpr int XD_MAX = 128;             // largest head_dim; the shared-memory tiles are sized for it
constexpr int X_TILE_BYTES = XT * XD_MAX * 2;
constexpr int X_HALF = X_TILE_BYTES / 2;
constexpr int X_THREADS = 320;           // TMA warp, MMA warp, 4 softmax warps, 4 store warps

struct XParams {
  FFDims dm;
  const uint8_t* alloc;
  const uint8_t* zimg;        // [BH] operand images of the heads' summaries (hi, then lo; written by the summary launch)
  const int* pos_mid;         // [N_mid]  flat coefficient index of each band rank
  const int* pos_high;        // [N_high]
  __nv_bfloat16* grid_hi;     // [g][N][d]: upper 16 bits of the value rounded to 24 bits
  uint8_t* grid_lo;           // [g][N][d]: the next 8 bits (the three-byte form the inverse passes read)
  float* grid_f32;            // [g][N][d] instead of the two (template parameter F32: grids whose inverse passes read fp32)
  int h0, g;                  // heads [h0, h0+g)
  int nkeys;                  // 3m rounded up to a multiple of 16
  int ybufs;                  // token-tile buffers in shared memory (1 or 2)
  const __nv_bfloat16* src[4];   // y_mid, v~_mid, y_high, v~_high: bases of the buffers the four maps cover
  int* status;
};

// per store warp: 32 channels of 32 tokens, 64 bytes of hi and 32 of lo each, or in fp32
__host__ __device__ constexpr int x_stage_bytes(bool reread) { return reread ? 32 * 128 : 32 * 96; }

struct XShared {
  uint64_t y_full[2], y_empty[2], z_ready, z_empty, s_full[2], p_full[2], d_full, d_empty;
  uint32_t tmem_base;
  int abort_flag;
  // keys a token attends to, as bit masks per band (mid, high) and 16-key chunk: the 3m summaries without the token's own
  // band's and without those of an empty mid band
  uint32_t keys[2][6];
  float inv[4][XT];          // 1 / row sum of a tile (the softmax may be two tiles ahead of the store warps)
};

struct XItem { int bh, band, tile; };

__device__ __forceinline__ void bulk_load(void* smem_dst, const void* src, uint32_t bytes, uint64_t* bar) {
  asm volatile("cp.async.bulk.shared::cluster.global.mbarrier::complete_tx::bytes [%0], [%1], %2, [%3];"
               ::"r"(smem_u32(smem_dst)), "l"((uint64_t)src), "r"(bytes), "r"(smem_u32(bar))
               : "memory");
}

__device__ __forceinline__ XItem x_decode(int h0, int it, int tm, int th) {
  XItem x;
  const int per = tm + th, rem = it % per;
  x.bh = h0 + it / per;
  x.band = rem < tm ? 1 : 2;
  x.tile = rem < tm ? rem : rem - tm;
  return x;
}
__device__ __forceinline__ void x_next(XItem& x, int tm, int th) {
  if (++x.tile == (x.band == 1 ? tm : th)) {
    x.tile = 0;
    if (x.band == 1) x.band = 2;
    else { ++x.bh; x.band = tm > 0 ? 1 : 2; }
  }
}

// NK = 16-key chunks of the score row (3m rounded up).
template <int NK, int XD, bool F32>
__global__ void __launch_bounds__(X_THREADS, 2)
exchange_tc_kernel(const __grid_constant__ CUtensorMap map_y_mid, const __grid_constant__ CUtensorMap map_v_mid,
                   const __grid_constant__ CUtensorMap map_y_high, const __grid_constant__ CUtensorMap map_v_high,
                   const XParams P) {
  extern __shared__ uint8_t smem_raw[];
  uint8_t* smem = (uint8_t*)(((uintptr_t)smem_raw + 1023) & ~(uintptr_t)1023);
  uint8_t* sY = smem;                                    // ybufs x 32 KB
  uint8_t* sZhi = smem + P.ybufs * X_TILE_BYTES;         // [2 halves][nkeys rows][128 B]
  uint8_t* sZlo = sZhi + 2 * P.nkeys * 128;
  constexpr bool REREAD = NK > 4;                         // one token tile: the residual comes from global memory
  uint8_t* sStage = sZlo + 2 * P.nkeys * 128;            // 4 x x_stage_bytes
  XShared& sh = *(XShared*)(sStage + 4 * x_stage_bytes(REREAD));
  const FFDims& dm = P.dm;
  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
  constexpr int nk = NK * 16, SB = NK <= 4 ? 2 : 1;      // keys; score buffers (64 columns apart)
  const int m = dm.m;
  const int tm_tiles = (int)((dm.Nmid + XT - 1) / XT), th_tiles = (int)((dm.Nhigh + XT - 1) / XT);
  const int total = P.g * (tm_tiles + th_tiles);
  const int chunk = (total + gridDim.x - 1) / gridDim.x;
  const int it0 = blockIdx.x * chunk;
  const int it1 = it0 + chunk < total ? it0 + chunk : total;

  if (threadIdx.x == 0) {
    for (int i = 0; i < 2; ++i) {
      mbar_init(&sh.y_full[i], 1); mbar_init(&sh.y_empty[i], REREAD ? 1 : 128); mbar_init(&sh.s_full[i], 1); mbar_init(&sh.p_full[i], 128);
    }
    mbar_init(&sh.z_ready, 1); mbar_init(&sh.z_empty, 1);
    mbar_init(&sh.d_full, 1); mbar_init(&sh.d_empty, 128);
    sh.abort_flag = 0;
    fence_mbar_init();
  }
  if (threadIdx.x >= 64 && threadIdx.x < 64 + 2 * NK) {
    const int band = (threadIdx.x - 64) / NK, c = (threadIdx.x - 64) % NK;
    uint32_t a = 0;
    for (int i = 0; i < 16; ++i) {
      const int j = c * 16 + i;
      const bool live = j < 3 * m && !(dm.Nmid == 0 && j >= m && j < 2 * m);
      if (live && (band == 0 ? j < m || j >= 2 * m : j < 2 * m)) a |= 1u << i;
    }
    sh.keys[band][c] = a;
  }
  if (warp == 1) { tmem_alloc(&sh.tmem_base, 256); tmem_relinquish(); }
  // The launch before this one is the low band's part of the exchange, which writes other positions of the same
  // grids: it let this launch start once the summaries were complete, and is waited for at the end only.
  ff_pdl_trigger();
  tc_fence_before();
  __syncthreads();
  tc_fence_after();
  const uint32_t tmem = sh.tmem_base;
  volatile int* abort_flag = &sh.abort_flag;
  // tensor-memory columns: S [0,128): one buffer of up to 96 columns or two of 64; P over the scores;  D [128,256)
  const int YB = P.ybufs;

  if (warp == 0) {
    if (lane == 0) {
      bool ok = true;
      int n = 0, prev_bh = -1, zc = 0;
      XItem x = x_decode(P.h0, it0, tm_tiles, th_tiles);
      for (int it = it0; it < it1 && ok; ++it, ++n, x_next(x, tm_tiles, th_tiles)) {
        const bool exec = P.alloc[x.bh] & (1 << x.band);
        const CUtensorMap* map = x.band == 1 ? (exec ? &map_y_mid : &map_v_mid) : (exec ? &map_y_high : &map_v_high);
        const int slice = exec ? x.bh : 2 * dm.BH + x.bh;
        const int slot = n % YB;
        FF_CLOCK(x0);
        if (n >= YB) ok = mbar_wait(&sh.y_empty[slot], ((n / YB) - 1) & 1, abort_flag);
        FF_CLOCK_ADD(lane == 0, 0, x0);
        if (!ok) break;
        mbar_arrive_expect_tx(&sh.y_full[slot], XT * XD * 2);
        tma_load_3d(sY + slot * X_TILE_BYTES, map, &sh.y_full[slot], 0, x.tile * XT, slice);
        if (XD == 128) tma_load_3d(sY + slot * X_TILE_BYTES + X_HALF, map, &sh.y_full[slot], 64, x.tile * XT, slice);
        if (x.bh != prev_bh) {
          // the head's summaries, once the MMAs of the previous head have read the old ones (staged and split by 128
          // threads of every CTA before: 48 rounds of 2-byte stores at the start of every head)
          prev_bh = x.bh;
          if (zc > 0) ok = mbar_wait(&sh.z_empty, (zc - 1) & 1, abort_flag);
          ++zc;
          if (!ok) break;
          const uint32_t bytes = 4u * (uint32_t)P.nkeys * 128u;
          mbar_arrive_expect_tx(&sh.z_ready, bytes);
          bulk_load(sZhi, P.zimg + (size_t)x.bh * bytes, bytes, &sh.z_ready);
        }
      }
    }
  } else if (warp == 1) {
    {
      const uint32_t idesc1 = idesc_bf16_f32(XT, nk, false, false);
      const uint32_t idesc2 = idesc_bf16_f32(XT, XD, false, true);
      // operand descriptors, once (assembling them for every instruction is slower than the instruction): token tiles, Z
      // as the K-major and as the MN-major operand (halves of 64 channels nk * 128 bytes apart), its lo image behind
      const uint64_t y_desc = smem_desc_sw128(smem_u32(sY), 16, 1024), zk_desc = smem_desc_sw128(smem_u32(sZhi), 16, 1024);
      const uint64_t zmn_desc = smem_desc_sw128(smem_u32(sZhi), nk * 128, 1024), zlo_step = (uint64_t)(2 * nk * 128 >> 4);
      bool ok = true;
      int prev_bh = -1, zc = 0;
      // S = Y (Zhi + Zlo)^T of the CTA's tile n, K = head_dim
      auto scores = [&](int n, const XItem& x) -> bool {
        if (x.bh != prev_bh) {                            // the head's summaries have arrived
          FF_CLOCK(x4);
          if (!mbar_wait_warp(&sh.z_ready, zc & 1, abort_flag)) return false;
          FF_CLOCK_ADD(lane == 0, 4, x4);
          ++zc; prev_bh = x.bh;
        }
        const int slot = n % YB;
        FF_CLOCK(x1);
        if (!mbar_wait_warp(&sh.y_full[slot], (n / YB) & 1, abort_flag)) return false;
        FF_CLOCK_ADD(lane == 0, 1, x1);
        tc_fence_after();
        const uint64_t y = y_desc + (uint64_t)(slot * (X_TILE_BYTES >> 4));
        const uint32_t s_tm = tmem + (SB == 2 ? (n & 1) * 64 : 0);
#pragma unroll
        for (int k = 0; k < XD / 16; ++k) {
          const uint64_t a = y + (uint64_t)(((k >> 2) * X_HALF + (k & 3) * 32) >> 4);
          const uint64_t zo = (uint64_t)(((k >> 2) * nk * 128 + (k & 3) * 32) >> 4);
          umma_ss(s_tm, a, zk_desc + zo, idesc1, k > 0 ? 1u : 0u);
          umma_ss(s_tm, a, zk_desc + zlo_step + zo, idesc1, 1u);
        }
        umma_commit(&sh.s_full[n & 1]);
        if (REREAD) umma_commit(&sh.y_empty[slot]);       // the tile has been read
        return true;
      };
      XItem x = x_decode(P.h0, it0, tm_tiles, th_tiles);
      if (it0 < it1) ok = scores(0, x);
      for (int it = it0, n = 0; it < it1 && ok; ++it, ++n) {
        // the next tile's scores ahead of this tile's update: into the other buffer, and against the same summaries
        const bool more = it + 1 < it1;
        XItem next = x;
        x_next(next, tm_tiles, th_tiles);
        const bool ahead = SB == 2 && more && next.bh == x.bh;
        if (ahead) ok = scores(n + 1, next);
        FF_CLOCK(x2);
        if (ok) ok = mbar_wait_warp(&sh.p_full[n & 1], (n >> 1) & 1, abort_flag);
        FF_CLOCK_ADD(lane == 0, 2, x2);
        FF_CLOCK(x3);
        if (ok && n >= 1) ok = mbar_wait_warp(&sh.d_empty, (n - 1) & 1, abort_flag);
        FF_CLOCK_ADD(lane == 0, 3, x3);
        if (!ok) break;
        tc_fence_after();
        const uint32_t p_tm = tmem + (SB == 2 ? (n & 1) * 64 : 0);
        uint32_t acc = 0;
#pragma unroll
        for (int k = 0; k < NK; ++k) {                    // D = (Phi + Plo) (Zhi + Zlo) without lo*lo, K = keys
          if (sh.keys[x.band - 1][k] == 0) continue;
          const uint64_t bh_ = zmn_desc + (uint64_t)(k * (2048 >> 4));
          umma_ts(tmem + 128, p_tm + k * 16, bh_, idesc2, acc);
          umma_ts(tmem + 128, p_tm + k * 16, bh_ + zlo_step, idesc2, 1u);
          umma_ts(tmem + 128, p_tm + k * 16 + 8, bh_, idesc2, 1u);
          acc = 1;
        }
        umma_commit(&sh.d_full);
        if (more && next.bh != x.bh) umma_commit(&sh.z_empty);
        if (more && !ahead) ok = scores(n + 1, next);
        x = next;
      }
    }
  } else if (warp < 6) {
    // ------------------------------------------------------------------ softmax warps
    const int quarter = warp & 3;
    const int row = quarter * 32 + lane;
    const uint32_t lane_addr = (uint32_t)(quarter * 32) << 16;
    const float sl2 = rsqrtf((float)XD) * 1.4426950408889634f;
    bool ok = true;
    int n = 0;
    XItem x = x_decode(P.h0, it0, tm_tiles, th_tiles);
    for (int it = it0; it < it1 && ok; ++it, ++n, x_next(x, tm_tiles, th_tiles)) {
      // ---- softmax over the 2m summaries of the other bands
      FF_CLOCK(x6);
      ok = __all_sync(0xffffffffu, mbar_wait(&sh.s_full[n & 1], (n >> 1) & 1, abort_flag));
      FF_CLOCK_ADD(row == 0, 6, x6);
      if (!ok) break;
      FF_CLOCK(x7);
      tc_fence_after();
      const uint32_t s_tm = tmem + lane_addr + (SB == 2 ? (n & 1) * 64 : 0);
      const uint32_t* masks = sh.keys[x.band - 1];
      // first sweep: the row maximum
      float mx0 = -INFINITY, mx1 = -INFINITY;
#pragma unroll 1
      for (int c = 0; c < NK; ++c) {
        const uint32_t keys = masks[c];
        if (keys == 0) continue;
        uint32_t r[16];
        tmem_ld16(s_tm + c * 16, r);
        tmem_wait_ld();
        if (keys == 0xffffu) {
#pragma unroll
          for (int i = 0; i < 16; i += 4) {
            mx0 = max3f(mx0, __uint_as_float(r[i]), __uint_as_float(r[i + 1]));
            mx1 = max3f(mx1, __uint_as_float(r[i + 2]), __uint_as_float(r[i + 3]));
          }
        } else {
#pragma unroll
          for (int i = 0; i < 16; ++i)
            if (keys & (1u << i)) mx0 = fmaxf(mx0, __uint_as_float(r[i]));
        }
      }
      const float mb = fmaxf(mx0, mx1) * sl2;
      const float2 sl22 = make_float2(sl2, sl2), nmb2 = make_float2(-mb, -mb), minus = make_float2(-1.f, -1.f);
      // second sweep: exponentials and their sum, P (unnormalised, bf16 hi + lo) over the chunk's own scores
      float2 den = make_float2(0.f, 0.f);
#pragma unroll 1
      for (int c = 0; c < NK; ++c) {
        const uint32_t keys = masks[c];
        if (keys == 0) continue;
        uint32_t r[16], ph[8], pl[8];
        tmem_ld16(s_tm + c * 16, r);
        tmem_wait_ld();
        if (keys != 0xffffu) {
#pragma unroll
          for (int i = 0; i < 16; ++i)
            if (!(keys & (1u << i))) r[i] = 0xff800000u;       // (-inf: exponential 0)
        }
#pragma unroll
        for (int i = 0; i < 8; ++i) {
          const float2 arg = __ffma2_rn(make_float2(__uint_as_float(r[2 * i]), __uint_as_float(r[2 * i + 1])), sl22, nmb2);
          const float2 p = make_float2(ex2(arg.x), ex2(arg.y));
          den = __fadd2_rn(den, p);
          const __nv_bfloat162 h2 = __floats2bfloat162_rn(p.x, p.y);
          ph[i] = *(const uint32_t*)&h2;
          const float2 l = __ffma2_rn(make_float2(__uint_as_float(ph[i] << 16), __uint_as_float(ph[i] & 0xffff0000u)), minus, p);
          const __nv_bfloat162 l2 = __floats2bfloat162_rn(l.x, l.y);
          pl[i] = *(const uint32_t*)&l2;
        }
        tmem_st8(s_tm + c * 16, ph);
        tmem_st8(s_tm + c * 16 + 8, pl);
      }
      sh.inv[n & 3][row] = 1.f / (den.x + den.y);
      tmem_wait_st();
      tc_fence_before();
      mbar_arrive(&sh.p_full[n & 1]);
      FF_CLOCK_ADD(row == 0, 7, x7);
    }
  } else {
    // ------------------------------------------------------------------ store warps
    const int quarter = warp & 3;                              // 32 tokens of the tile
    const uint32_t lane_addr = (uint32_t)(quarter * 32) << 16;
    uint8_t* st = sStage + quarter * x_stage_bytes(REREAD);
    bool ok = true;
    int n = 0;
    XItem x = x_decode(P.h0, it0, tm_tiles, th_tiles);
    for (int it = it0; it < it1 && ok; ++it, ++n, x_next(x, tm_tiles, th_tiles)) {
      const long long n_band = x.band == 1 ? dm.Nmid : dm.Nhigh;
      // ---- where the lane's tokens (8 i + r8 of the warp's) come from and go: looked up before the wait
      FF_CLOCK(x14);
      const int* pos = x.band == 1 ? P.pos_mid : P.pos_high;
      if (!REREAD) {
        const long long p = (long long)x.tile * XT + quarter * 32 + lane;
        int f = p < n_band ? __ldg(pos + p) : -1;
        if (f >= 0 && !FF_DBG_OK(f < dm.N && x.bh >= P.h0 && x.bh < P.h0 + P.g, P.status, 3)) f = -1;   // (debug build)
        f *= XD;                                           // element offset of the token's row in the head's grid, or < 0
        // the rows this lane stores pieces of: 8 i + lane / 4
        int out[4];
#pragma unroll
        for (int i = 0; i < 4; ++i) out[i] = __shfl_sync(0xffffffffu, f, 8 * i + (lane >> 2));
        const size_t obase = (size_t)(x.bh - P.h0) * dm.N * XD;
        __nv_bfloat16* const grid_hi = P.grid_hi + obase + (lane & 3) * 8;
        uint8_t* const grid_lo = P.grid_lo + obase + (lane & 3) * 8;
        float* const grid_f32 = P.grid_f32 + obase + (lane & 3) * 4;
        const int slot = n % YB, row = quarter * 32 + lane;
        const uint8_t* yrow = sY + slot * X_TILE_BYTES + row * 128;
        FF_CLOCK_ADD(threadIdx.x == 192, 14, x14);
        FF_CLOCK(x9);
        ok = __all_sync(0xffffffffu, mbar_wait(&sh.d_full, n & 1, abort_flag));
        FF_CLOCK_ADD(threadIdx.x == 192, 9, x9);
        if (!ok) break;
        FF_CLOCK(x10);
        tc_fence_after();
        const float2 s2 = make_float2(sh.inv[n & 3][row], sh.inv[n & 3][row]);
#pragma unroll 4
        for (int q = 0; q < XD / 32; ++q) {                // 32 channels
          uint32_t r[32];
          tmem_ld32(tmem + lane_addr + 128 + q * 32, r);
          tmem_wait_ld();
          if (q == XD / 32 - 1) {                          // D has been read
            tc_fence_before();
            mbar_arrive(&sh.d_empty);
          }
          if (F32) {
            // 16 channels at a time: four lanes store 64 bytes of a token
#pragma unroll
            for (int half = 0; half < 2; ++half) {
#pragma unroll
              for (int v = 0; v < 2; ++v) {                // 8 channels: 16 bytes of the swizzled token row
                const int c = q * 4 + half * 2 + v, r0 = half * 16 + v * 8;
                const uint4 yv = *(const uint4*)(yrow + (c >> 3) * X_HALF + (((c & 7) ^ (row & 7)) << 4));
                const uint32_t yw[4] = {yv.x, yv.y, yv.z, yv.w};
                float2 w[4];
#pragma unroll
                for (int k = 0; k < 4; ++k)
                  w[k] = __ffma2_rn(make_float2(__uint_as_float(r[r0 + 2 * k]), __uint_as_float(r[r0 + 2 * k + 1])), s2,
                                    make_float2(__uint_as_float(yw[k] << 16), __uint_as_float(yw[k] & 0xffff0000u)));
                *(float4*)(st + lane * 64 + (((2 * v) ^ ((lane >> 1) & 3)) << 4)) = make_float4(w[0].x, w[0].y, w[1].x, w[1].y);
                *(float4*)(st + lane * 64 + (((2 * v + 1) ^ ((lane >> 1) & 3)) << 4)) = make_float4(w[2].x, w[2].y, w[3].x, w[3].y);
              }
              if (q == XD / 32 - 1 && half == 1) mbar_arrive(&sh.y_empty[slot]);
              __syncwarp();
#pragma unroll
              for (int i = 0; i < 4; ++i) {
                const int t = 8 * i + (lane >> 2), piece = lane & 3;
                if (out[i] >= 0) *(float4*)(grid_f32 + out[i] + q * 32 + half * 16) = *(const float4*)(st + t * 64 + ((piece ^ ((t >> 1) & 3)) << 4));
              }
              __syncwarp();
            }
          } else {
#pragma unroll
            for (int v = 0; v < 4; ++v) {                    // 8 channels: 16 bytes of the swizzled token row
              const int c = q * 4 + v;
              const uint4 yv = *(const uint4*)(yrow + (c >> 3) * X_HALF + (((c & 7) ^ (row & 7)) << 4));
              const uint32_t yw[4] = {yv.x, yv.y, yv.z, yv.w};
              uint32_t hi[4], u[8];
#pragma unroll
              for (int k = 0; k < 4; ++k) {
                const float2 d = make_float2(__uint_as_float(r[8 * v + 2 * k]), __uint_as_float(r[8 * v + 2 * k + 1]));
                const float2 w = __ffma2_rn(d, s2, make_float2(__uint_as_float(yw[k] << 16), __uint_as_float(yw[k] & 0xffff0000u)));
                u[2 * k] = __float_as_uint(w.x) + FF_HALF24;
                u[2 * k + 1] = __float_as_uint(w.y) + FF_HALF24;
                hi[k] = ff_hi2(u[2 * k], u[2 * k + 1]);
              }
              *(uint4*)(st + lane * 64 + ((v ^ ((lane >> 1) & 3)) << 4)) = make_uint4(hi[0], hi[1], hi[2], hi[3]);
              // (lo: 32 bytes per row, 8-byte pieces XOR-swizzled with row / 4)
              *(uint2*)(st + 2048 + lane * 32 + ((v ^ ((lane >> 2) & 3)) << 3)) =
                  make_uint2(ff_lo4(u[0], u[1], u[2], u[3]), ff_lo4(u[4], u[5], u[6], u[7]));
            }
            // a NaN in the token or in a summary is in every score of the row: all of it is NaN (a branch, because a register
            // for the half that is added above spills)
            if (s2.x != s2.x)
              for (int v = 0; v < 4; ++v) *(uint4*)(st + lane * 64 + v * 16) = make_uint4(0x7fff7fff, 0x7fff7fff, 0x7fff7fff, 0x7fff7fff);
            if (q == XD / 32 - 1) mbar_arrive(&sh.y_empty[slot]);
            __syncwarp();
#pragma unroll
            for (int i = 0; i < 4; ++i) {
              const int t = 8 * i + (lane >> 2), piece = lane & 3;
              if (out[i] >= 0) {
                *(uint4*)(grid_hi + out[i] + q * 32) = *(const uint4*)(st + t * 64 + ((piece ^ ((t >> 1) & 3)) << 4));
                *(uint2*)(grid_lo + out[i] + q * 32) = *(const uint2*)(st + 2048 + t * 32 + ((piece ^ ((t >> 2) & 3)) << 3));
              }
            }
            __syncwarp();
          }
        }
        FF_CLOCK_ADD(threadIdx.x == 192, 10, x10);
        continue;
      }
      const int piece = lane & 3, r8 = lane >> 2;          // a lane's 8 channels of 32 and its token of eight, when storing
      // 16-byte chunk v of token t at v ^ (t mod 8)
      const uint8_t* st_rd0 = st + r8 * 128 + (((2 * piece) ^ r8) << 4);
      const uint8_t* st_rd1 = st + r8 * 128 + (((2 * piece + 1) ^ r8) << 4);
      const long long p0 = (long long)x.tile * XT + quarter * 32 + r8;
      const bool exec = P.alloc[x.bh] & (1 << x.band);
      const __nv_bfloat16* yrow = P.src[(x.band == 1 ? 0 : 2) + (exec ? 0 : 1)] +
                                  ((size_t)(exec ? x.bh : 2 * dm.BH + x.bh) * n_band + p0) * XD + piece * 8;
      const size_t obase = (size_t)(x.bh - P.h0) * dm.N * XD + piece * 8;
      __nv_bfloat16* const grid_hi = P.grid_hi + obase;
      uint8_t* const grid_lo = P.grid_lo + obase;
      float* const grid_f32 = P.grid_f32 + obase;
      int out[4];                                              // element offset of the token's row in the head's grid, or -1
      uint4 yv[4];
#pragma unroll
      for (int i = 0; i < 4; ++i) {
        int f = p0 + 8 * i < n_band ? __ldg(pos + p0 + 8 * i) : -1;
        if (f >= 0 && !FF_DBG_OK(f < dm.N && x.bh >= P.h0 && x.bh < P.h0 + P.g, P.status, 3)) f = -1;   // (debug build)
        out[i] = f * XD;
        yv[i] = f >= 0 ? __ldg((const uint4*)(yrow + 8 * i * XD)) : make_uint4(0, 0, 0, 0);
      }
      FF_CLOCK_ADD(threadIdx.x == 192, 14, x14);
      FF_CLOCK(x9);
      ok = __all_sync(0xffffffffu, mbar_wait(&sh.d_full, n & 1, abort_flag));
      FF_CLOCK_ADD(threadIdx.x == 192, 9, x9);
      if (!ok) break;
      FF_CLOCK(x10);
      tc_fence_after();
      const float* inv = sh.inv[n & 3] + quarter * 32 + r8;
#pragma unroll 1
      for (int q = 0; q < XD / 32; ++q) {
        {
          uint32_t r[32];
          tmem_ld32(tmem + lane_addr + 128 + q * 32, r);
          tmem_wait_ld();
#pragma unroll
          for (int v = 0; v < 8; ++v)
            *(uint4*)(st + lane * 128 + ((v ^ (lane & 7)) << 4)) = make_uint4(r[4 * v], r[4 * v + 1], r[4 * v + 2], r[4 * v + 3]);
        }
        if (q == XD / 32 - 1) {                            // D has been read
          tc_fence_before();
          mbar_arrive(&sh.d_empty);
        }
        __syncwarp();
#pragma unroll
        for (int i = 0; i < 4; ++i) {
          const float4 d0 = *(const float4*)(st_rd0 + i * 1024), d1 = *(const float4*)(st_rd1 + i * 1024);
          const float2 s2 = make_float2(inv[8 * i], inv[8 * i]);
          const uint32_t half = s2.x != s2.x ? 0u : FF_HALF24;     // (a row of NaN)
          const float2 dd[4] = {make_float2(d0.x, d0.y), make_float2(d0.z, d0.w), make_float2(d1.x, d1.y), make_float2(d1.z, d1.w)};
          const uint32_t yw[4] = {yv[i].x, yv[i].y, yv[i].z, yv[i].w};
          uint32_t hi[4], u[8];
          float2 w[4];
#pragma unroll
          for (int k = 0; k < 4; ++k) {
            const float2 v = w[k] = __ffma2_rn(dd[k], s2, make_float2(__uint_as_float(yw[k] << 16), __uint_as_float(yw[k] & 0xffff0000u)));
            u[2 * k] = __float_as_uint(v.x) + half;
            u[2 * k + 1] = __float_as_uint(v.y) + half;
            hi[k] = ff_hi2(u[2 * k], u[2 * k + 1]);
          }
          if (q + 1 < XD / 32 && out[i] >= 0) yv[i] = __ldg((const uint4*)(yrow + 8 * i * XD + (q + 1) * 32));
          if (F32) {
            if (out[i] >= 0) {
              *(float4*)(grid_f32 + out[i] + q * 32) = make_float4(w[0].x, w[0].y, w[1].x, w[1].y);
              *(float4*)(grid_f32 + out[i] + q * 32 + 4) = make_float4(w[2].x, w[2].y, w[3].x, w[3].y);
            }
          } else if (out[i] >= 0) {
            *(uint4*)(grid_hi + out[i] + q * 32) = make_uint4(hi[0], hi[1], hi[2], hi[3]);
            *(uint2*)(grid_lo + out[i] + q * 32) =
                make_uint2(ff_lo4(u[0], u[1], u[2], u[3]), ff_lo4(u[4], u[5], u[6], u[7]));
          }
        }
        __syncwarp();
      }
      FF_CLOCK_ADD(threadIdx.x == 192, 10, x10);
    }
  }

  tc_fence_before();
  __syncthreads();
  if (sh.abort_flag) {
    if (threadIdx.x == 0) atomicExch(P.status, FF_ERR_TIMEOUT | 0x300);   // low byte: status, next byte: which kernel
    const long long t0 = clock64();
    while (clock64() - t0 < 2000000) { }
    __syncthreads();
  }
  ff_pdl_join();
  if (warp == 1) {
    tc_fence_after();
    tmem_dealloc(tmem, 256);
  }
}

bool encode_rows_map(CUtensorMap* map, void* base, long long rows, int slices, int d) {
  cuuint64_t dims[3] = {(cuuint64_t)d, (cuuint64_t)rows, (cuuint64_t)slices};
  cuuint64_t strides[2] = {(cuuint64_t)d * 2, (cuuint64_t)rows * d * 2};
  cuuint32_t box[3] = {64, XT, 1};
  return ff_encode_map(map, CU_TENSOR_MAP_DATA_TYPE_BFLOAT16, 3, base, dims, strides, box, CU_TENSOR_MAP_SWIZZLE_128B,
                       CU_TENSOR_MAP_L2_PROMOTION_L2_256B);
}

}  // namespace

bool ffk_exchange_tc_supported(const FFDims& dm) {
  return !dm.fp32 && (dm.d == 128 || dm.d == 64) && dm.m >= 1 && dm.m <= 32 && dm.N < (1LL << 31);
}

// The form of the kernel a configuration uses.
typedef void (*XKernel)(CUtensorMap, CUtensorMap, CUtensorMap, CUtensorMap, XParams);
template <int D, bool F> static XKernel x_kernel_of(int nkeys) {
  switch (nkeys / 16) {
    case 1: return exchange_tc_kernel<1, D, F>;
    case 2: return exchange_tc_kernel<2, D, F>;
    case 3: return exchange_tc_kernel<3, D, F>;
    case 4: return exchange_tc_kernel<4, D, F>;
    case 5: return exchange_tc_kernel<5, D, F>;
    default: return exchange_tc_kernel<6, D, F>;
  }
}
static XKernel x_kernel(const FFDims& dm) {
  const int nkeys = ff_exchange_keys(dm.m);
  if (ff_fp32_grid(dm)) return dm.d == 128 ? x_kernel_of<128, true>(nkeys) : x_kernel_of<64, true>(nkeys);
  return dm.d == 128 ? x_kernel_of<128, false>(nkeys) : x_kernel_of<64, false>(nkeys);
}

cudaError_t ffk_exchange_tc_init(const FFDims& dm) {
  if (!ffk_exchange_tc_supported(dm)) return cudaSuccess;
  return cudaFuncSetAttribute(x_kernel(dm), cudaFuncAttributeMaxDynamicSharedMemorySize, 113 * 1024);
}

// Rank -> flat coefficient index tables of the mid and high bands (plan-owned device memory).
bool ffk_exchange_tc_build_tables(ff_plan* p) {
  const FFDims& dm = p->dm;
  int* host = (int*)malloc((size_t)(dm.Nmid + dm.Nhigh) * sizeof(int));
  if (!host) return false;
  for (int kt = 0; kt < dm.T; ++kt)
    for (int kh = 0; kh < dm.H; ++kh)
      for (int kw = 0; kw < dm.W; ++kw) {
        long long rank;
        const int band = ff_band_rank_of(dm, kt, kh, kw, &rank);
        const int f = (kt * dm.H + kh) * dm.W + kw;
        if (band == 1) host[rank] = f;
        else if (band == 2) host[dm.Nmid + rank] = f;
      }
  bool ok = cudaMalloc((void**)&p->pos_table, (size_t)(dm.Nmid + dm.Nhigh) * sizeof(int)) == cudaSuccess &&
            cudaMemcpy(p->pos_table, host, (size_t)(dm.Nmid + dm.Nhigh) * sizeof(int), cudaMemcpyHostToDevice) == cudaSuccess;
  free(host);
  return ok;
}

bool ffk_exchange_tc_prepare(ff_plan* p) {
  const FFDims& dm = p->dm;
  // (an empty mid band has no tiles; its maps are encoded over one row of the high band's buffers and never used)
  const long long nm = dm.Nmid > 0 ? dm.Nmid : 1;
  return encode_rows_map((CUtensorMap*)p->tmap_x[0], dm.Nmid > 0 ? p->buf.y_mid : p->buf.y_high, nm, dm.BH, dm.d) &&
         encode_rows_map((CUtensorMap*)p->tmap_x[1], dm.Nmid > 0 ? p->buf.spec_mid : p->buf.spec_high, nm, 3 * dm.BH, dm.d) &&
         encode_rows_map((CUtensorMap*)p->tmap_x[2], p->buf.y_high, dm.Nhigh, dm.BH, dm.d) &&
         encode_rows_map((CUtensorMap*)p->tmap_x[3], p->buf.spec_high, dm.Nhigh, 3 * dm.BH, dm.d);
}

// Exchange + recombination of the mid and high bands of heads [h0, h0+g) into the hi/lo grids (no lo grid: one of fp32).
cudaError_t ffk_exchange_tc(ff_plan* p, int h0, int g, void* grid_hi, void* grid_lo, cudaStream_t st) {
  const FFDims& dm = p->dm;
  XParams P;
  P.dm = dm; P.alloc = p->buf.alloc; P.zimg = p->buf.zimg;
  P.pos_mid = p->pos_table; P.pos_high = p->pos_table + dm.Nmid;
  P.grid_hi = (__nv_bfloat16*)grid_hi; P.grid_lo = (uint8_t*)grid_lo; P.grid_f32 = (float*)grid_hi;
  P.h0 = h0; P.g = g; P.nkeys = ff_exchange_keys(dm.m); P.status = p->buf.status;
  P.src[0] = (const __nv_bfloat16*)p->buf.y_mid; P.src[1] = (const __nv_bfloat16*)p->buf.spec_mid;
  P.src[2] = (const __nv_bfloat16*)p->buf.y_high; P.src[3] = (const __nv_bfloat16*)p->buf.spec_high;
  // Two CTAs per SM, two token tiles each up to 64 keys
  const int per_sm = 2;
  const bool reread = P.nkeys > 64;
  P.ybufs = reread ? 1 : 2;
  const size_t smem = P.ybufs * X_TILE_BYTES + 4 * (size_t)P.nkeys * 128 + 4 * x_stage_bytes(reread) + sizeof(XShared) + 1024;
  const long long tiles = (long long)g * ((dm.Nmid + XT - 1) / XT + (dm.Nhigh + XT - 1) / XT);
  const int grid = tiles < per_sm * p->sm_count ? (int)tiles : per_sm * p->sm_count;
  const CUtensorMap& m0 = *(const CUtensorMap*)p->tmap_x[0];
  const CUtensorMap& m1 = *(const CUtensorMap*)p->tmap_x[1];
  const CUtensorMap& m2 = *(const CUtensorMap*)p->tmap_x[2];
  const CUtensorMap& m3 = *(const CUtensorMap*)p->tmap_x[3];
  p->launches += 1;
  return ff_launch(x_kernel(dm), dim3(grid), dim3(X_THREADS), smem, st, m0, m1, m2, m3, P);
}

FF_CLOCKS_READ(exchange)
